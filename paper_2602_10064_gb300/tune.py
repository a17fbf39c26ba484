"""Autotuner for the FFT pass kernels of the slice path.

Every FFT pass kernel (spreading row pass, potential and band-limit column passes, the row
passes that form t, the multislice row and column passes) comes in variants: 16 or 32 elements
per thread (three- or two-pass transforms), two or three resident CTAs per SM, and for the
column passes twice the columns per CTA.  No single choice is best for all of them: on GB300
three CTAs per SM speed up the spreading pass but slow down the multislice row pass.

This script builds the library once per variant (TACAW_TUNE_FORCE), times every kernel class
at every transform length on representative runs with the library's own CUDA-event profiler,
twice over, and writes csrc/tuning_table.h with the fastest variant per (kernel, length).  A
variant replaces the default only when it is the fastest in both measurements, by at least 2%
(kernels of 10 to 30 us differ by more than that from one process to the next).  Entries that whole runs decided
otherwise are kept in WHOLE_RUNS.  Results of different variants agree to FP32 rounding (the
radix schedule changes the rounding order); the parity tests hold for every variant.

    python -m paper_2602_10064_gb300.tune [--out PATH] [--variants 0 2 ... 14]

Needs a GPU.  Synthetic inputs come from the repository's `workloads` module.
"""
from __future__ import annotations

import argparse
import concurrent.futures as cf
import json
import os
import shutil
import subprocess
import sys
import tempfile

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)

# kernel class (library profiler name; the slice row pass of one probe and of several are two) ->
# KernelId in k_slices.cu
KERNEL_IDS = {"splat_row": 0, "col_pot": 1, "row_pot_t": 2, "row_vt": 3, "col_t": 4, "row_tout": 5,
              "slice_row": 8, "slice_col": 9, "slice_row_scan": 10}
# classes whose kernels take the column-width bit (variant & 4); the others ignore it
COLUMN_CLASSES = {"col_pot", "col_t", "slice_col"}
N_KERNELS = 11
LENGTHS = (32, 64, 128, 256, 512, 1024, 96, 192, 384, 768, 1152)
TUNED_LENGTHS = LENGTHS[1:]
MIN_GAIN = 0.02
# (class, length) -> variant where a kernel's own time and that of a whole run (its launches back to back with
# the others') disagreed: the run had this one faster by 2 to 4%
WHOLE_RUNS = {("slice_row", 1024): 8}


def cases():
    """(transform length, workload factory): a plane wave and a 6 x 6 probe scan at each length, with
    the frames for about 1e8 grid points times slices (the launches fill the device several times)."""
    sys.path.insert(0, ROOT)
    import workloads
    out = []
    for n in TUNED_LENGTHS:
        r, S = max(2, n // 50), 8
        for scan in (0, 6):
            F = max(8, min(512, int(1.5e8 / (n * n * S)))) if not scan else max(4, min(64, int(4e7 / (n * n * S))))

            def make(n=n, r=r, S=S, scan=scan, F=F):
                w = workloads.diamond_si(n_frames=F, grid=n, n_slices=S, seed=n + scan, reps=(r, r, 2))
                if scan:
                    w.alpha_mrad, w.probes = 30.0, workloads.probe_grid(w.cell[0], w.cell[1], scan)
                return w

            out.append((n, make))
    return out


def measure(steps: int = 3) -> dict:
    """Per (kernel class, length): milliseconds per run, summed over the cases of that length."""
    import torch

    import paper_2602_10064_gb300 as T
    out = {}
    ctx = T.Context(0)
    for n, make in cases():
        w = make()
        ctx.load_form_factors(w.form_Z, w.form_coef)
        params, probe = T.params_of(w), T.probe_of(w)
        pos = torch.from_numpy(w.pos).cuda()
        Z = torch.from_numpy(w.Z).cuda()

        def run():
            ctx.run(params, pos, Z, probe, reduce=T.REDUCE_DETECTOR)

        def transmission(V):
            ctx.transmission(params, V)

        run()
        V = ctx.build_potential(params, pos[: min(8, w.n_frames)], Z)
        transmission(V)
        torch.cuda.synchronize()
        best = {}
        for fn in (run, lambda: transmission(V)):
            for _ in range(steps):
                T.tacaw_profile_begin(ctx.h)
                fn()
                torch.cuda.synchronize()
                prof = T.tacaw_profile_end(ctx.h)
                cur = {}
                for cls, (ms, _n, _b, _f) in prof.items():
                    if cls == "slice_row" and w.n_probes > 1:
                        cls = "slice_row_scan"
                    if cls in KERNEL_IDS:
                        cur[cls] = cur.get(cls, 0.0) + ms
                for cls, ms in cur.items():
                    key = f"{cls}@{n}"
                    best[key] = min(best.get(key, float("inf")), ms)
        for key, ms in best.items():
            out[key] = out.get(key, 0.0) + ms
        del pos, Z, V
    ctx.check()
    ctx.close()
    return out


def effective(v: int, cls: str, n: int) -> int:
    """The variant without the bits that change nothing for this kernel and length."""
    if n & (n - 1) or n < 128:
        v &= ~8
    return v if cls in COLUMN_CLASSES else v & ~4


def choose(results: dict) -> list:
    """table[kernel][length index]: the fastest variant, kept at 0 unless MIN_GAIN faster."""
    table = [[0] * len(LENGTHS) for _ in range(N_KERNELS)]
    keys = set().union(*(r.keys() for r in results.values()))
    for key in sorted(keys):
        cls, n = key.split("@")
        if 0 not in results or key not in results[0]:
            continue
        base = results[0][key]
        v_best, t_best = 0, base
        for v, r in results.items():
            if v != effective(v, cls, int(n)):
                continue
            if key in r and r[key] < t_best:
                v_best, t_best = v, r[key]
        if v_best != 0 and t_best > (1.0 - MIN_GAIN) * base:
            v_best = 0
        table[KERNEL_IDS[cls]][LENGTHS.index(int(n))] = v_best
    return table


def agreed(tables: list) -> list:
    """The entries that every measurement chose, else the default."""
    return [[v[0] if len(set(v)) == 1 else 0 for v in zip(*rows)] for rows in zip(*tables)]


def fastest(runs: list) -> dict:
    """{variant: {key: ms}}, the least of the measurements."""
    return {v: {k: min(r[v][k] for r in runs) for k in runs[0][v]} for v in runs[0]}


def whole_runs(table: list) -> list:
    """The table with the entries that whole runs decided."""
    out = [row[:] for row in table]
    for (cls, n), v in WHOLE_RUNS.items():
        out[KERNEL_IDS[cls]][LENGTHS.index(n)] = v
    return out


def digits(ms: float) -> str:
    """Milliseconds to better than the 2% that decide."""
    return f"{ms:.2f}" if ms >= 1 else f"{ms:.4f}"


def header(table: list, results: dict) -> str:
    names = {v: k for k, v in KERNEL_IDS.items()}
    rows = []
    for k in range(N_KERNELS):
        rows.append("    {" + ", ".join(str(x) for x in table[k]) + "},  // " + names.get(k, "probe (not tuned)"))
    lines = [
        "// Variant of each FFT pass kernel per transform length (see Tuned in k_slices.cu).",
        "// Written by paper_2602_10064_gb300/tune.py from CUDA-event timings of every variant on GB300",
        "// (variant & 2: more resident threads; & 4: wide column CTAs; & 8: 32 elements per thread), where whole",
        "// runs did not decide otherwise: " + ", ".join(f"{c}@{n} v{v}" for (c, n), v in WHOLE_RUNS.items()) + ".",
        "// ms per variant:",
    ]
    for key in sorted(set().union(*(r.keys() for r in results.values()))):
        lines.append("//   " + key + ": " + ", ".join(f"v{v} {digits(r[key])}" for v, r in sorted(results.items())
                                                  if key in r))
    lines += ["#pragma once", "", "namespace tacaw {", "",
              "// transform lengths of the columns of kTunedVariant",
              "constexpr int kTunedLengths[11] = {" + ", ".join(str(n) for n in LENGTHS) + "};",
              "",
              "// [kernel][index of N in kTunedLengths]",
              f"constexpr int kTunedVariant[{N_KERNELS}][11] = {{"] + rows + ["};", "",
              "constexpr int tuned_variant(int kernel, int n) {",
              "  for (int l = 0; l < 11; ++l)",
              "    if (kTunedLengths[l] == n) return (kernel >= 0 && kernel < " + str(N_KERNELS) + ") ? kTunedVariant[kernel][l] : 0;",
              "  return 0;",
              "}", "", "}  // namespace tacaw", ""]
    return "\n".join(lines)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--out", default=os.path.join(PKG, "csrc", "tuning_table.h"))
    ap.add_argument("--variants", type=int, nargs="*", default=list(range(0, 16, 2)))
    ap.add_argument("--measure", type=int, default=None, help=argparse.SUPPRESS)
    args = ap.parse_args()
    if args.measure is not None:
        sys.path.insert(0, ROOT)
        from paper_2602_10064_gb300 import _build
        _build.build()
        print(json.dumps(measure()))
        return
    runs = [{}, {}]
    with tempfile.TemporaryDirectory() as tmp:
        # one copy of the package per variant, built side by side, measured one after the other
        def build(v):
            at = os.path.join(tmp, str(v))
            for part in ("include", "workloads"):
                shutil.copytree(os.path.join(ROOT, part), os.path.join(at, part))
            shutil.copytree(PKG, os.path.join(at, os.path.basename(PKG)),
                            ignore=shutil.ignore_patterns("_build", "*.so*", "__pycache__"))
            env = dict(os.environ, TACAW_NVCC_DEFINES=f"-DTACAW_TUNE_FORCE={v}")
            r = subprocess.run([sys.executable, "-m", "paper_2602_10064_gb300._build"], cwd=at, env=env,
                               capture_output=True, text=True)
            if r.returncode != 0:
                raise SystemExit(f"variant {v} failed:\n{r.stdout[-2000:]}\n{r.stderr[-4000:]}")
            return at, env

        with cf.ThreadPoolExecutor(max_workers=max(1, (os.cpu_count() or 4) // 2)) as ex:
            built = list(ex.map(build, args.variants))
        for results in runs:
            for v, (at, env) in zip(args.variants, built):
                r = subprocess.run([sys.executable, "-m", "paper_2602_10064_gb300.tune", "--measure", str(v)], cwd=at,
                                   env=env, capture_output=True, text=True)
                if r.returncode != 0:
                    raise SystemExit(f"variant {v} failed:\n{r.stdout[-2000:]}\n{r.stderr[-4000:]}")
                results[v] = json.loads(r.stdout.strip().splitlines()[-1])
                print(f"variant {v}: " + ", ".join(f"{k} {digits(ms)}" for k, ms in sorted(results[v].items())),
                      flush=True)
    table = whole_runs(agreed([choose(r) for r in runs]))
    with open(args.out, "w") as fh:
        fh.write(header(table, fastest(runs)))
    print(f"wrote {args.out}")


if __name__ == "__main__":
    main()
