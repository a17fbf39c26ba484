"""What the performance of this framework is measured on: calls of its public entry points, as a
user's program makes them, over the range of sizes in real use.

Sizes come from the repository's own workloads (workloads/__init__.py): the 128^2, 256^2 and 512^2
crystal configurations, the precision study's 2048 frames, the 1152^2 minimal example and the
serving request mix, with frame counts cut so that a pass takes well under a second.

  run           Context.run: positions in, S(q, w) or the spectrum image out (the whole path)
  potential     Context.build_potential: slice potentials for inspection or for reuse
  transmission  Context.transmission: band-limited exp(i sigma V) from stored potentials
  propagate     Context.propagate: exit waves from stored potentials
  spectrum      Context.spectrum: the time transform of an exit-wave stack
  partial       spectrum_partial + intensity: one rank's share of a frame-sharded transform
"""
import math

import numpy as np
import torch

import paper_2602_10064_gb300 as T

DEV = "cuda"
PRECISION = {"fp32": T.DFT_FP32, "bf16x3": T.DFT_BF16X3, "tf32x3": T.DFT_TF32X3}
GRIDS = (64, 96, 128, 192, 256, 384, 512, 768, 1024, 1152)


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------
def _run(name, crystal, reps, nx, ny, slices, frames, scan, precision, detector):
    return dict(name=name, kind="run", crystal=crystal, rx=reps[0], ry=reps[1], rz=reps[2], nx=nx, ny=ny,
                slices=slices, frames=frames, scan=scan, precision=precision, detector=detector)


def listed():
    return [
        # the smallest configuration: a 64-atom cell, plane wave, default arithmetic; launches and
        # latency count (a user's first call, and the small requests of the serving mix)
        _run("run_si_128", "diamond", (2, 2, 2), 128, 128, 8, 64, 0, "fp32", False),
        # the 512^2 plane-wave configuration with a quarter of its frames: S(q, w) for a dispersion
        _run("run_rocksalt_512", "rocksalt", (10, 10, 10), 512, 512, 20, 256, 0, "bf16x3", False),
        # the benchmark's 16 x 16 probe scan with a quarter of its frames: a spectrum image
        _run("run_scan_256", "diamond", (6, 6, 2), 256, 256, 20, 64, 16, "bf16x3", True),
        # the paper's minimal example (16,000 atoms, 0.094 A sampling) with a tenth of its frames
        _run("run_minimal_1152", "diamond", (20, 20, 5), 1152, 1152, 54, 20, 0, "fp32", False),
        # a small scan on a rectangular grid that is no power of two, odd slice and frame counts
        _run("run_scan_192x96", "rocksalt", (6, 3, 3), 192, 96, 13, 51, 3, "fp32", True),
        # potentials of a few frames at the 512^2 configuration, two species
        dict(name="potential_512", kind="potential", crystal="rocksalt", rx=10, ry=10, rz=10, nx=512, ny=512,
             slices=20, frames=12),
        # transmission functions at the precision study's grid
        dict(name="transmission_1024", kind="transmission", nx=1024, ny=1024, slices=20, frames=4),
        # exit waves of a defocused, aberrated scan from stored potentials, one frame per call
        dict(name="propagate_scan_384", kind="propagate", nx=384, ny=384, slices=20, frames=1, probes=37),
        # the time transform of one exit-wave stack, default arithmetic, every q
        dict(name="spectrum_1024", kind="spectrum", probes=1, frames=1024, nq=256 * 256, band=0, precision="fp32",
             detector=False),
        # the spectrum image of a 32-probe stack over the in-band q of 256^2
        dict(name="spectrum_image_256", kind="spectrum", probes=32, frames=256, nq=256 * 256, band=256,
             precision="bf16x3", detector=True),
        # a trajectory cut to its equilibrated part: a frame count with a large prime factor
        dict(name="spectrum_501", kind="spectrum", probes=3, frames=501, nq=20001, band=0, precision="tf32x3",
             detector=False),
        # one of two ranks' share of a frame-sharded trajectory of 512 frames
        dict(name="partial_512", kind="partial", probes=1, frames=512, first=128, local=256, nq=256 * 256,
             detector=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["run"] * 6 + ["spectrum"] * 3 + ["potential", "propagate", "propagate", "transmission",
                                                         "partial"])
    nx = rng.choice(GRIDS)
    ny = nx if rng.random() < 0.75 else rng.choice(GRIDS)
    crystal = rng.choice(("diamond", "rocksalt"))
    reps = [rng.randint(2, 10) for _ in range(3)]
    if nx == ny and rng.random() < 0.75:
        reps[1] = reps[0]  # square pixels
    slices = rng.randint(5, 40)
    c = dict(kind=kind)
    if kind == "run":
        scan = 0 if rng.random() < 0.5 else rng.randint(2, 12)
        return dict(kind=kind, crystal=crystal, rx=reps[0], ry=reps[1], rz=reps[2], nx=nx, ny=ny, slices=slices,
                    frames=_log(rng, 16, 1024), scan=scan, precision=rng.choice(("fp32", "bf16x3", "tf32x3")),
                    detector=scan > 0 or rng.random() < 0.3)
    if kind == "potential":
        return dict(kind=kind, crystal=crystal, rx=reps[0], ry=reps[1], rz=reps[2], nx=nx, ny=ny, slices=slices,
                    frames=_log(rng, 1, 64))
    if kind == "transmission":
        return dict(kind=kind, nx=nx, ny=ny, slices=slices, frames=_log(rng, 1, 64))
    if kind == "propagate":
        return dict(kind=kind, nx=nx, ny=ny, slices=slices, frames=_log(rng, 1, 16),
                    probes=0 if rng.random() < 0.5 else _log(rng, 1, 128))
    if kind == "spectrum":
        n = rng.choice((96, 128, 192, 256, 384, 512))
        c.update(probes=_log(rng, 1, 64), frames=_log(rng, 16, 2048), nq=n * n, band=n,
                 precision=rng.choice(("fp32", "bf16x3", "tf32x3")), detector=rng.random() < 0.5)
        if rng.random() < 0.3:
            c.update(nq=_log(rng, 1000, 100000), band=0)
        return c
    frames = _log(rng, 16, 1024)
    local = max(1, frames // rng.choice((1, 2, 4)))
    return dict(kind=kind, probes=_log(rng, 1, 8), frames=frames, first=rng.randint(0, frames - local), local=local,
                nq=rng.choice((128, 192, 256)) ** 2, detector=rng.random() < 0.5)


def _state_bytes(case):
    """Device bytes of a case's inputs and outputs (not the library's scratch)."""
    if case["kind"] == "spectrum":
        pf = case["probes"] * case["frames"] * case["nq"]
        return pf * (8 if case["detector"] else 12)
    if case["kind"] == "partial":
        return 8 * case["probes"] * case["nq"] * (case["local"] + 2 * case["frames"])
    if case["kind"] == "run":
        probes = max(1, case["scan"] ** 2)
        out = probes * case["frames"] * (1 if case["detector"] else case["nx"] * case["ny"])
        return 4 * out + 12 * case["frames"] * 8 * case["rx"] * case["ry"] * case["rz"]
    n = case["frames"] * case["slices"] * case["nx"] * case["ny"]
    if case["kind"] == "propagate":
        return 4 * n + 8 * max(1, case["probes"]) * case["frames"] * case["nx"] * case["ny"]
    return n * (12 if case["kind"] == "transmission" else 4)


def draw(rng):
    """One more case; the counts (frames, then probes) shrink until it costs no more than the
    probe scan and holds no more than 4 GiB of inputs and outputs."""
    most = {"flops": 0.25 * work(listed()[2])["flops"], "bytes": 3e9}
    while True:
        c = _draw(rng)
        for _ in range(64):
            w = work(c)
            if w["flops"] <= most["flops"] and w["bytes"] <= most["bytes"] and _state_bytes(c) <= 4 << 30:
                return c
            if c.get("probes", 0) > 2 and rng.random() < 0.5:
                c["probes"] = max(1, int(c["probes"] * 0.7))
            elif c["frames"] > 4 and c["kind"] != "partial":
                c["frames"] = max(1, int(c["frames"] * 0.7))
            elif c["kind"] == "partial" and c["probes"] == 1:
                break
            elif c.get("scan", 0) > 2:
                c["scan"] -= 1


# ------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------
def _fft2_flops(nx, ny):
    return 5.0 * nx * ny * math.log2(nx * ny)


def _band_fraction(nx, ny):
    """Share of the grid inside the disc of radius (2/3) Nyquist of the coarser axis (square pixels
    or not, an estimate: only work() uses it)."""
    return math.pi / 4.0 * (2.0 / 3.0) ** 2


def work(case):
    k = case["kind"]
    F = case["frames"]
    if k == "run":
        nx, ny, S = case["nx"], case["ny"], case["slices"]
        A, P = 8 * case["rx"] * case["ry"] * case["rz"], max(1, case["scan"] ** 2)
        # potential: one transform; transmission: two; each wave and slice: two, and two products
        per_slice = 3 * _fft2_flops(nx, ny) + P * (2 * _fft2_flops(nx, ny) + 12.0 * nx * ny)
        nsel = _band_fraction(nx, ny) * nx * ny
        out = P * F * (1 if case["detector"] else nx * ny)
        return {"bytes": 12.0 * F * A + 4.0 * A + 4.0 * out,
                "flops": F * S * per_slice + P * nsel * 5.0 * F * math.log2(max(F, 2))}
    if k == "spectrum":
        nsel = case["nq"] if not case["band"] else _band_fraction(0, 0) * case["nq"]
        out = case["probes"] * F * (1 if case["detector"] else case["nq"])
        return {"bytes": 8.0 * case["probes"] * F * nsel + 4.0 * out,
                "flops": case["probes"] * nsel * F * (5.0 * math.log2(max(F, 2)) + 6.0)}
    if k == "partial":
        P, nq = case["probes"], case["nq"]
        out = P * F * (1 if case["detector"] else nq)
        return {"bytes": 8.0 * P * nq * (case["local"] + 1 + F) + 4.0 * out,
                "flops": P * nq * F * 5.0 * math.log2(max(F, 2))}
    nx, ny, S = case["nx"], case["ny"], case["slices"]
    n = float(F) * S * nx * ny
    if k == "potential":
        A = 8 * case["rx"] * case["ry"] * case["rz"]
        return {"bytes": 12.0 * F * A + 4.0 * n, "flops": F * S * 2 * _fft2_flops(nx, ny)}
    if k == "transmission":
        return {"bytes": 12.0 * n, "flops": F * S * 2 * _fft2_flops(nx, ny)}
    P = max(1, case["probes"])
    return {"bytes": 4.0 * n + 8.0 * P * F * nx * ny,
            "flops": F * S * (2 * _fft2_flops(nx, ny) + P * (2 * _fft2_flops(nx, ny) + 12.0 * nx * ny))}


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
_contexts = {}


def _context(Z):
    """The process's context for a set of species: a program creates one and keeps it."""
    key = tuple(sorted(set(Z)))
    if key not in _contexts:
        ctx = T.Context(0)
        ctx.load_form_factors(*_form_factors(key))
        _contexts[key] = ctx
    return _contexts[key]


def _form_factors(Zs):
    """Synthetic coefficients of Kirkland's functional form (f(0) of a few A), one row per species."""
    Zs = np.asarray(Zs, dtype=np.int32)
    coef = np.zeros((len(Zs), 12))
    for i, z in enumerate(Zs):
        s = (z / 14.0) ** 0.7
        coef[i, 0:6:2] = np.array([0.5, 1.5, 0.8]) * s
        coef[i, 1:6:2] = np.array([0.12, 1.1, 9.0]) * (14.0 / z) ** 0.2
        coef[i, 6:12:2] = np.array([0.06, 0.02, 0.005]) * s
        coef[i, 7:12:2] = np.array([0.6, 3.0, 18.0])
    return Zs, coef


_FCC = np.array([[0.0, 0.0, 0.0], [0.0, 0.5, 0.5], [0.5, 0.0, 0.5], [0.5, 0.5, 0.0]])


def _crystal(case):
    """Positions [A][3] (A), species [A] and the cell of a replicated diamond or rocksalt crystal."""
    if case["crystal"] == "diamond":
        a, basis, Z = 5.43, np.concatenate([_FCC, _FCC + 0.25]), [14] * 8
    else:
        a, basis, Z = 4.21, np.concatenate([_FCC, (_FCC + np.array([0.5, 0.0, 0.0])) % 1.0]), [12] * 4 + [8] * 4
    r = (case["rx"], case["ry"], case["rz"])
    off = np.stack(np.meshgrid(*(np.arange(k) for k in r), indexing="ij"), -1).reshape(-1, 1, 3)
    R = ((off + basis[None]) * a).reshape(-1, 3)
    return R, np.tile(np.array(Z, dtype=np.int32), off.shape[0]), np.array(r) * a


def _trajectory(case, seed):
    """Harmonic-mode displacements of 0.06 A RMS about the crystal, atoms' planes inside slices:
    positions float32 [F][A][3] on the device, species, cell."""
    R, Z, cell = _crystal(case)
    g = torch.Generator().manual_seed(seed)
    modes, F = 8, case["frames"]
    reps = torch.tensor([case["rx"], case["ry"], case["rz"]], dtype=torch.float64)
    Q = torch.round((2 * torch.rand(modes, 3, generator=g, dtype=torch.float64) - 1) * reps) / torch.from_numpy(cell)
    eps = torch.randn(modes, 3, generator=g, dtype=torch.float64)
    eps = eps / eps.norm(dim=1, keepdim=True)
    phase = 2 * math.pi * torch.rand(modes, generator=g, dtype=torch.float64)
    f_thz = 1.2 + 13.3 * torch.rand(modes, generator=g, dtype=torch.float64)
    amp = 0.06 * math.sqrt(6.0 / modes) * (0.5 + torch.rand(modes, generator=g, dtype=torch.float64))
    Rd = torch.from_numpy(R).to(DEV)
    t = torch.arange(F, dtype=torch.float64, device=DEV) * 5e-3
    pos = (Rd + torch.tensor([0.0, 0.0, 0.5 * cell[2] / case["slices"]], dtype=torch.float64, device=DEV)).repeat(F, 1, 1)
    for m in range(modes):
        arg = (2 * math.pi * (Rd @ Q[m].to(DEV)))[None] - (2 * math.pi * f_thz[m]).to(DEV) * t[:, None] + phase[m].to(DEV)
        pos += (amp[m] * eps[m]).to(DEV) * torch.cos(arg)[..., None]
    return pos.float().contiguous(), Z, cell


def _potentials(case, seed):
    """Smooth random slice potentials of a few hundred V*A at the peaks, [F][S][ny][nx] float32."""
    nx, ny, S, F = case["nx"], case["ny"], case["slices"], case["frames"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    kx = torch.fft.fftfreq(nx, device=DEV)
    ky = torch.fft.fftfreq(ny, device=DEV)
    blur = torch.exp(-0.5 * ((kx[None, :] / 0.08) ** 2 + (ky[:, None] / 0.08) ** 2))[:, : nx // 2 + 1]
    V = torch.empty(F, S, ny, nx, dtype=torch.float32, device=DEV)
    for f in range(F):
        v = torch.fft.irfft2(torch.fft.rfft2(torch.randn(S, ny, nx, generator=g, device=DEV)) * blur, s=(ny, nx))
        V[f] = 40.0 * (v / v.std()) ** 2
    return V


def _exit_waves(probes, frames, nq, seed):
    """A large static wave, a few modes of falling amplitude and noise: complex64 [P][F][nq]."""
    g = torch.Generator(device=DEV).manual_seed(seed)

    def normal(*shape):
        return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV))

    psi = torch.empty(probes, frames, nq, dtype=torch.complex64, device=DEV)
    freq = torch.rand(4, generator=g, device=DEV) - 0.5
    n = torch.arange(frames, device=DEV)
    for p in range(probes):
        base = normal(1, nq)
        psi[p] = base
        psi[p] += 1e-3 * normal(frames, nq)
        for m, a in enumerate((3e-2, 1e-2, 3e-3, 1e-3)):
            psi[p] += a * normal(1, nq) * torch.exp(2j * math.pi * freq[m] * n)[:, None]
    return psi


def _disc(n):
    """The q of an n x n grid inside the (2/3) band limit, ascending, int32."""
    m = torch.fft.fftfreq(n, 1.0 / n, device=DEV).double()
    return torch.nonzero((m[:, None] ** 2 + m[None, :] ** 2).reshape(-1) <= (n / 3.0) ** 2).reshape(-1).int()


def _probe(case, cell, device_seed=0):
    """The illumination: a plane wave, a periodic scan, or aberrated probes at scattered positions."""
    if case["kind"] == "run":
        n = case["scan"]
        if n == 0:
            return dict()
        i = np.arange(n * n)
        return dict(alpha_mrad=30.0, xy=np.stack([(i % n) * cell[0] / n, (i // n) * cell[1] / n], 1))
    if case["probes"] == 0:
        return dict()
    xy = np.random.default_rng(device_seed).random((case["probes"], 2)) * np.asarray(cell[:2])
    return dict(alpha_mrad=25.0, xy=xy, defocus=80.0, cs_mm=0.01, astig=15.0, astig_angle=0.4, coma=300.0,
                coma_angle=1.1)


def _cell_of(case):
    """The cell of stored potentials: 0.1 A pixels, slices 1 A thick."""
    return (0.1 * case["nx"], 0.1 * case["ny"], 1.0 * case["slices"])


def prepare(case, seed):
    k = case["kind"]
    s = {"case": case}
    if k in ("run", "potential"):
        pos, Z, cell = _trajectory(case, seed)
        s.update(ctx=_context(Z.tolist()), pos=pos, Z=torch.from_numpy(Z).to(DEV), cell=cell,
                 params=T.make_params(case["nx"], case["ny"], case["slices"], cell, dt_fs=5.0))
        if k == "run":
            s["probe"] = T.ProbeSpec(**_probe(case, cell))
        return s
    s["ctx"] = _context([14])
    if k in ("transmission", "propagate"):
        cell = _cell_of(case)
        s.update(V=_potentials(case, seed), params=T.make_params(case["nx"], case["ny"], case["slices"], cell))
        if k == "propagate":
            s["probe"] = T.ProbeSpec(**_probe(case, cell, seed))
        return s
    if k == "spectrum":
        s["psi"] = _exit_waves(case["probes"], case["frames"], case["nq"], seed)
        s["q"] = _disc(case["band"]) if case["band"] else None
        return s
    P, F, nq = case["probes"], case["frames"], case["nq"]
    psi = _exit_waves(P, case["local"], nq, seed)
    s.update(psi=psi, ref=psi[:, 0].clone())
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    k = case["kind"]
    if k == "run":
        return ctx.run(s["params"], s["pos"], s["Z"], s["probe"], precision=PRECISION[case["precision"]],
                       reduce=T.REDUCE_DETECTOR if case["detector"] else T.REDUCE_NONE)
    if k == "potential":
        return ctx.build_potential(s["params"], s["pos"], s["Z"])
    if k == "transmission":
        return ctx.transmission(s["params"], s["V"])
    if k == "propagate":
        return ctx.propagate(s["params"], s["V"], s["probe"])
    if k == "spectrum":
        return ctx.spectrum(s["psi"], precision=PRECISION[case["precision"]],
                            reduce=T.REDUCE_DETECTOR if case["detector"] else T.REDUCE_NONE, q_sel=s["q"])
    P, F, nq = case["probes"], case["frames"], case["nq"]
    tilde = torch.empty(P, F, nq, dtype=torch.complex64, device=DEV)
    T.tacaw_spectrum_partial(ctx.h, s["psi"], P, case["local"], case["first"], F, nq, s["ref"], None, 0, tilde)
    S = torch.empty((P, F) if case["detector"] else (P, F, nq), dtype=torch.float32, device=DEV)
    T.tacaw_intensity(ctx.h, tilde, P, F, nq, None, nq,
                      T.REDUCE_DETECTOR if case["detector"] else T.REDUCE_NONE, S)
    return {"tilde": tilde, "S": S}


# ------------------------------------------------------------------------------------------
# the same in 64 bits
# ------------------------------------------------------------------------------------------
_H, _QE, _ME, _C = 6.62607015e-34, 1.602176634e-19, 9.1093837015e-31, 299792458.0
_A0, _EPS0 = 0.529177210903, 8.8541878128e-12


def _wavelength(v):
    return _H / math.sqrt(2 * _ME * _QE * v * (1 + _QE * v / (2 * _ME * _C * _C))) * 1e10


def _sigma(v):
    gamma = 1 + _QE * v / (_ME * _C * _C)
    return 2 * math.pi * gamma * _ME * _QE * (_wavelength(v) * 1e-10) / (_H * _H) * 1e-10


def _k(n, L):
    return torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=DEV) / L


class _Grid:
    def __init__(self, case, cell, v=100e3):
        self.nx, self.ny, self.S = case["nx"], case["ny"], case["slices"]
        self.cell = [float(x) for x in cell]
        self.kx, self.ky = _k(self.nx, self.cell[0]), _k(self.ny, self.cell[1])
        self.k2 = self.ky[:, None] ** 2 + self.kx[None, :] ** 2
        kr = (2.0 / 3.0) * min(0.5 * self.nx / self.cell[0], 0.5 * self.ny / self.cell[1])
        self.mask = self.k2 <= kr * kr
        self.lam, self.sig = _wavelength(v), _sigma(v)
        dz = self.cell[2] / self.S
        self.prop = torch.where(self.mask, torch.exp(-1j * math.pi * self.lam * dz * self.k2), 0)

    def transmission(self, V):
        return torch.fft.ifft2(torch.fft.fft2(torch.exp(1j * self.sig * V)) * self.mask)

    def waves(self, probe):
        """Initial waves [P][ny][nx]."""
        root = math.sqrt(self.nx * self.ny)
        if not probe:
            return torch.full((1, self.ny, self.nx), 1.0 / root, dtype=torch.complex128, device=DEV)
        kmax = probe["alpha_mrad"] * 1e-3 / self.lam
        A = (self.k2 <= kmax * kmax).to(torch.complex128)
        phi = torch.atan2(self.ky[:, None].expand_as(self.k2), self.kx[None, :].expand_as(self.k2))
        k, g = torch.sqrt(self.k2), probe.get
        chi = math.pi * self.lam * self.k2 * (g("defocus", 0) + g("astig", 0) * torch.cos(2 * (phi - g("astig_angle", 0))))
        chi = chi + 2 * math.pi / 3 * g("coma", 0) * self.lam ** 2 * k ** 3 * torch.cos(phi - g("coma_angle", 0))
        chi = chi + 0.5 * math.pi * g("cs_mm", 0) * 1e7 * self.lam ** 3 * self.k2 ** 2
        A = A / math.sqrt(float(A.real.sum())) * torch.exp(-1j * chi)
        xy = torch.from_numpy(np.asarray(probe["xy"], dtype=np.float64)).to(DEV)
        shift = torch.exp(-2j * math.pi * (xy[:, 1, None, None] * self.ky[:, None] + xy[:, 0, None, None] * self.kx))
        return torch.fft.ifft2(A * shift) * root

    def propagate(self, t, psi):
        """Exit waves in k of the waves psi [P][ny][nx] through t [S][ny][nx]."""
        for s in range(self.S):
            psi = torch.fft.fft2(t[s] * psi) * self.prop
            if s < self.S - 1:
                psi = torch.fft.ifft2(psi)
        return psi / math.sqrt(self.nx * self.ny)

    def potential(self, pos, Z, coef):
        """V [S][ny][nx] of one frame: the direct Fourier sum over each slice's atoms."""
        Lx, Ly, Lz = self.cell
        p = pos.double()
        z = p[:, 2] - Lz * torch.floor(p[:, 2] / Lz)
        sl = torch.clamp(torch.floor(z / (Lz / self.S)), 0, self.S - 1).long()
        ix = torch.nonzero(self.mask.any(0)).reshape(-1)
        iy = torch.nonzero(self.mask.any(1)).reshape(-1)
        ex = torch.exp(-2j * math.pi * p[:, 0, None] * self.kx[ix])
        ey = torch.exp(-2j * math.pi * p[:, 1, None] * self.ky[iy])
        q2 = self.k2[iy][:, ix]
        pref = 2 * math.pi * _A0 * (_QE / (4 * math.pi * _EPS0) * 1e10) / (Lx * Ly)
        Vk = torch.zeros(self.S, self.ny, self.nx, dtype=torch.complex128, device=DEV)
        for z_, row in zip(*coef):
            f = sum(row[2 * i] / (q2 + row[2 * i + 1]) for i in range(3))
            f = f + sum(row[6 + 2 * i] * torch.exp(-row[7 + 2 * i] * q2) for i in range(3))
            mine = torch.nonzero(Z == int(z_)).reshape(-1)
            order = mine[torch.argsort(sl[mine], stable=True)]
            counts = torch.bincount(sl[mine], minlength=self.S).tolist()
            at = 0
            for s in range(self.S):
                j = order[at:at + counts[s]]
                at += counts[s]
                if len(j):
                    Vk[s][iy[:, None], ix[None, :]] += pref * f * (ey[j].T @ ex[j])
        return torch.fft.ifft2(Vk * self.mask).real * (self.nx * self.ny)


def _power(psi):
    """|F_t[psi - <psi>]|^2 of complex128 [F][n]."""
    return torch.fft.fft(psi - psi.mean(0, keepdim=True), dim=0).abs().square()


def _exact_run(case, seed):
    pos, Z, cell = _trajectory(case, seed)
    g, probe, F = _Grid(case, cell), _probe(case, cell), case["frames"]
    coef, Zd = _form_factors(sorted(set(Z.tolist()))), torch.from_numpy(Z).to(DEV)
    psi0 = g.waves(probe)
    P, q = psi0.shape[0], torch.nonzero(g.mask.reshape(-1)).reshape(-1)
    psi = torch.empty(P, F, len(q), dtype=torch.complex64 if P * F * len(q) > 1 << 33 else torch.complex128, device=DEV)
    for f in range(F):
        t = g.transmission(g.potential(pos[f], Zd, coef))
        for p in range(0, P, 64):
            psi[p:p + 64, f] = g.propagate(t, psi0[p:p + 64]).reshape(-1, g.ny * g.nx)[:, q]
    if case["detector"]:
        return torch.stack([_power(psi[p]).sum(1) for p in range(P)])
    out = torch.zeros(P, F, g.ny * g.nx, dtype=torch.float64, device=DEV)
    for p in range(P):
        out[p][:, q] = _power(psi[p])
    return out.reshape(P, F, g.ny, g.nx)


def exact(case, seed):
    k, F = case["kind"], case["frames"]
    w = work(case)
    if k == "run" and w["flops"] > 4e12:
        return None
    if k == "run":
        return _exact_run(case, seed)
    if k == "potential":
        pos, Z, cell = _trajectory(case, seed)
        g, coef, Zd = _Grid(case, cell), _form_factors(sorted(set(Z.tolist()))), torch.from_numpy(Z).to(DEV)
        return torch.stack([g.potential(pos[f], Zd, coef) for f in range(F)])
    if k == "transmission":
        g, V = _Grid(case, _cell_of(case)), _potentials(case, seed)
        out = torch.empty(V.shape, dtype=torch.complex128, device=DEV)
        for f in range(F):
            out[f] = g.transmission(V[f].double())
        return out
    if k == "propagate":
        cell = _cell_of(case)
        g, V = _Grid(case, cell), _potentials(case, seed)
        psi0 = g.waves(_probe(case, cell, seed))
        out = torch.empty(psi0.shape[0], F, g.ny, g.nx, dtype=torch.complex128, device=DEV)
        for f in range(F):
            t = g.transmission(V[f].double())
            for p in range(0, psi0.shape[0], 32):
                out[p:p + 32, f] = g.propagate(t, psi0[p:p + 32])
        return out
    if k == "spectrum":
        psi = _exit_waves(case["probes"], F, case["nq"], seed)
        q = _disc(case["band"]).long() if case["band"] else None
        out = []
        for p in range(case["probes"]):
            S = _power((psi[p] if q is None else psi[p][:, q]).to(torch.complex128))
            if case["detector"]:
                out.append(S.sum(1))
            elif q is None:
                out.append(S)
            else:
                out.append(torch.zeros(F, case["nq"], dtype=torch.float64, device=DEV).index_copy_(1, q, S))
        return torch.stack(out)
    psi = _exit_waves(case["probes"], case["local"], case["nq"], seed).to(torch.complex128)
    r = torch.zeros(case["probes"], F, case["nq"], dtype=torch.complex128, device=DEV)
    r[:, case["first"]:case["first"] + case["local"]] = psi - psi[:, :1]
    tilde = torch.fft.fft(r, dim=1)
    S = tilde.abs().square()
    S[:, 0] = 0
    return {"tilde": tilde, "S": S.sum(2) if case["detector"] else S}
