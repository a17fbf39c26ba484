"""Launches whose CTAs take up to eight waves through their columns and eight probes through their rows, with
a short last group, against chunks of frames so small that each CTA takes one: the same bits.  A CTA takes
several waves once there are 2 x 16 CTAs of one wave for each of the 152 SMs."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

FULL = 2 * 16 * 152


# grids of every length whose column pass loops, square (row stride fixed at compile time at 128 and 256
# points) and rectangular; one probe: the compact transmission row
@pytest.mark.parametrize("nx,ny,side,frames,slices,chunk", [
    (64, 64, 5, 390, 3, 20), (96, 96, 5, 260, 3, 20), (128, 128, 5, 261, 3, 10), (192, 192, 5, 87, 3, 8),
    (256, 256, 5, 73, 3, 3), (384, 384, 5, 27, 3, 2), (768, 768, 3, 22, 2, 2), (192, 96, 5, 260, 3, 8),
    (64, 256, 5, 73, 3, 3), (128, 128, 1, 1625, 2, 100)])
def test_groups_of_waves_give_the_same_bits(nx, ny, side, frames, slices, chunk):
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    w = workloads.diamond_si(n_frames=frames, grid=ny, n_slices=slices, seed=nx + ny)
    w.nx = nx
    if side > 1:
        w.alpha_mrad, w.probes = 30.0, workloads.probe_grid(w.cell[0], w.cell[1], side)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    # tiles hold at most 32 columns (16 above 192 points) of the band of the shorter reciprocal axis
    tiles = lambda n: -(-(2 * (min(nx, ny) // 3) + 1) // (32 if ny <= 192 else 16)) * n * side * side
    assert tiles(frames) >= FULL > tiles(chunk)
    with T.Context(0) as ctx:
        ctx.load_form_factors(w.form_Z, w.form_coef)
        p, pr, pos, Z = T.params_of(w), T.probe_of(w), dev(w.pos), dev(w.Z)
        out = [torch.empty((pr.n_probes, frames, ny, nx), device="cuda") for _ in range(2)]
        for o, c in zip(out, (0, chunk)):
            if c:
                ctx.set_option("max_chunk_frames", c)
            ctx.run(p, pos, Z, pr, precision=T.DFT_FP32, out=o)
        ctx.check()
        assert float(out[0].abs().max()) > 0
        assert torch.equal(out[0], out[1])
