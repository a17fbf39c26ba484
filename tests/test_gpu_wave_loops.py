"""Launches so large that a CTA of the slice passes takes several probes or waves one after the other
(the transmission row in registers up to 16 elements a thread, stashed in shared memory above; the
propagator kept through the column pass), against chunks so small that each CTA takes one: the same
arithmetic, so the same bits."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


# rows of 64, 128 and 256 points hold 8 or 16 elements a thread, those of 96, 384, 512 and 768 points 24 or
# 32; 5 x 5 probes split unevenly; one probe: the compact transmission row and the column pass alone
@pytest.mark.parametrize("grid,side,frames,chunk", [(64, 5, 36, 1), (96, 5, 24, 1), (128, 3, 48, 2), (256, 5, 10, 1),
                                                    (384, 5, 6, 1), (512, 3, 8, 1), (768, 3, 6, 1), (128, 1, 400, 40)])
def test_looped_launches_give_the_same_bits(grid, side, frames, chunk):
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    w = workloads.diamond_si(n_frames=frames, grid=grid, n_slices=3, seed=grid)
    if side > 1:
        w.alpha_mrad, w.probes = 30.0, workloads.probe_grid(w.cell[0], w.cell[1], side)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    with T.Context(0) as ctx:
        ctx.load_form_factors(w.form_Z, w.form_coef)
        p, pr, pos, Z = T.params_of(w), T.probe_of(w), dev(w.pos), dev(w.Z)
        whole = ctx.run(p, pos, Z, pr, precision=T.DFT_FP32)
        ctx.set_option("max_chunk_frames", chunk)
        parts = ctx.run(p, pos, Z, pr, precision=T.DFT_FP32)
        ctx.check()
        assert float(whole.abs().max()) > 0
        assert torch.equal(whole, parts)


@pytest.mark.parametrize("block", [1, 3])
def test_blocks_of_whole_slice_pairs_give_the_same_bits(block):
    # one species and more frames than a block of all 5 slices has room for: blocks of slices 2, 2, 1, against
    # blocks that cut the pairs
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    w = workloads.diamond_si(n_frames=130, grid=512, n_slices=5, seed=5)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    with T.Context(0) as ctx:
        ctx.load_form_factors(w.form_Z, w.form_coef)
        p, pr, pos, Z = T.params_of(w), T.probe_of(w), dev(w.pos), dev(w.Z)
        pairs = ctx.run(p, pos, Z, pr, precision=T.DFT_FP32)
        ctx.set_option("max_slice_block", block)
        cut = ctx.run(p, pos, Z, pr, precision=T.DFT_FP32)
        ctx.check()
        assert float(pairs.abs().max()) > 0
        assert torch.equal(pairs, cut)
