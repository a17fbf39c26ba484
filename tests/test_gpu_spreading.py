"""The spreading pass takes each warp's run of row-sorted candidates, on grids whose row transforms
take 4 to 72 threads (several rows a warp, rows across warps, whole warps): moving an atom by whole
grid rows moves its potential by them.  The atom sits on a grid point, so its outermost taps count (one
of them lost changes V by 1e-5).  Tolerance: four FP32 transforms on either side at 5 units of 2^-24
each."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("species", [[14], [8, 14]])
@pytest.mark.parametrize("n", [32, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1152])
def test_potential_moves_with_the_atom(n, species):
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    L = n * 0.125  # grid coordinates are exact
    params = T.make_params(n, n, 1, (L, L, 2.0))
    Z = torch.tensor([14], dtype=torch.int32, device="cuda")
    with T.Context(0) as ctx:
        ctx.load_form_factors(*workloads.placeholder_form_factors(species))
        ref = None
        for row in list(range(18)) + [n - 9, n - 2, n - 1]:
            pos = torch.tensor([[[1.0, 0.125 * row, 1.0]]], device="cuda")
            V = np.roll(ctx.build_potential(params, pos, Z).cpu().numpy()[0, 0], -row, axis=0).astype(np.float64)
            ref = V if ref is None else ref
            assert np.linalg.norm(V - ref) <= 40 * 2.0 ** -24 * np.linalg.norm(ref), row
