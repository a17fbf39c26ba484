"""tacaw_build_potential hands out every slice's V at that slice's own precision: a slice with one atom has
the same bits whether the slices around it hold none, one or thousands."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("species", [[14], [8, 14]])
@pytest.mark.parametrize("grid", [32, 96, 256, 512, 1152])
def test_sparse_slice_beside_a_dense_one(grid, species):
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    L, n = 20.0, 3000
    rng = np.random.default_rng(grid)
    atom = np.float32([[[7.3, 11.9, 1.0]]])  # slice 0 of 3, each 2 A
    dense = rng.uniform(0, L, (1, n, 3)).astype(np.float32)
    dense[:, :, 2] = 3.0  # slice 1
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    params = T.make_params(grid, grid, 3, (L, L, 6.0))
    Z = np.full(n + 1, 14, np.int32)
    with T.Context(0) as ctx:
        ctx.load_form_factors(*workloads.placeholder_form_factors(species))
        alone = ctx.build_potential(params, dev(atom), dev(Z[:1]))
        both = ctx.build_potential(params, dev(np.concatenate([atom, dense], axis=1)), dev(Z))
    assert float(alone[0, 0].abs().max()) > 0 and float(both[0, 1].abs().max()) > 0
    assert torch.equal(both[0, 0], alone[0, 0])
    assert not both[0, 2].any()
