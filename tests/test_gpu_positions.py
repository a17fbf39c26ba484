"""Positions without a place in the cell (not finite, or so far out that FP64 cannot wrap them) keep the grid
indices of the binning inside the grid."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

NAN, INF = float("nan"), float("inf")


def potential(T, ctx, w, pos, Z):
    import torch
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    V = ctx.build_potential(T.params_of(w), dev(pos), dev(Z))
    S = ctx.run(T.params_of(w), dev(pos), dev(Z), T.probe_of(w))
    ctx.check()
    return V, S


@pytest.mark.parametrize("grid", [32, 128])
@pytest.mark.parametrize("xy", [(NAN, 1.0), (1.0, NAN), (INF, 1.0), (1.0, -INF), (NAN, NAN), (-INF, NAN)])
def test_atom_without_a_finite_position_adds_nothing(grid, xy):
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    w = workloads.diamond_si(n_frames=4, grid=grid, n_slices=3)
    extra = np.tile(np.float32([*xy, 1.0]), (4, 1, 1))
    with T.Context(0) as ctx:
        ctx.load_form_factors(w.form_Z, w.form_coef)
        ref = potential(T, ctx, w, w.pos, w.Z)
        got = potential(T, ctx, w, np.concatenate([w.pos, extra], axis=1), np.append(w.Z, w.Z[:1]))
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])


@pytest.mark.parametrize("xyz", [(1e30, 1.0, 1.0), (1.0, -1e30, 1.0), (3e38, -3e38, 1.0), (1.0, 1.0, NAN), (1.0, 1.0, 1e30)])
def test_atom_beyond_every_cell_stays_on_the_grid(xyz):
    import __graft_entry__
    __graft_entry__.build()

    import paper_2602_10064_gb300 as T
    w = workloads.diamond_si(n_frames=2, grid=64, n_slices=3)
    extra = np.tile(np.float32(xyz), (2, 1, 1))
    with T.Context(0) as ctx:
        ctx.load_form_factors(w.form_Z, w.form_coef)
        V, S = potential(T, ctx, w, np.concatenate([w.pos, extra], axis=1), np.append(w.Z, w.Z[:1]))
    assert bool(V.isfinite().all()) and bool(S.isfinite().all())
