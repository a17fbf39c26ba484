"""tacaw_build_potential with a Z on the device that is not in the form-factor table: EINVAL, and the
caller's V stays as it was (the check is read before the first kernel that writes V)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def code_of(T, call):
    try:
        call()
    except T.TacawError as e:
        return e.code
    return T.TACAW_OK


@pytest.mark.parametrize("grid,frames,at", [(32, 1, 0), (32, 1, -1), (128, 40, 5)])
def test_rejected_call_leaves_the_output_alone(grid, frames, at):
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    w = workloads.diamond_si(n_frames=frames, grid=grid, n_slices=5)
    Zbad = w.Z.copy()
    Zbad[at] = 79
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    pos, good, bad = dev(w.pos), dev(w.Z), dev(Zbad)
    V = torch.empty((frames, 5, grid, grid), device="cuda")
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    with T.Context(0) as ctx:
        ctx.load_form_factors(w.form_Z, w.form_coef)
        ref = ctx.build_potential(T.params_of(w), pos, good)
        for i in range(6):  # rejected and accepted calls in turn, on two streams
            st = streams[(i // 2) % 2]
            with torch.cuda.stream(st):
                V.fill_(7.0)
                rc = code_of(T, lambda: T.tacaw_build_potential(ctx.h, T.params_of(w), pos, good if i % 2 else bad,
                                                                w.n_atoms, frames, V, st))
                assert rc == (T.TACAW_OK if i % 2 else T.TACAW_EINVAL)
                assert torch.equal(V, ref) if i % 2 else bool((V == 7.0).all())
            torch.cuda.synchronize()
        ctx.check()
