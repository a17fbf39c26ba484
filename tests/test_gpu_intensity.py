"""tacaw_intensity on rows that the four-column kernel takes and on those it leaves: the exact FP32
|psi~|^2 (one product rounded, one fused or separate: within 2 units of 2^-24), zero at bin 0."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,shift", [(4, 0), (1024, 0), (1028, 0), (1023, 0), (1026, 0), (1024, 1)])
def test_intensity_rows(nq, shift):
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    P, F = 2, 5
    g = torch.Generator(device="cuda").manual_seed(nq)
    pt = torch.randn(P, F, nq, 2, generator=g, device="cuda")
    buf = torch.full((P * F * nq + 1,), float("nan"), device="cuda")
    S = buf[shift:shift + P * F * nq].view(P, F, nq)  # shift 1: not 16-byte aligned
    with T.Context(0) as ctx:
        T.tacaw_intensity(ctx.h, pt, P, F, nq, None, nq, T.REDUCE_NONE, S)
        got = S.cpu().numpy().astype(np.float64)
    want = (pt.double() ** 2).sum(-1).cpu().numpy()
    want[:, 0] = 0.0
    assert np.all(np.abs(got - want) <= 2 * 2.0 ** -24 * want)
