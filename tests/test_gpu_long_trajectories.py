"""Trajectories of more than 2048 frames, which take the dense forms of the time transform (FP32, the split
tensor-core products, the partial transform), on both sides of that line, and the single products with a q
list and the detector sum; against FP64.

Tolerance: sums of 2 F products in FP32, whose roundings add at random to 2^-24 sqrt(2 F) of the result; four
times that, doubled by |.|^2.  The split products drop terms of 2^-16 of an operand (2e-5 in S), a single
one rounds both operands to 8 (BF16) or 11 (TF32) bits: 2 sqrt(2) 2^-9 and 2^-12, doubled by |.|^2."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_10064_gb300 as T
    return T


@pytest.fixture(scope="module")
def ctx(T):
    with T.Context(0) as c:
        yield c


def dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def power(psi):
    x = psi.astype(np.complex128)
    return np.abs(np.fft.fft(x - x.mean(axis=1, keepdims=True), axis=1)) ** 2


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / np.linalg.norm(b))


EXTRA = {"DFT_FP32": 0.0, "DFT_BF16X3": 2e-5, "DFT_TF32X3": 2e-5, "DFT_BF16": 4 * 2 ** 0.5 * 2.0 ** -9,
         "DFT_TF32": 4 * 2 ** 0.5 * 2.0 ** -12}


def tol(F, name):
    return 8 * (2 * F) ** 0.5 * 2.0 ** -24 + EXTRA[name]


def check(ctx, T, P, F, nq, name):
    psi = workloads.random_exit_waves(P, F, nq, seed=F, elastic=10.0, inelastic=0.01)
    ref, code = power(psi), getattr(T, name)
    q = np.sort(np.random.default_rng(F).choice(nq, 37, replace=False)).astype(np.int32)
    S = ctx.spectrum(dev(psi), precision=code).cpu().numpy()
    Sq = ctx.spectrum(dev(psi), precision=code, q_sel=dev(q)).cpu().numpy()
    SI = ctx.spectrum(dev(psi), precision=code, reduce=T.REDUCE_DETECTOR).cpu().numpy()
    SIq = ctx.spectrum(dev(psi), precision=code, reduce=T.REDUCE_DETECTOR, q_sel=dev(q)).cpu().numpy()
    ctx.check()
    assert rel(S, ref) < tol(F, name)
    assert rel(Sq[:, :, q], ref[:, :, q]) < tol(F, name)
    assert not Sq[:, :, np.setdiff1d(np.arange(nq), q)].any()
    assert rel(SI, ref.sum(axis=2)) < tol(F, name)
    assert rel(SIq, ref[:, :, q].sum(axis=2)) < tol(F, name)


@pytest.mark.parametrize("name", ["DFT_FP32", "DFT_BF16X3", "DFT_TF32X3"])
@pytest.mark.parametrize("F", [2047, 2048, 2049, 2100, 3000])
def test_spectrum_around_the_longest_fft(ctx, T, F, name):
    check(ctx, T, 2, F, 300, name)


@pytest.mark.parametrize("name", ["DFT_BF16", "DFT_TF32"])
@pytest.mark.parametrize("F", [17, 64, 2049])
def test_single_products_with_q_list_and_detector(ctx, T, F, name):
    check(ctx, T, 2, F, 300, name)


@pytest.mark.parametrize("F,f0,nf", [(2049, 0, 2049), (2100, 700, 33), (3000, 1500, 1500)])
def test_partial_transform_of_a_long_trajectory(ctx, T, F, f0, nf):
    import torch
    P, nq = 2, 70
    psi = workloads.random_exit_waves(P, nf, nq, seed=F + nf, elastic=1.0, inelastic=0.01)
    ref = workloads.random_exit_waves(P, 1, nq, seed=F + nf, elastic=1.0, inelastic=0.0)[:, 0]
    q = np.arange(3, 64, 2).astype(np.int32)
    x = np.zeros((P, F, nq), dtype=np.complex128)
    x[:, f0:f0 + nf] = psi.astype(np.complex128) - ref[:, None].astype(np.complex128)
    want = np.fft.fft(x, axis=1)
    for qsel, cols in ((None, slice(None)), (q, q)):
        n = nq if qsel is None else len(q)
        out = torch.empty(P, F, n, 2, device="cuda")
        T.tacaw_spectrum_partial(ctx.h, torch.view_as_real(dev(psi)), P, nf, f0, F, nq, torch.view_as_real(dev(ref)),
                                 None if qsel is None else dev(qsel), 0 if qsel is None else n, out)
        got = torch.view_as_complex(out).cpu().numpy()
        assert np.linalg.norm(got - want[:, :, cols]) < tol(F, "DFT_FP32") * np.linalg.norm(want[:, :, cols])
