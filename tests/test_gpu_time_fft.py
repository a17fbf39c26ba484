"""The FFT time transform at the edges of its frame counts (engine lengths, chirp-z lengths on both
sides of a power of two, the shortest and the longest) and of its column tiles, against FP64.

Tolerance: the relative rounding of the residual and of two transforms of length M (chirp-z) at one
unit 2^-24 per butterfly level, doubled by |.|^2: 2 (2 log2 M + 8) 2^-24."""
import math

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


def tol(F):
    return 2 * (2 * math.log2(max(4 * F, 32)) + 8) * 2.0 ** -24


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, dtype=np.float64) - b) / np.linalg.norm(b))


FRAMES = [2, 16, 17, 31, 32, 33, 64, 65, 96, 127, 128, 192, 200, 256, 257, 384, 501, 512, 513, 768, 1000, 1024, 1025,
          1152, 1999, 2048]


@pytest.mark.parametrize("F", FRAMES)
def test_full_and_detector_summed_spectrum(ctx, T, F):
    P, nq = 2, 261  # 8 C + a ragged tile for every tile width; over one CTA of the detector sum
    psi = workloads.random_exit_waves(P, F, nq, seed=F, elastic=10.0, inelastic=0.01)
    ref = power(psi)
    for code in (T.DFT_FP32, T.DFT_BF16X3, T.DFT_TF32X3):
        assert rel(ctx.spectrum(dev(psi), precision=code).cpu().numpy(), ref) < tol(F)
        SI = ctx.spectrum(dev(psi), precision=code, reduce=T.REDUCE_DETECTOR).cpu().numpy()
        assert rel(SI, ref.sum(axis=2)) < tol(F)
    q = np.sort(np.random.default_rng(F).choice(nq, 37, replace=False)).astype(np.int32)
    S = ctx.spectrum(dev(psi), q_sel=dev(q)).cpu().numpy()
    want = np.zeros_like(ref)
    want[:, :, q] = ref[:, :, q]
    assert rel(S, want) < tol(F) and not S[:, :, np.setdiff1d(np.arange(nq), q)].any()


@pytest.mark.parametrize("F,f0,nf", [(32, 0, 32), (33, 5, 11), (96, 90, 6), (200, 100, 100), (512, 128, 256), (1025, 1, 1000),
                                     (2048, 2047, 1)])
def test_partial_transform(ctx, T, F, f0, nf):
    import torch
    P, nq = 2, 45
    psi = workloads.random_exit_waves(P, nf, nq, seed=F + nf, elastic=1.0, inelastic=0.01)
    ref = workloads.random_exit_waves(P, 1, nq, seed=F + nf, elastic=1.0, inelastic=0.0)[:, 0]
    x = np.zeros((P, F, nq), dtype=np.complex128)
    x[:, f0:f0 + nf] = psi.astype(np.complex128) - ref[:, None].astype(np.complex128)
    out = torch.empty(P, F, nq, 2, device="cuda")
    T.tacaw_spectrum_partial(ctx.h, torch.view_as_real(dev(psi)), P, nf, f0, F, nq, torch.view_as_real(dev(ref)), None,
                             0, out)
    got = torch.view_as_complex(out).cpu().numpy()
    assert np.linalg.norm(got - np.fft.fft(x, axis=1)) < tol(F) * np.linalg.norm(np.fft.fft(x, axis=1))


@pytest.mark.parametrize("F", [1, 8, 64, 100, 1024])
def test_constant_columns_give_exactly_zero(ctx, T, F):
    psi = np.repeat(workloads.random_exit_waves(1, 1, 40, seed=3, elastic=1e3), F, axis=1)
    assert not ctx.spectrum(dev(psi)).cpu().numpy().any()
