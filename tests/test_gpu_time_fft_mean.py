"""The frame mean and the residual of the FFT time transform to FP64-class precision, and its sums where
they leave the FP32 range."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2602_10064_gb300 as T
    return T


def dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("F", [32, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1152, 2048])
def test_bin_zero_of_a_column_whose_first_frame_stands_out(T, F):
    """psi = a, b, b, ..., b.  The residual sums to zero, so bin 0 holds only roundings: with the mean exact
    to far below FP32, one per r_n = psi_n - mean and one per level of the sum, each at most 2^-24 of the
    moduli summed.  |X_0| <= (2 log2 F + 8) 2^-24 sum |r_n|.  A mean rounded to FP32 is off by up to
    2^-24 |a - b| in every frame alike, F of which add up."""
    q = 300
    g = np.random.default_rng(F)
    z = lambda: (g.standard_normal(q) + 1j * g.standard_normal(q)).astype(np.complex64)
    psi = np.repeat(z()[None, None], F, axis=1)
    psi[0, 0] = z()
    x = psi.astype(np.complex128)
    bound = (2 * math.log2(F) + 8) * 2.0 ** -24 * np.abs(x - x.mean(axis=1, keepdims=True)).sum(axis=1)[0]
    with T.Context(0) as ctx:
        S = ctx.spectrum(dev(psi)).cpu().numpy()[0, 0].astype(np.float64)
        SI = float(ctx.spectrum(dev(psi), reduce=T.REDUCE_DETECTOR).cpu().numpy()[0, 0])
    assert np.all(S <= bound ** 2), float((np.sqrt(S) / bound).max())
    assert SI <= (bound ** 2).sum()


@pytest.mark.parametrize("F", [3, 7, 49, 100, 127, 200, 501, 768, 1000, 1151, 1999])
def test_constant_columns_give_exactly_zero_at_odd_frame_counts(T, F):
    g = np.random.default_rng(F)
    psi = np.repeat((g.standard_normal(700) + 1j * g.standard_normal(700)).astype(np.complex64)[None, None], F, axis=1)
    with T.Context(0) as ctx:
        assert not ctx.spectrum(dev(psi)).cpu().numpy().any()
        assert not ctx.spectrum(dev(psi), reduce=T.REDUCE_DETECTOR).cpu().numpy().any()


@pytest.mark.parametrize("F", [32, 50, 192, 256, 512, 700, 1024, 2048])
def test_spectrum_image_beyond_the_largest_float(T, F):
    """261 columns of one frequency, |psi~|^2 = 1e38 each: every summand is finite, their sum is not.  The
    image is infinite in that bin, as the FP64 sum rounded to float is, and finite in all others."""
    n, m0 = np.arange(F), 5
    wave = np.sqrt(1e38) / F * np.exp(2j * np.pi * m0 * n / F)
    psi = np.repeat(wave.astype(np.complex64)[None, :, None], 261, axis=2)
    with T.Context(0) as ctx:
        S = ctx.spectrum(dev(psi)).cpu().numpy()[0]
        SI = ctx.spectrum(dev(psi), reduce=T.REDUCE_DETECTOR).cpu().numpy()[0]
    assert np.isfinite(S).all() and np.all(np.abs(S[m0] / 1e38 - 1) < 1e-4)
    assert np.isposinf(SI[m0])
    assert np.isfinite(np.delete(SI, m0)).all()
