"""Slice binning where its comparisons stand in for the divisions of the definition."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 3, 20, 256])
def test_slices_at_cell_and_slice_edges(S):
    """Positions on and next to slice boundaries, cell boundaries and several cells away: the slice of
    the FP64 definition floor(z_w / dz), z_w = z - Lz floor(z / Lz), exactly."""
    import __graft_entry__
    __graft_entry__.build()
    import torch

    import paper_2602_10064_gb300 as T
    Lz = 10.86
    z = (np.arange(-2 * S, 3 * S + 1, dtype=np.float64) * (Lz / S)).astype(np.float32)
    z = np.concatenate([z, np.nextafter(z, np.float32(-1e9)), np.nextafter(z, np.float32(1e9)),
                        np.float32([0.0, -0.0, 1e-30, -1e-30, 1e4, -1e4, 3e7, -3e7])])
    pos = np.zeros((1, len(z), 3), dtype=np.float32)
    pos[0, :, 2] = z
    with T.Context(0) as ctx:
        got = ctx.bin_slices(T.make_params(32, 32, S, (Lz, Lz, Lz)), torch.from_numpy(pos).cuda()).cpu().numpy()[0]
    z = z.astype(np.float64)
    zw = z - Lz * np.floor(z / Lz)
    assert np.array_equal(got, np.clip(np.floor(zw / (Lz / S)), 0, S - 1).astype(np.int32))
