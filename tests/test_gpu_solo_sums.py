"""Rounding of the sums over channels in a frame beamformed alone."""
import numpy as np
import pytest

import paper_2311_00482_gb300 as bf
from test_gpu_parity import torch  # noqa: F401

pytestmark = pytest.mark.gpu
f32 = np.float32


def test_dmas_sums_round_no_more_than_pairs_of_channels(torch):  # noqa: F811
    """Records that are constant in time make every interpolated sample exact, so DMAS
    ((sum of roots)^2 - sum of magnitudes) / 2 is off by the roots' and the sums' rounding
    only.  Over 64 such frames it is no further from 64 bits than with FP32 sums that add
    two channels at a time to a running sum (the roots here rounded correctly there by
    numpy, on the GPU within a unit in the last place).  The image is large enough for
    one warp per row pair to add all 64 channels."""
    ne, ns, frames = 64, 256, 64
    grid = (640, 192, -1e-3, 1e-3, 1e-3, 4e-3)
    rng = np.random.default_rng(0)
    v = rng.integers(1, 32768, (frames, ne)).astype(np.int16)
    h = bf.bf_create(ne, 0.05e-3, 0.01, grid, 20e6, 5e6, 1540.0)
    try:
        got = np.empty(frames)
        out = torch.empty((1, grid[0], grid[1]), device="cuda")
        for k in range(frames):
            rf = torch.from_numpy(np.repeat(v[k][None, :, None], ns, 2)).cuda()
            torch.cuda.synchronize()
            bf.bf_beamform(h, rf, ns, [0.0], bf.BF_DMAS, out)
            bf.bf_sync(h)
            assert float(out.max() - out.min()) == 0.0
            got[k] = float(out[0, 0, 0])
    finally:
        bf.bf_destroy(h)
    w = v.astype(np.float64)
    exact = (np.sqrt(w).sum(1) ** 2 - w.sum(1)) / 2
    t1 = t2 = np.zeros(frames, f32)
    q = np.sqrt(v.astype(f32))
    for c in range(0, ne, 2):
        t1 = f32(t1 + f32(q[:, c] + q[:, c + 1]))
        t2 = f32(t2 + f32(v[:, c].astype(f32) + v[:, c + 1].astype(f32)))
    pairs = 0.5 * (t1.astype(float) ** 2 - t2.astype(float))
    assert np.linalg.norm(got - exact) <= np.linalg.norm(pairs - exact)
