"""Envelopes at the edges of the transform sizes: every depth class of the
envelope stage (power-of-two depths, the convolved ones around them, the smallest
and the largest), odd column counts, with and without the band-pass."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf

pytestmark = pytest.mark.gpu

DEPTHS = (1, 2, 3, 16, 17, 31, 32, 33, 64, 65, 128, 129, 256, 257, 511, 513, 1024, 1025, 1750,
          2048, 2049, 4095, 4096)


@pytest.mark.parametrize("nz", DEPTHS)
def test_envelope_depth(nz):
    """env of the device's own beamformed image against the float64 analytic signal.

    Tolerance: a transform of 2^13 points is 13 radix-2 equivalents, each adding at
    most 2 u of relative 2-norm error (u = 2^-24: the twiddle's and the addition's
    rounding); forward and inverse give 52 u, the two parts r and h together
    52 sqrt(2) u = 4.4e-6 of the column norm (the operators' norms are at most 1)."""
    import torch

    nx, ne, ns = 37, 16, 512
    z1 = 5e-3 + 40e-6 * max(nz - 1, 1)
    grid = (nx, nz, -2e-3, 2e-3, 5e-3, z1)
    rng = np.random.default_rng(nz)
    rf = torch.from_numpy(rng.integers(-3000, 3000, (1, ne, ns), dtype=np.int16)).cuda()
    h = bf.bf_create(ne, 0.3e-3, 1.5, grid, 20e6, 5e6, 1540.0)
    try:
        flags = bf.BF_DAS | bf.BF_DMAS
        y = torch.empty((2, nx, nz), device="cuda")
        env = torch.full((2, nx, nz), -1.0, device="cuda")
        torch.cuda.synchronize()
        bf.bf_beamform(h, rf, ns, [0.0], flags, y)
        bf.bf_beamform(h, rf, ns, [0.0], flags | bf.BF_OUT_ENV, env)
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    y, env = y.cpu().numpy().astype(np.float64), env.cpu().numpy().astype(np.float64)
    dz = (z1 - 5e-3) / max(nz - 1, 1)
    for k in range(2):
        ref = oracle.envelope(y[k], bandpass=k == 1, dz=dz, c=1540.0, f0=5e6)
        assert np.linalg.norm(env[k] - ref) <= 4.4e-6 * np.linalg.norm(y[k])


@pytest.mark.parametrize("nz", (300, 800, 1024, 1750, 3000))
def test_band_passed_envelope_repeats(nz):
    """The band-passed image takes two inverse transforms one after the other in the same
    exchange buffer: on a full chip every pass gives the same bits."""
    import torch

    nx, ne, ns = 2048, 4, 512
    grid = (nx, nz, -2e-3, 2e-3, 5e-3, 5e-3 + 40e-6 * (nz - 1))
    rng = np.random.default_rng(nz)
    rf = torch.from_numpy(rng.integers(-3000, 3000, (1, ne, ns), dtype=np.int16)).cuda()
    h = bf.bf_create(ne, 0.3e-3, 1.5, grid, 20e6, 5e6, 1540.0)
    try:
        env = [torch.full((1, nx, nz), -1.0, device="cuda") for _ in range(30)]
        torch.cuda.synchronize()
        for e in env:
            bf.bf_beamform(h, rf, ns, [0.0], bf.BF_DMAS | bf.BF_OUT_ENV, e)
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    for e in env[1:]:
        assert torch.equal(e, env[0])
