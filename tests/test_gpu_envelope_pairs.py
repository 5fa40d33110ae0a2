"""Depths that are no power of two: two image columns share a transform, and neither's
values reach the other's envelope.  Elements far apart make columns that see one
element (or a cluster) each."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf
from test_gpu_parity import torch  # noqa: F401

pytestmark = pytest.mark.gpu
DEPTHS = (3, 20, 33, 100, 300, 700, 1750, 3000)
Z0, Z1, NS = 5e-3, 14e-3, 512


def images(torch, xe, columns, nz, rf, flags, p=2.0):  # noqa: F811
    """The frame's image and envelope over `columns` columns at 0 .. 40 mm."""
    grid = (columns, nz, 0.0, 40e-3, Z0, Z1)
    h = bf.bf_create(len(xe), 1e-3, 1.0, grid, 20e6, 5e6, 1540.0, x_elem_m=np.asarray(xe))
    try:
        if p != 2.0:
            bf.bf_set_pdas_order(h, p)
        d = torch.from_numpy(rf).cuda()
        nm = bf.n_modes(flags)
        y = torch.empty((nm, columns, nz), device="cuda")
        env = torch.full((nm, columns, nz), -1.0, device="cuda")
        torch.cuda.synchronize()
        bf.bf_beamform(h, d, NS, [0.0], flags, y)
        bf.bf_beamform(h, d, NS, [0.0], flags | bf.BF_OUT_ENV, env)
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    return y.cpu().numpy().astype(np.float64), env.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("nz", DEPTHS)
def test_zero_column_stays_zero(torch, nz):  # noqa: F811
    rng = np.random.default_rng(nz)
    xe = 0.5e-3 * np.arange(4)
    rf = rng.integers(-30000, 30000, (1, 4, NS), dtype=np.int16)
    y, env = images(torch, xe, 2, nz, rf, bf.BF_DAS | bf.BF_DMAS)
    assert np.any(y[:, 0] != 0) and np.all(y[:, 1] == 0)
    assert np.all(env[:, 1] == 0)


@pytest.mark.parametrize("nz", DEPTHS)
def test_quiet_column_keeps_its_precision(torch, nz):  # noqa: F811
    """Amplitudes of 3 and 30000 side by side, on either side; the tolerance is the
    transforms' (test_envelope_depth), relative to each column's own norm."""
    rng = np.random.default_rng(nz)
    rf = np.stack([rng.integers(-a, a + 1, NS) for a in (3, 30000, 3)]).astype(np.int16)[None]
    y, env = images(torch, [0.0, 40e-3 / 3, 80e-3 / 3], 4, nz, rf, bf.BF_DAS)
    for c in range(3):
        ref = oracle.envelope(y[0, c:c + 1], bandpass=False, dz=(Z1 - Z0) / (nz - 1), c=1540.0, f0=5e6)[0]
        assert np.linalg.norm(env[0, c] - ref) <= 4.4e-6 * np.linalg.norm(y[0, c])


@pytest.mark.parametrize("nz", (20, 300, 1750))
def test_overflowing_column_keeps_to_itself(torch, nz):  # noqa: F811
    """pDAS of order 16 over 256 elements overflows; the column beside it sees one element,
    whose power of its root is finite."""
    rng = np.random.default_rng(nz)
    xe = np.append(1e-5 * np.arange(256), 40e-3)
    rf = rng.integers(1000, 30000, (1, 257, NS), dtype=np.int16)
    y, env = images(torch, xe, 2, nz, rf, bf.BF_PDAS, p=16.0)
    assert not np.all(np.isfinite(y[0, 0])) and np.all(np.isfinite(y[0, 1]))
    ref = oracle.envelope(y[0, 1:2], bandpass=False, dz=(Z1 - Z0) / (nz - 1), c=1540.0, f0=5e6)[0]
    assert np.linalg.norm(env[0, 1] - ref) <= 4.4e-6 * np.linalg.norm(y[0, 1])
    assert not np.any(np.isfinite(env[0, 0]))
