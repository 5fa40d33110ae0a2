"""Two channel records of a frame share the demodulation's transform, and neither's values
reach the other's analytic signal.  Elements far apart make columns that see one each."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf
from test_gpu_parity import assert_close, torch  # noqa: F401

pytestmark = pytest.mark.gpu
FS, F0, C = 20e6, 5e6, 1540.0
XE = np.array([0.0, 40e-3 / 3, 80e-3 / 3])


def frame(torch, amplitudes, ns):  # noqa: F811
    nz, z0 = 40, 0.2 * ns * C / (2 * FS)
    grid = (4, nz, 0.0, 40e-3, z0, min(3 * z0, 13e-3))
    rng = np.random.default_rng(ns)
    rf = np.stack([rng.integers(-a, a + 1, ns) for a in amplitudes]).astype(np.int16)[None]
    ref = oracle.beamform_iq(oracle.demodulate(rf, FS, F0), XE, np.zeros(1), grid, FS, C, 1.0, F0)
    h = bf.bf_create(3, 1e-3, 1.0, grid, FS, F0, C, x_elem_m=XE)
    try:
        out = torch.full((2, 4, nz), -1.0, device="cuda")
        d = torch.from_numpy(rf).cuda()
        torch.cuda.synchronize()
        bf.bf_beamform(h, d, ns, [0.0], bf.BF_IQDAS | bf.BF_BBDMAS, out)
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    return out.cpu().numpy().astype(np.float64), ref


@pytest.mark.parametrize("ns", [32, 64, 128, 256, 512])
def test_dead_channel_stays_zero(torch, ns):  # noqa: F811
    got, _ = frame(torch, (0, 30000, 0), ns)
    assert np.any(got[:, 1] != 0)
    assert np.all(got[:, 0] == 0) and np.all(got[:, 2] == 0)


@pytest.mark.parametrize("ns", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("amplitudes", [(3, 30000, 3), (30000, 3, 30000)])
def test_quiet_channel_keeps_its_precision(torch, ns, amplitudes):  # noqa: F811
    got, ref = frame(torch, amplitudes, ns)
    for c in range(3):  # the tolerances of the full images, per column
        assert_close(got[0, c], ref["iqdas"][c], bf.BF_PREC_FP32, "iq-das")
        assert_close(got[1, c], ref["bbdmas"][c], bf.BF_PREC_FP32, "bb-dmas")
