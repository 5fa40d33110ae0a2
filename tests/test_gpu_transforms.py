"""Edges of the register transforms: demodulation at every record length (through
IQ-DAS) and odd channel counts, and the allocation-free display stage at every depth."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf
import synth
from test_gpu_parity import assert_close, grid_of, make_handle, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,ne", [(4, 3), (16, 2), (32, 5), (64, 1), (128, 7), (256, 33),
                                   (512, 64), (1024, 31), (4096, 9), (8192, 3)])
def test_demodulated_records(torch, ns, ne):  # noqa: F811
    """IQ-DAS of a grid whose delays stay inside the record, tolerance of test_gpu_parity."""
    c, fs = 1540.0, 20e6
    z1 = 0.45 * (ns - 2) * c / fs
    acq = synth.SPECKLE_POINTS_128.with_(nx=35, nz=max(20, ns // 64), n_elements=ne, n_samples=ns, x0_m=-1e-4,
                                         x1_m=1e-4, z0_m=0.3 * z1, z1_m=z1, pitch_m=2e-5)
    rng = np.random.default_rng(ns)
    rf = rng.integers(-20000, 20000, (1, ne, ns), dtype=np.int16)
    ref = oracle.beamform_iq(oracle.demodulate(rf, acq.fs_hz, acq.f0_hz), acq.x_elements(),
                             acq.angles_rad, grid_of(acq), acq.fs_hz, acq.c_mps, acq.f_number, acq.f0_hz)
    h = make_handle(acq)
    try:
        rf_d = torch.from_numpy(rf).cuda()
        out = torch.full((1, acq.nx, acq.nz), float("nan"), device="cuda")
        bf.bf_beamform(h, rf_d, ns, acq.angles_rad, bf.BF_IQDAS, out)
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    assert_close(out[0].cpu().numpy().astype(np.float64), ref["iqdas"], bf.BF_PREC_FP32, "iq-das")


@pytest.mark.parametrize("nz", [1, 8, 16, 32, 64, 128, 256, 1024, 2048, 4096])
@pytest.mark.parametrize("band", [0, 1])
def test_static_stage_depths(torch, nz, band):  # noqa: F811
    """dB of the float64 analytic signal of the same image: an envelope error of
    4.4e-6 of the column norm (test_gpu_envelope_depths) moves a pixel's dB by at most
    8.686 E / max(env, floor) + 8.686 E / peak, floor = 10^(-70/20) peak."""
    nx, z0 = 37, 5e-3
    z1 = z0 + 40e-6 * max(nz - 1, 1)
    rng = np.random.default_rng(nz)
    y = rng.normal(0, 1000.0, (nx, nz)).astype(np.float32)
    big = torch.zeros(nx * nz + 1, device="cuda")
    outs = [torch.zeros(nx * nz, device="cuda"), big[1:]]  # 16-byte aligned, and 4 bytes off
    yd = torch.from_numpy(y).cuda()
    for out in outs:
        bf.bf_logdb_static(yd, nx, nz, z0, z1, 5e6, 1540.0, band, out)
    torch.cuda.synchronize()
    got = [o.cpu().numpy().astype(np.float64).reshape(nx, nz) for o in outs]
    np.testing.assert_array_equal(got[0], got[1])
    dz = (z1 - z0) / max(nz - 1, 1)
    env = oracle.envelope(y.astype(np.float64), bandpass=bool(band), dz=dz, c=1540.0, f0=5e6)
    peak = env.max()
    if peak == 0:
        assert np.all(got[0] == -70.0)
        return
    err = 4.4e-6 * np.linalg.norm(y, axis=1, keepdims=True)
    tol = 8.686 * err / np.maximum(env, 10 ** (-3.5) * peak) + 8.686 * err.max() / peak + 1e-4
    assert np.all(np.abs(got[0] - oracle.log_compress(env)) <= tol)


@pytest.mark.parametrize("ne,ns,na", [(2, 2, 1), (9, 15, 2), (8, 16, 1), (16, 15, 1), (16, 16, 2), (17, 100, 1),
                                      (33, 513, 3), (64, 1024, 1), (65, 2049, 2), (300, 64, 1),
                                      (3, 4096, 1)])
@pytest.mark.parametrize("stolt", [False, True])
def test_fk_sizes(torch, ne, ns, na, stolt):  # noqa: F811
    """Both transform families around their boundary (32 points along either axis) and
    odd channel counts; tolerance of test_gpu_fk (2e-5 of the image's norm)."""
    rng = np.random.default_rng(ne * 5000 + ns)
    angles = np.deg2rad(np.linspace(-6.0, 6.0, na)) if na > 1 else np.array([0.0])
    rf = rng.integers(-20000, 20000, (na, ne, ns), dtype=np.int16)
    h = bf.bf_create(ne, 0.3e-3, 1.5, (8, 8, -1e-3, 1e-3, 5e-3, 6e-3), 20e6, 5e6, 1540.0)
    try:
        out = torch.full((ne, ns), float("nan"), device="cuda")
        bf.bf_fkmig(h, torch.from_numpy(rf).cuda(), ns, angles, bf.BF_FK_STOLT if stolt else 0, out)
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    ref = (oracle.fk_stolt if stolt else oracle.fk_migrate)(rf, 0.3e-3, angles, 20e6, 1540.0)
    got = out.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
