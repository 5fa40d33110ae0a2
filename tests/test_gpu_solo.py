"""Frames beamformed alone (the solo tiles): every angle-group size, every split
(rows per tile), channel counts around the runs one window copy brings, irregular
and widely spaced elements, coarse pixels, and the serving engine's switch between a
lone request and one with partners, against the oracle (tolerances of
test_gpu_parity)."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf
import synth
from test_gpu_parity import assert_close, grid_of, make_handle, oracle_all, run_gpu, torch  # noqa: F401

pytestmark = pytest.mark.gpu
ALL = bf.BF_DAS | bf.BF_DMAS | bf.BF_CF


def record(acq):
    return synth.speckle_points_frame(acq)[0]


# 96 x 60: few tiles (split 4); 320 x 256: split 2; 608 x 272: split 1, tiles cut on both sides
@pytest.mark.parametrize("shape", [(95, 61), (318, 250), (607, 271)])
@pytest.mark.parametrize("na", [1, 2, 3, 5])
def test_angle_groups_and_splits(torch, shape, na):  # noqa: F811
    acq = synth.SPECKLE_POINTS_128.with_(nx=shape[0], nz=shape[1],
                                         angles_deg=synth.angles_linspace(na))
    rf = record(acq)
    ref = oracle_all(acq, rf)
    prec = (bf.BF_PREC_FP32, bf.BF_PREC_FP16, bf.BF_PREC_BF16)[na % 3]
    got = run_gpu(torch, acq, rf, ALL | prec)
    for k, name in enumerate(("das", "dmas", "cf")):
        assert_close(got[k], ref[name], prec, name)


@pytest.mark.parametrize("ne", [2, 3, 5, 31, 66])
def test_channel_counts(torch, ne):  # noqa: F811
    acq = synth.SPECKLE_POINTS_128.with_(n_elements=ne, nx=70, nz=45, angles_deg=(-7.0, 2.0, 9.0))
    rf = record(acq)
    ref = oracle_all(acq, rf)
    got = run_gpu(torch, acq, rf, bf.BF_DAS | bf.BF_DMAS)
    assert_close(got[0], ref["das"], bf.BF_PREC_FP32, "das")
    assert_close(got[1], ref["dmas"], bf.BF_PREC_FP32, "dmas")


@pytest.mark.parametrize("gap", [0.0, 6e-3])
def test_irregular_elements_and_coarse_pixels(torch, gap):  # noqa: F811
    """Uneven element spacing (with a gap as wide as many pitches), depth steps of 14
    samples: windows too long for the copies of four channels."""
    rng = np.random.default_rng(3)
    ne, ns, nx, nz = 21, 1024, 40, 33
    xe = np.cumsum(rng.uniform(0.15e-3, 0.6e-3, ne))
    xe[ne // 2:] += gap
    xe -= xe.mean()
    grid = (nx, nz, -5e-3, 5e-3, 2e-3, 2e-3 + 0.55e-3 * (nz - 1))
    angles = np.deg2rad([-12.0, 0.0, 12.0, 20.0])
    rf = rng.integers(-9000, 9000, (4, ne, ns), dtype=np.int16)
    h = bf.bf_create(ne, 0.3e-3, 1.1, grid, 20e6, 5e6, 1540.0, x_elem_m=xe)
    try:
        out = torch.full((1, nx, nz), float("nan"), device="cuda")
        bf.bf_beamform(h, torch.from_numpy(rf).cuda(), ns, angles, bf.BF_DAS, out)
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    ref = oracle.beamform(rf, xe, angles, grid, 20e6, 1540.0, 1.1)["das"]
    # white noise: terms cancel, so against the terms' scale (as the degenerate cases)
    assert np.max(np.abs(out[0].cpu().numpy() - ref)) <= 1e-5 * 4 * ne * 2 ** 15


def test_lone_and_paired_requests_agree(torch):  # noqa: F811
    acq = synth.SPECKLE_POINTS_128.with_(nx=130, nz=90, angles_deg=(-5.0, 0.0, 5.0))
    rf = record(acq)
    ref = oracle_all(acq, rf)
    h = make_handle(acq)
    try:
        for n in (1, 2, 5):
            bf.bf_engine_pause(True)
            t = [bf.bf_submit(h, rf, acq.n_samples, acq.angles_rad, bf.BF_DAS | bf.BF_DMAS)
                 for _ in range(n)]
            bf.bf_engine_pause(False)
            for x in t:
                out = np.empty((2, acq.nx, acq.nz), np.float32)
                assert bf.bf_poll(h, x, out, timeout_us=30_000_000) == bf.BF_OK
                assert_close(out[0].astype(np.float64), ref["das"], bf.BF_PREC_FP32, "das")
                assert_close(out[1].astype(np.float64), ref["dmas"], bf.BF_PREC_FP32, "dmas")
        many = [rf] * 6  # four of them in one job on two-row tiles
        outs = [np.empty((2, acq.nx, acq.nz), np.float32) for _ in many]
        t = bf.bf_submit_many(h, many, acq.n_samples, acq.angles_rad, bf.BF_DAS | bf.BF_DMAS)
        assert bf.bf_poll_many(h, t, outs, timeout_us=30_000_000) == bf.BF_OK
        for out in outs:
            assert_close(out[0].astype(np.float64), ref["das"], bf.BF_PREC_FP32, "das")
            assert_close(out[1].astype(np.float64), ref["dmas"], bf.BF_PREC_FP32, "dmas")
    finally:
        bf.bf_destroy(h)
