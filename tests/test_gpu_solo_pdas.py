"""The solo tiles' pDAS over every split and several angle groups, alone and with the other
combiners, against the oracle (tolerances of test_gpu_pdas); and a request that stays
alone in its launch against bf_beamform, bit for bit (one plan, one kernel)."""
import functools

import numpy as np
import pytest

import paper_2311_00482_gb300 as bf
import synth
from test_gpu_parity import assert_close, make_handle, oracle_all, run_gpu, torch  # noqa: F401
from test_gpu_pdas import pdas_ref, run_pdas

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_forced_tiles(monkeypatch):
    monkeypatch.delenv("BF_TILE_ROWS", raising=False)


@functools.lru_cache(maxsize=None)
def case(shape, na, p):
    acq = synth.SPECKLE_POINTS_128.with_(nx=shape[0], nz=shape[1], angles_deg=synth.angles_linspace(na))
    rf, _ = synth.speckle_points_frame(acq)
    return acq, rf, {**oracle_all(acq, rf), "pdas": pdas_ref(acq, rf, p)}


# 95 x 61: split 4; 318 x 250: split 2; 607 x 271: split 1, tiles cut on both sides
@pytest.mark.parametrize("shape", [(95, 61), (318, 250), (607, 271)])
@pytest.mark.parametrize("na,p", [(1, 3.0), (2, 2.0), (3, 3.0), (5, 2.0), (5, 3.0)])
@pytest.mark.parametrize("others", [0, bf.BF_DAS | bf.BF_DMAS | bf.BF_CF])
def test_angle_groups_and_splits(torch, shape, na, p, others):  # noqa: F811
    acq, rf, ref = case(shape, na, p)
    got = run_pdas(torch, acq, rf, others | bf.BF_PDAS, p)
    names = ("das", "dmas", "cf", "pdas") if others else ("pdas",)
    for k, name in enumerate(names):
        assert_close(got[k], ref[name], bf.BF_PREC_FP32, "%s p=%g" % (name, p))


@pytest.mark.parametrize("flags", [bf.BF_DAS | bf.BF_DMAS, bf.BF_DMAS | bf.BF_CF, bf.BF_PDAS])
@pytest.mark.parametrize("stage", [bf.BF_OUT_RF, bf.BF_OUT_ENV, bf.BF_OUT_LOGDB])
def test_lone_request_equals_bf_beamform(torch, flags, stage):  # noqa: F811
    acq = synth.SPECKLE_POINTS_128.with_(nx=130, nz=90, angles_deg=(-5.0, 0.0, 5.0))
    rf, _ = synth.speckle_points_frame(acq)
    h = make_handle(acq)
    try:
        want = run_gpu(torch, acq, rf, flags | stage, h=h)
        for _ in range(2):
            t = bf.bf_submit(h, rf, acq.n_samples, acq.angles_rad, flags | stage)
            out = np.empty(want.shape, np.float32)
            assert bf.bf_poll(h, t, out, timeout_us=30_000_000) == bf.BF_OK
            assert np.array_equal(out.astype(np.float64), want)
    finally:
        bf.bf_destroy(h)
