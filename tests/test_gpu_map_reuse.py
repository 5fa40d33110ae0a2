"""Handles of different grids made, used and destroyed in turn: their plans' tensor maps
take each other's device addresses, and every image still matches the oracle."""
import pytest

import paper_2311_00482_gb300 as bf
import synth
from test_gpu_parity import assert_close, make_handle, oracle_all, run_gpu, torch  # noqa: F401

pytestmark = pytest.mark.gpu
SHAPES = ((64, 48), (96, 40), (33, 80), (160, 24))


@pytest.mark.parametrize("rows", [None, "2", "4"])  # solo tiles, and the shared ones
def test_maps_at_reused_addresses(torch, monkeypatch, rows):  # noqa: F811
    if rows:
        monkeypatch.setenv("BF_TILE_ROWS", rows)
    else:
        monkeypatch.delenv("BF_TILE_ROWS", raising=False)
    acqs = [synth.SPECKLE_POINTS_128.with_(nx=nx, nz=nz, angles_deg=(-6.0, 3.0)) for nx, nz in SHAPES]
    rfs = [synth.speckle_points_frame(a)[0] for a in acqs]
    refs = [oracle_all(a, rf) for a, rf in zip(acqs, rfs)]
    for turn in range(6):
        for acq, rf, ref in zip(acqs, rfs, refs):
            h = make_handle(acq)
            try:
                got = run_gpu(torch, acq, rf, bf.BF_DAS | bf.BF_DMAS, h=h)
            finally:
                bf.bf_destroy(h)
            assert_close(got[0], ref["das"], bf.BF_PREC_FP32, "das")
            assert_close(got[1], ref["dmas"], bf.BF_PREC_FP32, "dmas")
