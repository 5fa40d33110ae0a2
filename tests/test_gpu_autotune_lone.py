"""What bf_autotune decides for frames that share their plan with no other."""
import numpy as np
import pytest

import paper_2311_00482_gb300 as bf
import synth
from test_gpu_parity import assert_close, make_handle, oracle_all, run_gpu, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_forced_tiles(monkeypatch):
    monkeypatch.delenv("BF_TILE_ROWS", raising=False)


@pytest.mark.parametrize("shape,flags", [((100, 140), bf.BF_DAS | bf.BF_DMAS), ((512, 300), bf.BF_DAS)])
def test_tuning_a_batch_leaves_lone_frames_their_tiles(torch, shape, flags):  # noqa: F811
    """A lone frame's bits depend on its tiles only: after a batch was tuned they are those
    of a handle that was not."""
    acq = synth.SPECKLE_POINTS_128.with_(nx=shape[0], nz=shape[1], angles_deg=(-5.0, 1.0, 5.0))
    rf, _ = synth.speckle_points_frame(acq)
    plain = run_gpu(torch, acq, rf, flags)
    h = make_handle(acq)
    try:
        res = bf.bf_autotune(h, acq.n_samples, acq.angles_rad, flags, frames=16)
        got = run_gpu(torch, acq, rf, flags, h=h)
        assert np.array_equal(got, plain)
        info = bf.bf_plan_info(h, acq.n_samples, acq.angles_rad, flags)
        assert info["rows"] == res["rows"]
        cf = run_gpu(torch, acq, rf, bf.BF_CF, h=h)
        assert np.array_equal(cf, run_gpu(torch, acq, rf, bf.BF_CF))
    finally:
        bf.bf_destroy(h)


@pytest.mark.parametrize("flags", [bf.BF_DAS | bf.BF_DMAS, bf.BF_DMAS | bf.BF_CF, bf.BF_DAS | bf.BF_PDAS])
@pytest.mark.parametrize("frames", [1, 3])
def test_tuned_lone_frames_match_the_oracle(torch, flags, frames):  # noqa: F811
    acq = synth.SPECKLE_POINTS_128.with_(nx=130, nz=90, angles_deg=(-5.0, 5.0))
    rf, _ = synth.speckle_points_frame(acq)
    ref = oracle_all(acq, rf)
    h = make_handle(acq)
    try:
        bf.bf_autotune(h, acq.n_samples, acq.angles_rad, flags, frames=frames)
        got = run_gpu(torch, acq, rf, flags, h=h)
        names = [n for n, b in (("das", bf.BF_DAS), ("dmas", bf.BF_DMAS), ("cf", bf.BF_CF)) if flags & b]
        for k, name in enumerate(names):
            assert_close(got[k], ref[name], bf.BF_PREC_FP32, name)
        assert np.array_equal(got, run_gpu(torch, acq, rf, flags, h=h))
    finally:
        bf.bf_destroy(h)


def test_tuned_pixels_too_coarse_for_the_default_tiles(torch):  # noqa: F811
    """Depth steps of 310 samples: a 32-row tile's window fits no CTA, a 16-row tile's does.
    Refused by default, served once tuned, in lone calls too."""
    nx, nz, ne, ns = 16, 40, 8, 16384
    z1 = 39 * 310 * 1540.0 / 40e6
    grid = (nx, nz, -2e-3, 2e-3, 0.0, z1)
    rf = torch.randint(-9000, 9000, (1, ne, ns), dtype=torch.int16, device="cuda")
    out = torch.empty((1, nx, nz), device="cuda")
    h = bf.bf_create(ne, 0.3e-3, 1.0, grid, 20e6, 5e6, 1540.0)
    try:
        torch.cuda.synchronize()
        with pytest.raises(bf.BFError):
            bf.bf_beamform(h, rf, ns, [0.0], bf.BF_DAS, out)
        res = bf.bf_autotune(h, ns, [0.0], bf.BF_DAS, frames=4)
        assert res["rows"] == 2
        bf.bf_beamform(h, rf, ns, [0.0], bf.BF_DAS, out)
        bf.bf_sync(h)
        import oracle

        xe = (np.arange(ne) - 0.5 * (ne - 1)) * 0.3e-3
        ref = oracle.beamform(rf.cpu().numpy(), xe, np.zeros(1), grid, 20e6, 1540.0, 1.0)["das"]
        assert np.max(np.abs(out[0].cpu().numpy() - ref)) <= 1e-5 * ne * 2 ** 15
    finally:
        bf.bf_destroy(h)
