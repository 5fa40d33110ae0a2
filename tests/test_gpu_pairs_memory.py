"""Device memory of the staged sample pairs: a frame that rides in another's job needs no
room for a job of its own."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

import paper_2311_00482_gb300 as bf
import synth
from test_gpu_parity import assert_close, make_handle, oracle_all, torch  # noqa: F401

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("frames", [16, 18, 19])
def test_batch_memory(torch, monkeypatch, frames):  # noqa: F811
    """Batches of one plan hold at most two frames' pairs per frame, and a bit."""
    monkeypatch.delenv("BF_TILE_ROWS", raising=False)
    acq = synth.CYST_WIRES_512.with_(n_samples=2048, angles_deg=tuple(np.linspace(-6, 6, 16)), nx=256, nz=256)
    pairs = 16 * acq.n_elements * 2056 * 8
    rf = torch.zeros((16, acq.n_elements, 2048), dtype=torch.int16, device="cuda")
    out = torch.zeros((1, 256, 256), device="cuda")
    h = make_handle(acq)
    try:
        bf.Batch([(h, rf, 2048, acq.angles_rad, bf.BF_DAS, out)] * frames).close()  # plans, graph memory
        before = torch.cuda.mem_get_info()[0]
        b = bf.Batch([(h, rf, 2048, acq.angles_rad, bf.BF_DAS, out)] * frames)
        used = before - torch.cuda.mem_get_info()[0]
        b.close()
    finally:
        bf.bf_destroy(h)
    assert used <= 2.1 * frames * pairs + (64 << 20)


def test_fours_in_served_and_batched_frames(torch, monkeypatch):  # noqa: F811
    """Seven and nine frames with records of their own: every image is its own frame's."""
    monkeypatch.delenv("BF_TILE_ROWS", raising=False)
    acq = synth.SPECKLE_POINTS_128.with_(nx=300, nz=256, angles_deg=(-5.0, 5.0))
    rfs = [synth.speckle_points_frame(acq, seed=k)[0] for k in range(9)]
    refs = [oracle_all(acq, rf)["das"] for rf in rfs]
    h = make_handle(acq)
    try:
        for n in (7, 9):
            bf.bf_engine_pause(True)
            t = [bf.bf_submit_many(h, rfs[:n], acq.n_samples, acq.angles_rad, bf.BF_DAS),
                 [bf.bf_submit(h, rfs[0], acq.n_samples, acq.angles_rad, bf.BF_DAS)],
                 bf.bf_submit_many(h, rfs[9 - n:], acq.n_samples, acq.angles_rad, bf.BF_DAS)]
            bf.bf_engine_pause(False)
            for tickets, ref in zip(t, (refs[:n], refs[:1], refs[9 - n:])):
                outs = [np.empty((1, acq.nx, acq.nz), np.float32) for _ in tickets]
                assert bf.bf_poll_many(h, tickets, outs, timeout_us=30_000_000) == bf.BF_OK
                for o, r in zip(outs, ref):
                    assert_close(o[0].astype(np.float64), r, bf.BF_PREC_FP32, "served das")
            dev = [torch.from_numpy(rf).cuda() for rf in rfs[:n]]
            outs = [torch.empty((1, acq.nx, acq.nz), device="cuda") for _ in dev]
            torch.cuda.synchronize()
            b = bf.Batch([(h, d, acq.n_samples, acq.angles_rad, bf.BF_DAS, o) for d, o in zip(dev, outs)])
            b.launch()
            torch.cuda.synchronize()
            b.close()
            for o, r in zip(outs, refs):
                assert_close(o[0].cpu().numpy().astype(np.float64), r, bf.BF_PREC_FP32, "batch das")
    finally:
        bf.bf_destroy(h)


def test_served_frames_fit_the_budget_of_two_rooms_each():
    """In a process of its own (the engine's slots outlive a test): eight 512 x 512 frames
    submitted together are admitted with memory for two frames' pairs each."""
    code = textwrap.dedent("""
        import numpy as np
        import paper_2311_00482_gb300 as bf
        import synth
        acq = synth.CYST_WIRES_512.with_(n_samples=2048)
        h = bf.bf_create(acq.n_elements, acq.pitch_m, acq.f_number,
                         (acq.nx, acq.nz, acq.x0_m, acq.x1_m, acq.z0_m, acq.z1_m), acq.fs_hz,
                         acq.f0_hz, acq.c_mps)
        na, ne = len(acq.angles_rad), acq.n_elements
        rf, _ = synth.cyst_wires_frame(acq)
        base = 2 * na * ne * 2048 + 4 * acq.nx * acq.nz + 4096
        bf.bf_engine_configure(memory_budget_bytes=8 * (base + 2 * na * ne * 2056 * 8))
        bf.bf_engine_pause(True)
        t = bf.bf_submit_many(h, [rf] * 8, 2048, acq.angles_rad, bf.BF_DAS)
        bf.bf_engine_pause(False)
        outs = [np.empty((1, acq.nx, acq.nz), np.float32) for _ in t]
        assert len(t) == 8
        assert bf.bf_poll_many(h, t, outs, timeout_us=30_000_000) == bf.BF_OK
        assert all(np.array_equal(o, outs[0]) for o in outs)
        print("admitted")
    """)
    env = {k: v for k, v in os.environ.items() if k != "BF_TILE_ROWS"}
    env["PYTHONPATH"] = ROOT
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env, cwd=ROOT,
                       timeout=300)
    assert r.returncode == 0 and "admitted" in r.stdout, r.stdout + r.stderr
