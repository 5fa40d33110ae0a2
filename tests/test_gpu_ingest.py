"""Records to sample pairs over odd record lengths and alignments: the beamformed
images against the float64 oracle, in launches of one unit per thread and of several,
alone and in jobs of two and four frames."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf

pytestmark = pytest.mark.gpu

FS, F0, C, PITCH, FNUM = 20e6, 5e6, 1540.0, 0.3e-3, 1.2


@pytest.mark.parametrize("ns", (61, 1000, 2047))
@pytest.mark.parametrize("frames,angles,ne", ((1, 1, 32), (2, 1, 32), (4, 1, 32), (1, 96, 64), (96, 1, 64)))
@pytest.mark.parametrize("prec", (bf.BF_PREC_FP32, bf.BF_PREC_FP16, bf.BF_PREC_BF16))
def test_records_against_oracle(prec, frames, angles, ne, ns):
    """Frames of one plan in a batch.  Tolerance: FP32 as elsewhere (1e-5 of the image's
    norm, mostly the delays'); the stored sample's rounding is at most 2^-11 (FP16) and
    2^-8 (BF16) of it, and the image is linear in the samples."""
    import torch

    z1 = 1e-3 + 0.45 * ns / FS * C / 2
    grid = (40, 48, -2e-3, 2e-3, 1e-3, z1)
    rng = np.random.default_rng(ns + frames + angles)
    ang = np.deg2rad(np.linspace(-3, 3, angles)) if angles > 1 else np.zeros(1)
    rf = rng.integers(-20000, 20000, (frames, angles, ne, ns)).astype(np.int16)
    size = angles * ne * ns
    raw = torch.zeros(frames * (size + 8) + 8, dtype=torch.int16, device="cuda")
    recs = []
    for k in range(frames):  # the last frame at an odd multiple of two bytes
        at = k * ((size + 7) // 8 * 8) + (1 if k == frames - 1 else 0)
        recs.append(raw[at:at + size].view(angles, ne, ns))
    for v, r in zip(recs, rf):
        v.copy_(torch.from_numpy(r))
    out = [torch.empty((1, grid[0], grid[1]), device="cuda") for _ in range(frames)]
    h = bf.bf_create(ne, PITCH, FNUM, grid, FS, F0, C)
    try:
        torch.cuda.synchronize()
        batch = bf.Batch([(h, v, ns, ang, bf.BF_DAS | prec, o) for v, o in zip(recs, out)])
        batch.launch()
        batch.status()
        batch.close()
    finally:
        bf.bf_destroy(h)
    xe = (np.arange(ne) - (ne - 1) / 2) * PITCH
    tol = {bf.BF_PREC_FP32: 1e-5, bf.BF_PREC_FP16: 2.0 ** -11, bf.BF_PREC_BF16: 2.0 ** -8}[prec]
    for k in sorted({0, frames // 2, frames - 1}):
        ref = oracle.beamform(rf[k], xe, ang, grid, FS, C, FNUM)["das"].reshape(grid[0], grid[1])
        got = out[k].cpu().numpy()[0].astype(np.float64)
        assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
