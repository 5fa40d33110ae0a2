"""The envelope of a constant column is that constant, exactly: at a power-of-two depth its
transform has one bin (sums of equal integers), the Hilbert part is zero, and the correctly
rounded root of the rounded square of an integer below 2^15 is that integer."""
import numpy as np
import pytest

import paper_2311_00482_gb300 as bf
from test_gpu_parity import torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz", [64, 256, 1024])
def test_constant_columns(torch, nz):  # noqa: F811
    nx, ns = 3, 512
    grid = (nx, nz, -1e-3, 1e-3, 5e-3, 12e-3)
    h = bf.bf_create(1, 0.3e-3, 0.01, grid, 20e6, 5e6, 1540.0)
    values = np.concatenate([np.arange(1, 32768, 331), np.arange(4097, 32768, 577)]).astype(np.int16)
    out = torch.full((len(values), nx, nz), -1.0, device="cuda")
    rf = [torch.full((1, 1, ns), int(v), dtype=torch.int16, device="cuda") for v in values]
    torch.cuda.synchronize()
    try:
        for k in range(len(values)):
            bf.bf_beamform(h, rf[k], ns, [0.0], bf.BF_DAS | bf.BF_OUT_ENV, out[k:k + 1])
        bf.bf_sync(h)
    finally:
        bf.bf_destroy(h)
    want = torch.from_numpy(values.astype(np.float32))[:, None, None].expand(-1, nx, nz)
    assert torch.equal(out.cpu(), want)
