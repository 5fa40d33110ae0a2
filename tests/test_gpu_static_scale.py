"""bf_logdb_static does not depend on the image's scale: scaled by a power of two, an image
gives the same bits.  Every step before the logarithm scales exactly (sums, products with
constants, one square root of a sum of squares inside the range), and the logarithm is
taken of a quotient, in which the scale cancels: the tolerance is zero."""
import numpy as np
import pytest

import paper_2311_00482_gb300 as bf
from test_gpu_parity import torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nz,nx", [(32, 40), (64, 33), (512, 70), (4096, 5)])
@pytest.mark.parametrize("band", [0, 1])
@pytest.mark.parametrize("power", [-40, -3, 30])
def test_scaled_images_give_the_same_decibels(torch, nz, nx, band, power):  # noqa: F811
    rng = np.random.default_rng(nz + band)
    y = (rng.standard_normal((nx, nz)) * 10.0 ** rng.uniform(-3, 0, (nx, 1))).astype(np.float32)
    z1 = 5e-3 + 40e-6 * (nz - 1)
    db = []
    for k in (0, power):
        yd = torch.from_numpy(np.ldexp(y, k)).cuda()
        out = torch.full((nx, nz), float("nan"), device="cuda")
        torch.cuda.synchronize()
        bf.bf_logdb_static(yd, nx, nz, 5e-3, z1, 5e6, 1540.0, band, out)
        torch.cuda.synchronize()
        db.append(out)
    assert float(db[0].max()) == 0.0 and float(db[0].min()) >= -70.0
    assert torch.equal(db[0], db[1])
