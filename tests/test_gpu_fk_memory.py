"""The f-k stage's scratch: the spectra of every angle once, and angles worked off in
several groups give the oracle's image."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf
import synth
from test_gpu_fk import check, run_fk
from test_gpu_parity import make_handle, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("na", [5, 7])
def test_several_groups_of_angles(torch, na):  # noqa: F811
    """256 elements of 4096 samples: 16.8 MB of spectra per angle, three angles at a time."""
    acq = synth.CYST_WIRES_512.with_(n_elements=256, n_samples=4096,
                                     angles_deg=tuple(np.linspace(-9, 9, na)))
    rng = np.random.default_rng(na)
    rf = rng.integers(-3000, 3000, (na, 256, 4096), dtype=np.int16)
    ref = oracle.fk_migrate(rf, acq.pitch_m, acq.angles_rad, acq.fs_hz, acq.c_mps)
    check(run_fk(torch, acq, rf), ref, "fk %d angles" % na)


def test_scratch_of_many_angles(torch):  # noqa: F811
    ne, ns, na = 256, 4096, 24
    acq = synth.CYST_WIRES_512.with_(n_elements=ne, n_samples=ns, angles_deg=tuple(np.linspace(-9, 9, na)))
    rf = torch.zeros((na, ne, ns), dtype=torch.int16, device="cuda")
    out = torch.zeros((ne, ns), device="cuda")
    nt, nk = 8192, 512
    run_fk(torch, acq.with_(angles_deg=(0.0,)), rf[:1].cpu().numpy())  # tables of the library
    h = make_handle(acq)
    try:
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        bf.bf_fkmig(h, rf, ns, acq.angles_rad, bf.BF_OUT_RF, out)
        bf.bf_sync(h)
        used = before - torch.cuda.mem_get_info()[0]
    finally:
        bf.bf_destroy(h)
    spectra = na * (nt // 2 + 1) * nk * 8
    mapping = na * (nt // 2) * nk * 12
    image = (nt // 2) * nk * 8
    assert used <= 1.01 * spectra + mapping + image + (96 << 20)
