"""Arguments of a batch's frames are checked before the library reads through them."""
import ctypes
import mmap
import time

import numpy as np
import pytest

import paper_2311_00482_gb300 as bf
import synth
from test_gpu_parity import make_handle, torch  # noqa: F401

pytestmark = pytest.mark.gpu


def guarded_doubles(n):
    """n doubles that end where a page without access begins, and what keeps them alive."""
    page = mmap.PAGESIZE
    m = mmap.mmap(-1, 2 * page)
    base = ctypes.addressof(ctypes.c_char.from_buffer(m))
    libc = ctypes.CDLL(None, use_errno=True)
    libc.mprotect.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]
    assert libc.mprotect(base + page, page, 0) == 0
    p = ctypes.cast(base + page - 8 * n, ctypes.POINTER(ctypes.c_double))
    for k in range(n):
        p[k] = 0.01 * k
    return p, m


@pytest.mark.parametrize("n_angles", [0, -1, 257, 1 << 20])
@pytest.mark.parametrize("bad", [0, 1])
def test_angle_counts_out_of_range_are_refused_unread(torch, n_angles, bad):  # noqa: F811
    acq = synth.SPECKLE_POINTS_128.with_(nx=16, nz=16)
    lib = bf.load()
    h = make_handle(acq)
    rf = torch.zeros((2, acq.n_elements, acq.n_samples), dtype=torch.int16, device="cuda")
    out = torch.zeros((1, 16, 16), device="cuda")
    angles, keep = guarded_doubles(2)
    try:
        arr = (bf.bf_frame * 2)()
        for k in range(2):
            arr[k] = bf.bf_frame(h, rf.data_ptr(), acq.n_samples, angles, n_angles if k == bad else 2,
                                 bf.BF_DAS, out.data_ptr())
        b = ctypes.c_void_p()
        assert lib.bf_batch_create(arr, 2, ctypes.byref(b)) == bf.BF_EINVAL
        assert not b.value
    finally:
        bf.bf_destroy(h)
        del keep


def test_large_batches_are_prepared_in_linear_time(torch):  # noqa: F811
    """Frames with 256 angles each: comparing every frame with every other would read
    4 GB of angles for 1400 frames and sixteen times that for four times as many; the
    preparation of four times the frames takes less than eight times as long."""
    acq = synth.SPECKLE_POINTS_128.with_(nx=4, nz=4, n_elements=1)
    h = make_handle(acq)
    na, ns = 256, 16
    angles = np.linspace(-0.1, 0.1, na)
    rf = torch.zeros((na, 1, ns), dtype=torch.int16, device="cuda")
    out = torch.zeros((1, 4, 4), device="cuda")

    def prepare(n):
        t = time.perf_counter()
        b = bf.Batch([(h, rf, ns, angles, bf.BF_DAS, out)] * n)
        t = time.perf_counter() - t
        b.close()
        return t

    try:
        prepare(350)
        small, large = min(prepare(350) for _ in range(3)), min(prepare(1400) for _ in range(3))
        assert large < 8 * small
    finally:
        bf.bf_destroy(h)
