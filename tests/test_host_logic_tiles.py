"""The rules that choose a frame's tiles by the frames that share its plan, on the CPU."""
import os
import shutil
import subprocess

import pytest

from test_host_logic import CSRC, ROOT, cuda_include

F32, IQ = 0, 3
SOLO = 7  # + log2 of the split
FOURS = {F32: 6, IQ: 4}
PAIRS = 0


@pytest.fixture(scope="module")
def choose(tmp_path_factory):
    inc = cuda_include()
    if inc is None or shutil.which("g++") is None:
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("t") / "tile_choice_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + CSRC, "-I" + inc,
                    os.path.join(ROOT, "tests", "tile_choice_check.cpp"), "-o", exe], check=True)

    def rooms(cap, peers, fixed):
        args = [str(int(x)) for x in (cap, peers, fixed)]
        out = subprocess.run([exe, *args], check=True, capture_output=True, text=True).stdout
        return [int(x) for x in out.split()]

    def run(prec, nx, nz, peers, ns=2048, na=1, sms=152, alone=False, shares=True):
        args = [str(int(x)) for x in (prec, ns, na, nx, nz, sms, alone, shares, peers)]
        return int(subprocess.run([exe, *args], check=True, capture_output=True, text=True).stdout)

    run.rooms = rooms
    return run


@pytest.mark.parametrize("prec", [F32, IQ])
@pytest.mark.parametrize("nx,nz,peers,fours", [(512, 512, 3, False), (512, 512, 4, True), (512, 512, 5, True),
                                               (512, 512, 8, True), (512, 512, 11, True),
                                               (64, 64, 4, False), (64, 64, 12, False), (64, 64, 60, True),
                                               (128, 128, 4, False), (128, 128, 12, False),
                                               (128, 128, 16, True), (256, 256, 4, True), (64, 1750, 4, True)])
def test_fours_need_tiles_for_the_sms(choose, prec, nx, nz, peers, fours):
    assert choose(prec, nx, nz, peers) == (FOURS[prec] if fours else PAIRS)


@pytest.mark.parametrize("peers", [6, 7])
def test_frames_left_behind_a_four(choose, peers):
    assert choose(F32, 512, 512, peers, na=1) == PAIRS
    assert choose(F32, 512, 512, peers, na=3) == FOURS[F32]
    assert choose(IQ, 512, 512, peers, na=1) == FOURS[IQ]


def test_iq_records_that_share_no_job(choose):
    assert choose(IQ, 64, 64, 4, ns=8192) == FOURS[IQ]
    assert choose(IQ, 64, 64, 2, ns=8192) == PAIRS
    assert choose(IQ, 64, 64, 1, ns=8192, alone=True) == PAIRS


def test_combiners_that_share_no_job(choose):
    assert choose(F32, 512, 512, 16, shares=False) == PAIRS


@pytest.mark.parametrize("nx,nz,split", [(64, 64, 2), (256, 224, 2), (256, 256, 1), (416, 256, 1),
                                         (512, 512, 0)])
@pytest.mark.parametrize("peers", [1, 16])
def test_lone_frames_split_by_their_own_tiles(choose, nx, nz, split, peers):
    assert choose(F32, nx, nz, peers, alone=True) == SOLO + split


@pytest.mark.parametrize("cap", [1, 2, 4])
@pytest.mark.parametrize("peers", range(1, 14))
def test_rooms_hold_the_jobs_of_a_batch(choose, cap, peers):
    """Frames join jobs in order, fours, then pairs, then alone: the first of a job holds it."""
    want, left = [], peers
    while left:
        nf = max(n for n in (1, 2, 4) if n <= min(cap, left))
        want += [nf] + [1] * (nf - 1)
        left -= nf
    assert choose.rooms(cap, peers, True) == want


@pytest.mark.parametrize("peers", range(4, 21))
def test_rooms_of_served_frames(choose, peers):
    """No more than two frames' pairs each on average, and a lead for every four."""
    rooms = choose.rooms(4, peers, False)
    assert sum(rooms) <= 2 * peers
    assert rooms[:peers // 4 * 4] == [4, 1, 1, 1] * (peers // 4)
    assert rooms[peers // 4 * 4:] == [2] * (peers % 4)
    assert choose.rooms(2, peers, False) == [2] * peers
