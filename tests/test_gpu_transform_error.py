"""Rounding errors of the register transforms against 64 bits."""
import numpy as np
import pytest

import oracle
import paper_2311_00482_gb300 as bf
import synth
from test_gpu_fk import run_fk
from test_gpu_parity import torch  # noqa: F401

pytestmark = pytest.mark.gpu
f32 = np.float32


def fma(a, b, c):
    """FP32 fused multiply-add (the product is exact in 64 bits)."""
    return f32(np.float64(a) * np.float64(b) + np.float64(c))


def radix4(re, im):
    """Radix-4 Stockham transform in FP32 along the last axis (a last radix-2 pass where the
    length asks for one), every twiddle rounded once, products with fused multiply-adds."""
    m, ns = re.shape[-1], 1

    def turned(a, b, num, den):
        ang = -2 * np.pi * num / den
        wr, wi = f32(np.cos(ang)), f32(np.sin(ang))
        return fma(a, wr, -f32(b * wi)), fma(a, wi, f32(b * wr))

    while 4 * ns <= m:
        j = np.arange(m // 4)
        r = j & (ns - 1)
        v = [(re[..., j + p * m // 4], im[..., j + p * m // 4]) for p in range(4)]
        v = [v[0]] + [turned(*v[p], p * r, 4 * ns) for p in range(1, 4)]
        s0 = v[0][0] + v[2][0], v[0][1] + v[2][1]
        d0 = v[0][0] - v[2][0], v[0][1] - v[2][1]
        s1 = v[1][0] + v[3][0], v[1][1] + v[3][1]
        d1 = v[1][1] - v[3][1], -(v[1][0] - v[3][0])  # times -i
        o = ((j - r) << 2) + r
        re, im = np.empty_like(re), np.empty_like(im)
        for k, (a, b, sg) in enumerate(((s0, s1, 1), (d0, d1, 1), (s0, s1, -1), (d0, d1, -1))):
            re[..., o + k * ns] = a[0] + f32(sg) * b[0]
            im[..., o + k * ns] = a[1] + f32(sg) * b[1]
        ns *= 4
    if ns < m:
        j = np.arange(m // 2)
        b = turned(re[..., j + m // 2], im[..., j + m // 2], j, m)
        a = re[..., j], im[..., j]
        re = np.concatenate([a[0] + b[0], a[0] - b[0]], -1)
        im = np.concatenate([a[1] + b[1], a[1] - b[1]], -1)
    return re, im


@pytest.mark.parametrize("seed", [0, 1])
def test_band_passed_envelope_is_no_further_off_than_radix_4(torch, seed):  # noqa: F811
    """bf_logdb_static with the band-pass, where the band holds little of the signal (its
    spectrum peaks at 0.2 per row, the band begins at 0.44): the error is the forward
    transform's rounding that falls into the band.  It is no larger than that of the
    radix-4 transform with once-rounded twiddles over the same columns."""
    nx, nz = 2000, 512
    rng = np.random.default_rng(seed)
    t = np.arange(-16, 17)
    pulse = np.exp(-t * t / 50.0) * np.cos(2 * np.pi * 0.2 * t)
    g = rng.standard_normal((nx, nz + 32))
    y = f32(1000 * sum(pulse[j] * g[:, j:j + nz] for j in range(33)))
    lo = int(np.ceil(2 * 5e6 / 1540.0 * 35e-3 / (nz - 1) * nz))
    k = np.minimum(np.arange(nz), nz - np.arange(nz))
    sign = np.where(np.arange(nz) * 2 < nz, 1.0, -1.0)

    def envelope(spec):  # of the pairs a + i b, in 64 bits
        spec = np.where(k >= lo, spec, 0)
        z, h = np.fft.ifft(spec), np.fft.ifft(np.where(2 * k == nz, 0, -1j * sign) * spec)
        return np.hypot(z.real, h.real), np.hypot(z.imag, h.imag)

    exact = envelope(np.fft.fft(y[::2].astype(float) + 1j * y[1::2]))
    re, im = radix4(y[::2], y[1::2])
    four = envelope(re.astype(float) + 1j * im)
    out = torch.full((nx, nz), float("nan"), device="cuda")
    yd = torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    bf.bf_logdb_static(yd, nx, nz, 5e-3, 40e-3, 5e6, 1540.0, 1, out)
    torch.cuda.synchronize()
    db = out.cpu().numpy().astype(float)
    peak = max(e.max() for e in exact)
    keep = [e > peak * 10 ** -3.4 for e in exact]  # above the -70 dB floor

    def error(env):
        return np.sqrt(sum((((a - b) ** 2)[m]).sum() for a, b, m in zip(env, exact, keep)))

    ours = 10 ** (db / 20) * peak
    assert error((ours[::2], ours[1::2])) <= error(four)


def test_fk_phases_of_long_delays(torch):  # noqa: F811
    """A transmit of 20 degrees over 128 elements: lateral delays of up to 85 samples, 43
    half turns at the last bin, 21 at the pulse's.  A phase formed in one FP32 product is
    off by 21 pi 2^-25 = 2e-6 rms, the image with it; without that the transforms (42
    radix-2 equivalents of 0.6 u each, as a random walk 2.3e-7) and the tabulated weights
    (u / sqrt(12) each, twice) are left.  Tolerance: twice their sum."""
    acq = synth.CYST_WIRES_512.with_(n_elements=128, n_samples=2048, angles_deg=(20.0,))
    rf, _ = synth.cyst_wires_frame(acq)
    got = run_fk(torch, acq, rf)
    ref = oracle.fk_migrate(rf, acq.pitch_m, acq.angles_rad, acq.fs_hz, acq.c_mps)
    assert np.linalg.norm(got - ref) <= 2 * (2.3e-7 + 0.4e-7) * np.linalg.norm(ref)
