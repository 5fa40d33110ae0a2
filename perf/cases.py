"""Workloads that a user of this beamformer runs, one pass of each through the public calls.

Every case is one kind of program:

  frame    bf_beamform of one device-resident frame, the same buffers again and
           again (an interactive view that is reprocessed)
  ring     bf_beamform of a short sequence of frames on one handle, each in
           buffers of its own (live imaging from a ring of acquisition buffers)
  batch    one prepared graph over frames of one grid, on the tiles that
           bf_autotune picks (offline reconstruction of a recording)
  uneven   one prepared graph over frames of different grids and angle counts
  serve    bf_submit_many_into / bf_poll_many of requests of several grids, in
           page-locked host memory on both sides (the serving path)
  fk       bf_fkmig of one frame (plane-wave f-k migration)
  logdb    bf_logdb_static of one image (the allocation-free display stage)

Sizes are those of the repository's workloads (synth/, bench.py): 128 x 128 x
1024 samples, 512 x 512 x 2048, the paper's depth x lateral grids at 50 MHz,
64-1024 pixels per side with 1-11 plane waves, 1024 x 1024 x 128 elements x
4096 samples x 7 angles, and f-k migration of 64 x 2048 records.
"""
import math

import numpy as np
import torch

import paper_2311_00482_gb300 as bf

DEV = "cuda"
MODES = {"das": bf.BF_DAS, "dmas": bf.BF_DMAS, "cf": bf.BF_CF, "pdas": bf.BF_PDAS,
         "iqdas": bf.BF_IQDAS, "bbdmas": bf.BF_BBDMAS}
PREC = {"fp32": bf.BF_PREC_FP32, "fp16": bf.BF_PREC_FP16, "bf16": bf.BF_PREC_BF16}
OUT = {"rf": bf.BF_OUT_RF, "env": bf.BF_OUT_ENV, "logdb": bf.BF_OUT_LOGDB}
F_NUMBER = 1.5
C_MPS = 1540.0


def _frame(name, nx, nz, ne, ns, na, modes, prec="fp32", out="rf", f0=5e6, fs=20e6, z0=5e-3,
           z1=40e-3, width=19.2e-3, pdas_p=2.0, kind="frame", frames=1):
    case = {"name": name, "kind": kind, "nx": nx, "nz": nz, "ne": ne, "ns": ns, "na": na,
            "modes": modes, "prec": prec, "out": out, "f0": f0, "fs": fs, "z0": z0, "z1": z1,
            "width": width, "pdas_p": pdas_p, "frames": frames}
    if name is None:  # a drawn case
        del case["name"]
    return case


def listed():
    return [
        # the smallest configuration: a preview image, where latency and launches count
        _frame("frame_128_das", 128, 128, 64, 1024, 1, "das"),
        # the paper's deepest grid (1750 x 64, 50 MHz, 7.5 MHz, 3 cm): odd depth, display output
        _frame("frame_1750x64_das_db", 64, 1750, 64, 2048, 1, "das", out="logdb", f0=7.5e6,
               fs=50e6, z0=1e-3, z1=30e-3, width=18.9e-3),
        # the ordinary display frame: both combiners, envelope, log compression
        _frame("frame_512_dmas_db", 512, 512, 64, 2048, 1, "das+dmas", out="logdb"),
        # ragged grid, compounded, pDAS of order 3 on bfloat16 records, envelope output
        _frame("frame_300x384_pdas_bf16", 300, 384, 64, 2048, 3, "das+pdas", prec="bf16",
               out="env", pdas_p=3.0),
        # the largest single frame: 128 elements, 7 angles, FP16 records, all RF combiners
        _frame("frame_1024_cf_fp16", 1024, 1024, 128, 4096, 7, "das+dmas+cf", prec="fp16",
               z1=30e-3, width=38.4e-3),
        # live imaging: eight frames through one handle, three angles each
        _frame("ring_256_dmas_db", 256, 256, 64, 1024, 3, "das+dmas", out="logdb", z1=17e-3,
               kind="ring", frames=8),
        # offline reconstruction of a recording: the benchmark's step
        _frame("batch_512x64_dmas_db", 512, 512, 64, 2048, 1, "das+dmas", out="logdb",
               kind="batch", frames=64),
        # the same for IQ data: IQ-DAS and BB-DMAS magnitudes
        _frame("batch_512x16_iq_db", 512, 512, 64, 2048, 1, "iqdas+bbdmas", out="logdb",
               kind="batch", frames=16),
        # frames of different grids and angle counts in one launch (64-1024 px, 1-11 angles)
        {"name": "uneven_32_db", "kind": "uneven", "frames": 32, "nmin": 64, "nmax": 1024,
         "amax": 11, "ne": 64, "ns": 2048, "prec": "fp32", "out": "logdb"},
        # serving: requests of four grids (128-1024 px, 1-7 angles), host to host
        {"name": "serve_16_db_fp16", "kind": "serve", "frames": 16, "grids": 4, "nmin": 128,
         "nmax": 1024, "amax": 7, "ne": 64, "ns": 2048, "prec": "fp16", "out": "logdb"},
        # f-k migration of one record, three angles, display output
        {"name": "fk_64x2048x3_db", "kind": "fk", "ne": 64, "ns": 2048, "na": 3, "out": "logdb",
         "stolt": False},
        # display stage of an image the caller holds, second-harmonic band-pass
        {"name": "logdb_512x512_band", "kind": "logdb", "nx": 512, "nz": 512, "band": True},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["frame"] * 5 + ["ring", "batch", "batch_iq", "uneven", "serve", "fk", "logdb"])
    if kind == "fk":
        return {"kind": "fk", "ne": _log_int(rng, 24, 128), "ns": _log_int(rng, 300, 4096),
                "na": rng.randint(1, 3), "out": rng.choice(["rf", "logdb"]),
                "stolt": rng.random() < 0.5}
    if kind == "logdb":
        nz = 1 << rng.randint(7, 12)
        return {"kind": "logdb", "nx": _log_int(rng, 32, (1 << 20) // nz), "nz": nz,
                "band": rng.random() < 0.5}
    if kind == "uneven":
        return {"kind": "uneven", "frames": rng.randint(6, 28), "nmin": 64, "nmax": 1024,
                "amax": rng.randint(3, 11), "ne": 64, "ns": _log_int(rng, 1024, 2048),
                "prec": rng.choice(["fp32", "fp16"]), "out": rng.choice(["rf", "logdb"])}
    if kind == "serve":
        return {"kind": "serve", "frames": rng.randint(4, 14), "grids": rng.randint(1, 4),
                "nmin": 128, "nmax": 1024, "amax": 7, "ne": 64, "ns": 2048,
                "prec": rng.choice(["fp32", "fp16"]), "out": "logdb"}
    if kind == "batch_iq":
        return _frame(None, _log_int(rng, 96, 512), _log_int(rng, 96, 512), 64,
                      1 << rng.randint(10, 11), 1, rng.choice(["iqdas", "iqdas+bbdmas"]),
                      out=rng.choice(["rf", "logdb"]), kind="batch", frames=rng.randint(1, 12))
    if kind == "batch":
        return _frame(None, _log_int(rng, 96, 512), rng.choice([256, 512, 1024, _log_int(rng, 128, 700)]),
                      64, _log_int(rng, 1024, 2048), 1, rng.choice(["das", "das+dmas"]),
                      prec=rng.choice(["fp32", "fp16"]), out=rng.choice(["env", "logdb"]),
                      kind="batch", frames=rng.randint(3, 28))
    nx, nz = _log_int(rng, 48, 900), _log_int(rng, 64, 1800)
    na = rng.randint(1, 7)
    z1 = min(40e-3, 5e-3 + nz * 60e-6)  # depth steps that hold the second-harmonic band
    if kind == "ring":
        return _frame(None, min(nx, 400), min(nz, 400), 64, _log_int(rng, 700, 2048), min(na, 5),
                      rng.choice(["das", "das+dmas"]), out=rng.choice(["rf", "logdb"]),
                      z1=min(z1, 29e-3), kind="ring", frames=rng.randint(2, 10))
    return _frame(None, nx, nz, rng.choice([32, 64, 96, 128]), _log_int(rng, 700, 4096),
                  na, rng.choice(["das", "dmas", "das+dmas", "das+cf", "das+dmas+cf", "pdas"]),
                  prec=rng.choice(["fp32", "fp32", "fp16", "bf16"]),
                  out=rng.choice(["rf", "env", "logdb"]), z1=z1, pdas_p=rng.choice([2.0, 3.0]))


# ------------------------------------------------------------------- inputs --

def _angles(na, span_deg=10.0):
    deg = [0.0] if na == 1 else list(np.linspace(-span_deg, span_deg, na))
    return np.deg2rad(np.asarray(deg, dtype=np.float64))


def _elements(ne, pitch):
    return (np.arange(ne, dtype=np.float64) - 0.5 * (ne - 1)) * pitch


def _records(seed, ne, pitch, ns, angles, f0, fs, width, z0, z1):
    """int16 echoes [A][N][Ns] on the GPU: speckle and point targets answered with a
    Gaussian-modulated two-cycle pulse, white noise at 40 dB.  Contributions are
    summed as integers, so the records depend on the seed alone."""
    rng = np.random.default_rng(seed)
    k = 1500
    x = rng.uniform(-width / 2 - 2e-3, width / 2 + 2e-3, k)
    z = rng.uniform(max(z0 - 2e-3, 0.5e-3), z1 + 2e-3, k)
    amp = rng.rayleigh(1.0, k) * rng.choice(np.array([-1.0, 1.0]), k)
    amp[:8] = 20.0
    s = 2.0 / (2.3548 * f0)
    half = 4 * s
    taps = torch.arange(int(math.ceil(2 * half * fs)) + 2, device=DEV)
    xt, zt, at = (torch.from_numpy(v).to(DEV) for v in (x, z, amp))
    xe = torch.from_numpy(_elements(ne, pitch)).to(DEV)[:, None]
    rx = torch.sqrt((xt - xe) ** 2 + zt * zt)
    acc = torch.zeros((len(angles), ne, ns), dtype=torch.int64, device=DEV)
    chan = torch.arange(ne, device=DEV)[:, None, None] * ns
    for a, th in enumerate(angles):
        t = (xt * math.sin(th) + zt * math.cos(th) + rx) / C_MPS
        n = torch.ceil((t - half) * fs).to(torch.int64)[:, :, None] + taps
        tau = n / fs - t[:, :, None]
        w = at[None, :, None] * torch.exp(-tau * tau / (2 * s * s)) * torch.cos(2 * math.pi * f0 * tau)
        w = torch.where((n >= 0) & (n < ns) & (tau.abs() <= half), w, 0.0)
        acc[a].view(-1).scatter_add_(0, (n.clamp(0, ns - 1) + chan).view(-1),
                                     torch.round(w * 2.0 ** 24).to(torch.int64).view(-1))
    clean = acc.to(torch.float64) * 2.0 ** -24
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    rms = math.sqrt(float((acc.abs() >> 12).square().sum()) * 2.0 ** -24 / acc.numel())
    clean += torch.randn(clean.shape, generator=gen, dtype=torch.float64, device=DEV) * (0.01 * rms)
    scale = 0.9 * 32767.0 / max(float(clean.abs().max()), 1e-30)
    return torch.round(clean * scale).clamp(-32768, 32767).to(torch.int16)


_STREAM = []


def _stream():
    """The program's imaging stream, shared by its handles."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


class State:
    """What the program holds: handles, buffers, a prepared batch."""

    def __init__(self, case):
        self.case, self.handles, self.batch = case, [], None

    def handle(self, nx, nz, ne, pitch, f0, fs, width, z0, z1):
        h = bf.bf_create(ne, pitch, F_NUMBER, (nx, nz, -width / 2, width / 2, z0, z1), fs, f0, C_MPS)
        bf.bf_set_stream(h, _stream())
        self.handles.append(h)
        return h

    def __del__(self):
        if self.batch is not None:
            self.batch.close()
        for h in self.handles:
            bf.bf_destroy(h)


def _flags(case, modes=None):
    f = PREC[case["prec"]] | OUT[case["out"]]
    for m in (modes or case["modes"]).split("+"):
        f |= MODES[m]
    return f


def _mixed(case):
    """Frame descriptions of the uneven and serving cases (sizes belong to the case,
    not to the seed): (nx, nz, angles, modes) each."""
    rng = np.random.default_rng(case["frames"] * 1000 + case["amax"])
    if case["kind"] == "uneven":
        return [(int(rng.integers(case["nmin"], case["nmax"] + 1)),
                 int(rng.integers(case["nmin"], case["nmax"] + 1)),
                 int(rng.integers(1, case["amax"] + 1)), "das" if k % 2 == 0 else "dmas")
                for k in range(case["frames"])]
    out = []
    for k in range(case["grids"]):
        n = int(rng.integers(case["nmin"] // 64, case["nmax"] // 64 + 1)) * 64
        out.append((n, n, int(rng.integers(1, case["amax"] + 1)), "das" if k % 2 == 0 else "dmas"))
    return out


def _frame_inputs(case, seed):
    """Records [frames][A][N][Ns] of a frame, ring or batch case: up to four
    acquisitions, the further ones shifted in time."""
    nf = case["frames"]
    base = [_records(seed * 7 + k, case["ne"], 0.3e-3, case["ns"], _angles(case["na"]), case["f0"],
                     case["fs"], case["width"], case["z0"], case["z1"]) for k in range(min(nf, 4))]
    return torch.stack([torch.roll(base[k % 4], 5 * (k // 4), dims=2) for k in range(nf)])


def _mixed_inputs(case, seed):
    """Records per frame of an uneven or serving case: angles of one acquisition of
    11 plane waves, shifted in time from frame to frame."""
    rf11 = _records(seed, case["ne"], 0.3e-3, case["ns"], _angles(11), 5e6, 20e6, 19.2e-3, 5e-3, 40e-3)
    every, rfs, angs = _angles(11), [], []
    per = [case["frames"] // case["grids"] + (k < case["frames"] % case["grids"])
           for k in range(case["grids"])] if case["kind"] == "serve" else [1] * case["frames"]
    k = 0
    for (nx, nz, na, modes), n in zip(_mixed(case), per):
        sel = [5] if na == 1 else [int(round(v)) for v in np.linspace(0, 10, na)]
        for _ in range(n):
            rfs.append(torch.roll(rf11[sel], 3 * k, dims=2).contiguous())
            k += 1
        angs.append(every[sel])
    return rfs, angs, per


def prepare(case, seed):
    st = State(case)
    kind = case["kind"]
    if kind in ("frame", "ring", "batch"):
        h = st.handle(case["nx"], case["nz"], case["ne"], 0.3e-3, case["f0"], case["fs"],
                      case["width"], case["z0"], case["z1"])
        st.flags, st.angles = _flags(case), _angles(case["na"])
        if st.flags & bf.BF_PDAS:
            bf.bf_set_pdas_order(h, case["pdas_p"])
        st.rf = _frame_inputs(case, seed)
        st.out = torch.zeros((case["frames"], bf.n_modes(st.flags), case["nx"], case["nz"]),
                             dtype=torch.float32, device=DEV)
        torch.cuda.synchronize()
        if kind == "batch":
            bf.bf_autotune(h, case["ns"], st.angles, st.flags, frames=min(case["frames"], 16))
            st.batch = bf.Batch([(h, st.rf[k], case["ns"], st.angles, st.flags, st.out[k])
                                 for k in range(case["frames"])])
    elif kind == "uneven":
        rfs, angs, _ = _mixed_inputs(case, seed)
        st.rf, st.outs, frames = rfs, [], []
        for (nx, nz, na, modes), rf, ang in zip(_mixed(case), rfs, angs):
            h = st.handle(nx, nz, case["ne"], 0.3e-3, 5e6, 20e6, 19.2e-3, 5e-3, 40e-3)
            st.outs.append(torch.zeros((1, nx, nz), dtype=torch.float32, device=DEV))
            frames.append((h, rf, case["ns"], ang, _flags(case, modes), st.outs[-1]))
        torch.cuda.synchronize()
        st.batch = bf.Batch(frames)
    elif kind == "serve":
        rfs, angs, per = _mixed_inputs(case, seed)
        st.calls, k = [], 0
        for (nx, nz, na, modes), ang, n in zip(_mixed(case), angs, per):
            h = st.handle(nx, nz, case["ne"], 0.3e-3, 5e6, 20e6, 19.2e-3, 5e-3, 40e-3)
            host = [r.cpu().pin_memory() for r in rfs[k:k + n]]
            out = torch.zeros((n, 1, nx, nz), dtype=torch.float32).pin_memory()
            st.calls.append((h, host, ang, _flags(case, modes) | bf.BF_DEST_ONE_BUFFER, out))
            k += n
    elif kind == "fk":
        h = st.handle(64, 64, case["ne"], 0.3e-3, 5e6, 20e6, 19.2e-3, 5e-3, 40e-3)
        st.angles = _angles(case["na"], 7.0)
        st.flags = OUT[case["out"]] | (bf.BF_FK_STOLT if case["stolt"] else 0)
        depth = case["ns"] * C_MPS / (2 * 20e6)
        st.rf = _records(seed, case["ne"], 0.3e-3, case["ns"], st.angles, 5e6, 20e6,
                         case["ne"] * 0.3e-3, 0.1 * depth, 0.8 * depth)
        st.out = torch.zeros((case["ne"], case["ns"]), dtype=torch.float32, device=DEV)
    else:  # a beamformed image: echoes of a short pulse along depth, column by column
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed))
        t = torch.arange(-16, 17, device=DEV, dtype=torch.float32)
        pulse = torch.exp(-t * t / 50.0) * torch.cos(2 * math.pi * 0.2 * t)
        g = torch.randn((case["nx"], case["nz"] + 32), generator=gen, device=DEV)
        cols = torch.zeros((case["nx"], case["nz"]), device=DEV)
        for j in range(33):
            cols += pulse[j] * g[:, j:j + case["nz"]]
        st.y = (cols * 1000.0).contiguous()
        st.out = torch.zeros_like(st.y)
    torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------- pass --

def run(st):
    case = st.case
    kind = case["kind"]
    if kind in ("frame", "ring"):
        h = st.handles[0]
        for k in range(case["frames"]):
            bf.bf_beamform(h, st.rf[k], case["ns"], st.angles, st.flags, st.out[k])
        return st.out
    if kind == "batch":
        st.batch.launch()
        return st.out
    if kind == "uneven":
        st.batch.launch()
        return st.outs
    if kind == "serve":
        tickets = [bf.bf_submit_many_into(h, host, case["ns"], ang, flags, list(out))
                   for h, host, ang, flags, out in st.calls]
        for (h, _, _, _, _), t in zip(st.calls, tickets):
            bf.bf_poll_many(h, t)
        return [out for _, _, _, _, out in st.calls]
    if kind == "fk":
        bf.bf_fkmig(st.handles[0], st.rf, case["ns"], st.angles, st.flags, st.out)
        return st.out
    bf.bf_logdb_static(st.y, case["nx"], case["nz"], 5e-3, 40e-3, 5e6, C_MPS, case["band"], st.out)
    return st.out


# --------------------------------------------------------------------- work --

def _active(nx, nz, ne, pitch, width, z0, z1):
    """(pixel, channel) pairs inside the F-number aperture."""
    xe = _elements(ne, pitch)
    xs = np.linspace(-width / 2, width / 2, nx)[:, None]
    r = (np.linspace(z0, z1, nz) / (2 * F_NUMBER))[None, :]
    return int((np.searchsorted(xe, xs + r, "right") - np.searchsorted(xe, xs - r, "left")).sum())


# operations per active (pixel, channel, angle): per frame interpolation (2) and the
# combiner's terms (a root counts one); the delay (6) belongs to the geometry
_TERMS = {"das": 1, "dmas": 3, "cf": 2, "pdas": 3, "iqdas": 9, "bbdmas": 8}


def _image_work(nx, nz, modes, out):
    """Envelope (forward and inverse transform of the real column pairs) and log."""
    if out == "rf" or "iqdas" in modes or "bbdmas" in modes:
        return 0.0
    per = 5.0 * nz * math.log2(max(nz, 2))
    return sum(nx / 2 * per * (3 if m == "dmas" else 2) + 4.0 * nx * nz for m in modes.split("+"))


def work(case):
    kind = case["kind"]
    if kind in ("frame", "ring", "batch"):
        act = _active(case["nx"], case["nz"], case["ne"], 0.3e-3, case["width"], case["z0"],
                      case["z1"]) * case["na"]
        nm = len(case["modes"].split("+"))
        per = 2 + sum(_TERMS[m] for m in case["modes"].split("+"))
        nf, px = case["frames"], case["nx"] * case["nz"]
        return {"bytes": nf * (2.0 * case["na"] * case["ne"] * case["ns"] + 4.0 * nm * px),
                "flops": act * (6.0 + nf * per) + nf * _image_work(case["nx"], case["nz"],
                                                                   case["modes"], case["out"])}
    if kind in ("uneven", "serve"):
        b = fl = 0.0
        per = [case["frames"] // case["grids"] + (k < case["frames"] % case["grids"])
               for k in range(case["grids"])] if kind == "serve" else [1] * case["frames"]
        for (nx, nz, na, modes), n in zip(_mixed(case), per):
            b += n * (2.0 * na * case["ne"] * case["ns"] + 4.0 * nx * nz)
            fl += _active(nx, nz, case["ne"], 0.3e-3, 19.2e-3, 5e-3, 40e-3) * na * \
                (6.0 + n * (2 + _TERMS[modes])) + n * _image_work(nx, nz, modes, case["out"])
        return {"bytes": b, "flops": fl}
    if kind == "fk":
        nt, nk = _fk_sizes(case["ne"], case["ns"])
        fl = case["na"] * (case["ne"] * 2.5 * nt * math.log2(nt) +
                           nt / 2 * (5.0 * nk * math.log2(nk) + 8.0 * nk)) + \
            nt / 2 * 5.0 * nk * math.log2(nk) + case["ne"] * 5.0 * nt * math.log2(nt)
        return {"bytes": 2.0 * case["na"] * case["ne"] * case["ns"] + 4.0 * case["ne"] * case["ns"],
                "flops": fl}
    return {"bytes": 8.0 * case["nx"] * case["nz"],
            "flops": _image_work(case["nx"], case["nz"], "dmas" if case["band"] else "das", "logdb")}


# -------------------------------------------------------------------- exact --

def _linspace(lo, hi, n):
    return np.array([lo]) if n == 1 else lo + np.arange(n, dtype=np.float64) * ((hi - lo) / (n - 1))


def _beamform64(rfs, angles, ne, nx, nz, fs, f0, width, z0, z1, modes, pdas_p):
    """Images [frames][modes][nx][nz] in float64 by the definitions of include/bf.h.
    rfs: [frames][A][N][Ns] int16."""
    modes = modes.split("+")
    nf, na, ns = rfs.shape[0], rfs.shape[1], rfs.shape[3]
    iq = "iqdas" in modes or "bbdmas" in modes
    xe = torch.from_numpy(_elements(ne, 0.3e-3)).to(DEV)
    xs = torch.from_numpy(_linspace(-width / 2, width / 2, nx)).to(DEV)
    zs = torch.from_numpy(_linspace(z0, z1, nz)).to(DEV)
    out = torch.zeros((nf, len(modes), nx, nz), dtype=torch.float64, device=DEV)
    r = f0 / fs
    if iq:
        m = torch.zeros(ns, dtype=torch.float64, device=DEV)
        m[0] = 1.0
        m[1:(ns + 1) // 2] = 2.0
        if ns % 2 == 0:
            m[ns // 2] = 1.0
        k = torch.arange(ns, device=DEV, dtype=torch.float64)
        u = torch.fft.ifft(torch.fft.fft(rfs.to(torch.float64)) * m) * torch.exp(-2j * math.pi * f0 * k / fs)
    else:
        u = rfs.to(torch.float64)
    step = max(1, (1 << 24) // (nz * ne))
    off = (torch.arange(ne, device=DEV) * ns)[None, None, :]
    for c0 in range(0, nx, step):
        xp = xs[c0:c0 + step, None, None]
        zp = zs[None, :, None]
        inside = (xp - xe).abs() <= zp / (2.0 * F_NUMBER)
        rx = torch.sqrt((xp - xe) ** 2 + zp * zp)
        count = inside.sum(2).to(torch.float64)
        acc = [{} for _ in range(nf)]
        for a in range(na):
            n = (xp * math.sin(angles[a]) + zp * math.cos(angles[a]) + rx) * (fs / C_MPS)
            kf = torch.floor(n)
            ok = inside & (kf >= 0) & (kf <= ns - 2)
            al = n - kf
            idx = kf.clamp(0, ns - 2).to(torch.int64) + off
            turn = torch.exp(2j * math.pi * r * n) if iq else None
            for f in range(nf):
                flat = u[f, a].reshape(-1)
                v = (1.0 - al) * flat[idx] + al * flat[idx + 1]
                if iq:
                    v = v * turn
                v = torch.where(ok, v, 0.0)
                A = acc[f]

                def add(key, val, A=A):
                    A[key] = A[key] + val if key in A else val

                if "das" in modes or "cf" in modes or "iqdas" in modes:
                    add("s", v.sum(2))
                if "cf" in modes:
                    add("q", (v * v).sum(2))
                if "dmas" in modes:
                    t = torch.sign(v) * v.abs().sqrt()
                    add("dmas", (t.sum(2) ** 2 - v.abs().sum(2)) / 2.0)
                if "pdas" in modes:
                    t = (torch.sign(v) * v.abs() ** (1.0 / pdas_p)).sum(2)
                    add("pdas", torch.sign(t) * t.abs() ** pdas_p)
                if "bbdmas" in modes:
                    g = v.abs().sqrt()
                    t = torch.where(g > 0, v / torch.where(g > 0, g, 1.0), 0.0).sum(2)
                    add("bb", (t / torch.where(count > 0, count, 1.0)) ** 2)
        for f in range(nf):
            A = acc[f]
            for i, mode in enumerate(modes):
                if mode == "das":
                    y = A["s"]
                elif mode == "cf":
                    den = na * count * A["q"]
                    y = torch.where(den > 0, A["s"] ** 2 / torch.where(den > 0, den, 1.0) * A["s"], 0.0)
                elif mode == "iqdas":
                    y = A["s"].abs()
                elif mode == "bbdmas":
                    y = A["bb"].abs()
                else:
                    y = A[mode]
                out[f, i, c0:c0 + step] = y
    return out


def _envelope64(y, band, dz, f0):
    L = y.shape[-1]
    h = torch.zeros(L, dtype=torch.float64, device=y.device)
    h[0] = 1.0
    h[1:(L + 1) // 2] = 2.0
    if L % 2 == 0:
        h[L // 2] = 1.0
    if band:
        f = torch.arange(L, device=y.device, dtype=torch.float64) * C_MPS / (2.0 * L * dz)
        h = torch.where((f >= f0) & (f <= 3.0 * f0), h, 0.0)
        h[0] = 0.0
    return torch.fft.ifft(torch.fft.fft(y) * h).abs()


def _log64(env):
    peak = env.max()
    return torch.where(env > 0, (20.0 * torch.log10(env / peak)).clamp(-70.0, 0.0), -70.0)


def _stage64(y, modes, out, dz, f0):
    """Output stage of images [modes][nx][nz]."""
    if out == "rf":
        return y
    res = []
    for i, m in enumerate(modes.split("+")):
        e = y[i] if m in ("iqdas", "bbdmas") else _envelope64(y[i], m == "dmas", dz, f0)
        res.append(_log64(e) if out == "logdb" else e)
    return torch.stack(res)


def _fk_sizes(ne, ns):
    return 1 << (2 * ns - 1).bit_length(), 1 << (2 * ne - 1).bit_length()


def _fk64(rf, angles, ne, stolt):
    ns, fs, pitch = rf.shape[2], 20e6, 0.3e-3
    nt, nk = _fk_sizes(ne, ns)
    half = nt // 2
    dz = C_MPS / (2.0 * fs)
    x = torch.from_numpy(_elements(ne, pitch)).to(DEV)
    b = torch.arange(half + 1, device=DEV, dtype=torch.float64)
    m = torch.arange(nk, device=DEV)
    X = (torch.where(m < nk // 2, m, m - nk).to(torch.float64) * (nt * dz / (nk * pitch)))[None, :]
    Q = torch.arange(1, half + 1, device=DEV, dtype=torch.float64)[:, None]
    spec = torch.zeros((nt, nk), dtype=torch.complex128, device=DEV)
    for a, th in enumerate(angles):
        s, c = math.sin(th), math.cos(th)
        D = torch.fft.rfft(rf[a].to(torch.float64), n=nt, dim=1)
        D = D * torch.exp(1j * math.pi * b[None, :] * x[:, None] * s / (nt * dz))
        D = torch.fft.fft(D, n=nk, dim=0)
        if stolt:
            beta = math.sqrt(1.0 + c - 0.5 * s * s)
            Qp = (Q - s * X) / beta
            rad = torch.sqrt(X * X + Qp * Qp)
            pos, w = (2.0 / beta) * rad, Qp / (beta * beta * rad)
            ok = (Qp > 0) & (pos >= 0) & (pos < half)
        else:
            den, num = X * s + Q * c, X * X + Q * Q
            pos, w = num / den, (Q * den - 0.5 * num * c) / (den * den)
            ok = (den > 0) & ((2.0 * X - pos * s).abs() <= pos) & (pos >= 0) & (pos < half)
        pos = torch.where(ok, pos, 0.0)
        i0 = torch.floor(pos).to(torch.int64)
        al = pos - i0
        col = m[None, :].expand_as(i0)
        v = (1 - al) * D[col, i0] + al * D[col, (i0 + 1).clamp(max=half)]
        spec[1:half + 1] += torch.where(ok, v * w, 0.0)
    return torch.fft.ifft2(spec)[:ns, :ne].abs().T.contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("frame", "ring", "batch"):
        rf = _frame_inputs(case, seed)
        dz = (case["z1"] - case["z0"]) / max(case["nz"] - 1, 1)
        y = _beamform64(rf, _angles(case["na"]), case["ne"], case["nx"], case["nz"], case["fs"],
                        case["f0"], case["width"], case["z0"], case["z1"], case["modes"],
                        case["pdas_p"])
        return torch.stack([_stage64(v, case["modes"], case["out"], dz, case["f0"]) for v in y])
    if kind in ("uneven", "serve"):
        rfs, angs, per = _mixed_inputs(case, seed)
        res, k = [], 0
        for (nx, nz, na, modes), ang, n in zip(_mixed(case), angs, per):
            y = _beamform64(torch.stack(rfs[k:k + n]), ang, case["ne"], nx, nz, 20e6, 5e6, 19.2e-3,
                            5e-3, 40e-3, modes, 2.0)
            dz = 35e-3 / max(nz - 1, 1)
            im = torch.stack([_stage64(v, modes, case["out"], dz, 5e6) for v in y])
            res.append(im if kind == "serve" else im[0])
            k += n
        return res
    st = prepare(case, seed)
    if kind == "fk":
        img = _fk64(st.rf, st.angles, case["ne"], case["stolt"])
        return _log64(img) if case["out"] == "logdb" else img
    return _log64(_envelope64(st.y.to(torch.float64), case["band"], 35e-3 / (case["nz"] - 1), 5e6))
