// Beamforming of frames that share their plan with no other frame: single calls,
// and the frames of uneven batches (Eq. (1), Sec. II-B; RF combiners).
//
// What such a frame can share is its angles: the receive distance of a (pixel,
// channel) does not depend on the plane wave.  A pipeline stage holds a group of
// channels for up to four angles; per (pixel, channel) the distance's reciprocal
// square root and reciprocal are formed once, and each angle adds its transmit
// term, one fused multiply-add away.  With fewer angles in the group several
// channels are walked at a time instead, so a thread always has about eight
// independent samples in flight (two rows x four angle-channel pairs).
//
// Persistent CTAs of eight consumer warps and a producer warp walk the launch's
// (job, tile) list.  A tile is 32 columns (one per lane) x 16 / SPLIT rows: a
// consumer warp takes two rows (the halves of the paired FP32 instructions) and
// every SPLIT-th channel of a stage; the SPLIT warps of a row pair add up their
// sums through shared memory at the end of an angle group.  Launches with few
// tiles run with SPLIT = 2 or 4: that many times the tiles, each with fewer
// channels per warp, so a small image still fills the chip.
//
// Bound: latency, with no unit saturated: 15.5 instructions per active (pixel, channel,
// angle) for DAS and 18.2 for DMAS of 1-11 angles (19.9 and 24.3 before) fill 59-65 % of
// the issue slots, the FMA pipe 42-48 %, special functions 33 % (DAS) to 55 % (DMAS),
// shared memory 19-45 %, with 23-24 warps per SM.  Scalar instead of paired sums (13 %
// more instructions), or the receive distance as a polynomial without special functions,
// take the same time or longer.
// Measured against the tiles of beamform_kernel that these frames used: whole passes
// of 32 uneven frames 2712 -> 1844 us (1647 with the launches side by side and the ingest
// of today), of one 1024 x 1024 x 128 x 7-angle frame with DAS + DMAS + CF in FP16
// 403 -> 260 us, of a 300 x 384 pDAS frame 73.8 -> 45.6 us (43.1 with dependent
// launches); a 512 x 512 frame of one angle 22.1 -> 18.7 us of beamforming.
#pragma once

#include <limits.h>

#include <algorithm>
#include <type_traits>

#include "../../include/bf.h"
#include "bf_device.cuh"
#include "bf_internal.h"
#include "bf_launch.cuh"

namespace bfi {
namespace {

struct SoloHeader {
    uint64_t full[kSoloStages];   // producer -> consumers: the stage's copies have landed
    uint64_t empty[kSoloStages];  // consumers -> producer: every consumer warp is done with it
    // per staged channel and angle of the group: the address a sample index of zero
    // would have (see SoloAcc::M); one entry more is read ahead
    int4 ent[kSoloStages][kMaxGroup + 1];
    // per row band: the stage's channels (bits) that every pixel of the band counts
    // for every angle of the group [0 .. 7], and those that only some do [8 .. 15]
    uint32_t mask[kSoloStages][2 * kWarps];
    // the tile's delay tables of the stage's angles, written where an angle group
    // starts: integer part and remainder of the column terms [32] and the row
    // terms [16]; kappa z of the rows
    int tK[kSoloStages][kSoloAngles][kTileCols + 16];
    float tF[kSoloStages][kSoloAngles][kTileCols + 16];
    float tZ[kSoloStages][16];
};
constexpr int kSoloHeaderBytes = (int)(sizeof(SoloHeader) + 127) / 128 * 128;

// Sums a warp hands to the others of its row pair: per angle T1 (DMAS) and P1 (pDAS);
// T2 (DMAS), S1 and the squares (CF).  Row pairs, one per lane.
__host__ __device__ constexpr int solo_sums(int na, bool dmas, bool cf, bool pdas)
{
    return na * ((dmas ? 1 : 0) + (pdas ? 1 : 0)) + (dmas ? 1 : 0) + 1 + (cf ? 1 : 0);
}
__host__ __device__ constexpr int solo_exchange_bytes(int split, int na, bool dmas, bool cf, bool pdas)
{
    return split > 1 ? (kWarps - kWarps / split) * solo_sums(na, dmas, cf, pdas) * 32 * 8 : 0;
}

__device__ __forceinline__ void sts_b64(uint32_t a, f32x2_t v)
{
    asm volatile("st.shared.b64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

__device__ __forceinline__ f32x2_t lds_b64(uint32_t a)
{
    f32x2_t v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ int4 lds_int4(uint32_t a)
{
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(a));
    return v;
}

__device__ __forceinline__ void tma_3d(void *dst, const CUtensorMap *map, int x, int y, int z,
                                       uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// Barrier of the `threads` threads of a row band, with an OR over them.
__device__ __forceinline__ bool bar_or(int id, int threads, bool x)
{
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %3, 0;\n\t"
        "barrier.cta.red.or.pred q, %1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"(id), "r"(threads), "r"((unsigned)x)
        : "memory");
    return r != 0;
}

// What a consumer thread carries through a tile of jobs with up to NA angles per
// stage; the two rows in the halves.
template <int NA>
struct SoloAcc {
    f32x2_t Z;      // kappa z
    f32x2_t F[NA];  // remainders of the transmit + depth term, minus 1/2
    // the rounding constant plus the integer part of that term (relative to the
    // tile's first pixel): x + M rounds x and adds the integer part in one addition,
    // and the bits of the sum, times the pair size, plus the channel's entry are the
    // sample pair's address
    f32x2_t M[NA];
    f32x2_t S1, Su2;
    f32x2_t T1[NA], P1[NA];
    f32x2_t T2;  // of all the group's angles, which only enter the image as their sum
    f32x2_t Yd, Yp;
};

// Where a channel that counts partly finds what its test needs.
struct SoloCheck {
    uint32_t rows, rstep;  // its counted rows of the first angle; from angle to angle
    uint32_t win, wstep;   // its window of the first angle; from angle to angle
    uint32_t last;         // offset of a window's last pair
    int r_first;
};

// NCH channels x AN angles into the two pixels of this thread.  CHECK: test each
// pixel's row against the channel's counted rows of each angle, and hold the address
// inside the window; otherwise every pixel of the band counts the channel, so the
// plan's windows hold every index (the planner checks them, two pairs of margin on
// either side of the tile's extremes).
template <int PREC, bool DMAS, bool CF, bool PDAS, int NA, int AN, int NCH, bool CHECK>
__device__ __forceinline__ void solo_channels(SoloAcc<NA> &A, const int4 (&E)[NCH], const float (&D)[NCH],
                                              const SoloCheck &K, float inv_p, bool square)
{
    constexpr uint32_t PB = PairIO<PREC>::kBytes;
    // Channels walked together are added up before they enter the running sums, which so
    // take half or a quarter of the roundings (one angle: sixteen for 64 channels).
    constexpr bool FIRST = NCH > 1;
    f32x2_t sum = 0, roots[AN], proots[AN];
#pragma unroll
    for (int c = 0; c < NCH; ++c) {
        const f32x2_t D2 = pk2(D[c], D[c]);
        float a, b;
        const f32x2_t s = fma2(A.Z, A.Z, D2);
        upk2(s, a, b);
        const f32x2_t r = mul2(s, pk2(rsqrt_approx(a), rsqrt_approx(b)));
        upk2(add2(r, A.Z), a, b);
        const f32x2_t R = pk2(rcp_approx(a), rcp_approx(b));
        const int ent[4] = {E[c].x, E[c].y, E[c].z, E[c].w};
        f32x2_t squares = 0;
#pragma unroll
        for (int k = 0; k < AN; ++k) {
            const f32x2_t x = fma2(D2, R, A.F[k]);
            const f32x2_t m = add2(x, A.M[k]);
            float m0, m1, l0, l1;
            upk2(m, m0, m1);
            upk2(sub2(x, sub2(m, A.M[k])), l0, l1);
            const uint32_t win = K.win + (uint32_t)k * K.wstep;
            const uint32_t p0 = pair_at<PB, CHECK>(m0, (uint32_t)ent[k], win, K.last);
            const uint32_t p1 = pair_at<PB, CHECK>(m1, (uint32_t)ent[k], win, K.last);
            float v0 = PairIO<PREC>::interp(p0, l0);
            float v1 = PairIO<PREC>::interp(p1, l1);
            if (CHECK) {
                const int2 vr = lds_rows(K.rows + (uint32_t)k * K.rstep);
                const unsigned span = (unsigned)(vr.y - vr.x);
                v0 = (unsigned)(K.r_first - vr.x) <= span ? v0 : 0.f;
                v1 = (unsigned)(K.r_first + 1 - vr.x) <= span ? v1 : 0.f;
            }
            const f32x2_t v = pk2(v0, v1);
            if (FIRST)
                sum = c == 0 && k == 0 ? v : add2(sum, v);
            else
                A.S1 = add2(A.S1, v);
            if (DMAS) {
                const f32x2_t q = pk2(copysignf(sqrt_approx(fabsf(v0)), v0),
                                      copysignf(sqrt_approx(fabsf(v1)), v1));
                if (FIRST)
                    roots[k] = c == 0 ? q : add2(roots[k], q);
                else
                    A.T1[k] = add2(A.T1[k], q);
                // a channel's angles first, so that T2 is no longer a sum than per angle
                squares = AN == 1 ? fma2(q, q, A.T2) : k == 0 ? mul2(q, q) : fma2(q, q, squares);
            }
            if (CF)
                A.Su2 = fma2(v, v, A.Su2);
            if (PDAS) {
                const f32x2_t q = pk2(pdas_root(v0, inv_p, square), pdas_root(v1, inv_p, square));
                if (FIRST)
                    proots[k] = c == 0 ? q : add2(proots[k], q);
                else
                    A.P1[k] = add2(A.P1[k], q);
            }
        }
        if (DMAS)
            A.T2 = AN == 1 ? squares : add2(A.T2, squares);
    }
    if (FIRST) {
        A.S1 = add2(A.S1, sum);
#pragma unroll
        for (int k = 0; k < AN; ++k) {
            if (DMAS)
                A.T1[k] = add2(A.T1[k], roots[k]);
            if (PDAS)
                A.P1[k] = add2(A.P1[k], proots[k]);
        }
    }
}

// Resident CTAs per SM the register budget is sized for.  (One angle, 512 x 512 DAS +
// DMAS: 19.5 / 18.7 / 20.7 us at two / three / four; while these jobs ran with the
// registers of four angles, which spilled at three, 24.9.  1024 x 1024 x 128 elements, 7
// angles, DAS + DMAS + CF in FP16, whole pass: 269.5 us at two, 259.5 at three; with a T2
// per angle, which left room for two only, 272.  32 uneven frames 1667 us at two
// throughout, 1647 now, 1660 with a T2 per angle.)
template <bool DMAS, bool CF, bool PDAS, int NA>
constexpr int solo_min_blocks()
{
    if (NA == 1)
        return 3;
    return PDAS && (DMAS || CF) ? 2 : 3;
}

// NA: angles of a stage, 1 (jobs of one angle) or kSoloAngles.
template <int PREC, bool DMAS, bool CF, bool PDAS, int SPLIT, int NA>
__global__ void __launch_bounds__(kThreads + 32, (solo_min_blocks<DMAS, CF, PDAS, NA>()))
    solo_kernel(const BfJob *__restrict__ jobs, const int *__restrict__ tile_prefix, int njobs,
                int total_tiles, int stage_stride, int *__restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    SoloHeader &sh = *reinterpret_cast<SoloHeader *>(smem);
    constexpr int PB = PairIO<PREC>::kBytes;
    constexpr int BANDS = kWarps / SPLIT, TR = 2 * BANDS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int EX = solo_exchange_bytes(SPLIT, NA, DMAS, CF, PDAS);
    auto stage_base = [&](int st) { return smem + kSoloHeaderBytes + EX + (size_t)st * stage_stride; };

    dependents_may_start();
    if (threadIdx.x == 0) {
        for (int st = 0; st < kSoloStages; ++st) {
            mbar_init(&sh.full[st], 1);
            mbar_init(&sh.empty[st], kWarps);
        }
        mbar_fence_init();
    }
    __syncthreads();

    // Stage layout: float dx^2 [G][32], counted rows short2 [angle][G][32], windows
    // [angle][G][wmax]; angle group k holds the angles k na / ngr .. (k + 1) na / ngr - 1.
    if (warp == kWarps) {
        // ================= producer warp: a step's record (masks, window starts) into
        // the header, its tables and windows by tensor copies.  A copy costs the
        // issuing warp about 65 cycles, so one copy brings the windows of a run of
        // (up to four) adjacent channels, which start at the same pair.
        wait_for_producer();  // the staged pairs (and the deadlines start here)
        unsigned r = 0;
        int mapped = -1;  // the job whose maps were acquired last
        for (int tg = blockIdx.x; tg < total_tiles; tg += gridDim.x) {
            const unsigned long long deadline = global_ns() + kWaitNs;
            const int jb = find_job(tile_prefix, njobs, tg);
            const BfJob *J = jobs + jb;
            const int tile = tg - __ldg(tile_prefix + jb);
            const int nx = J->nx, nz = J->nz, ne = J->ne, G = J->group, wmax = J->wmax, na = J->na;
            const int tiles_x = J->tiles_x, ntiles = tiles_x * J->tiles_z;
            const int tx = tile % tiles_x, tz = tile / tiles_x;
            const int ngr = J->ang_groups, ngroups = (ne + G - 1) / G, steps = ngr * ngroups;
            const int amax = (na + ngr - 1) / ngr, box = J->box, run = J->run;
            const CUtensorMap *rf_map = J->rf_map;
            if (jb != mapped)
                maps_acquire(J);
            mapped = jb;
            // this lane's run of channels and angle, its word of the step's record
            const int runs = G / run, kq = lane / runs, cq = lane - kq * runs;
            const int words = solo_record_words(amax, runs);
            const int *__restrict__ rec = J->wtab + (size_t)tile * words;
            const size_t rec_step = (size_t)ntiles * words;
            const int cx = min(tx * kTileCols + lane, nx - 1), rz = min(tz * TR + lane, nz - 1);
            const unsigned table = (unsigned)G * kTileCols * 4;
            int w0 = kNoWindow, mk = 0;
            auto record = [&](int s) {
                w0 = lane < amax * runs ? __ldg(rec + s * rec_step + 2 * kWarps + lane) : kNoWindow;
                mk = lane < 2 * kWarps ? __ldg(rec + s * rec_step + lane) : 0;
            };
            record(0);
            int ag = 0, g = 0, kref = 0;
            for (int s = 0; s < steps; ++s, ++r) {
                const int st = (int)(r % kSoloStages);
                const unsigned use = r / kSoloStages;
                const int i0 = g * G, a0 = ag * na / ngr, an = (ag + 1) * na / ngr - a0;
                const int w = w0, m = mk;
                int ck[NA] = {}, rk[NA] = {};
                float cf[NA] = {}, rf[NA] = {}, z = 0.f;
                if (g == 0) {
                    z = __ldg(J->rowZ + rz);
#pragma unroll
                    for (int k = 0; k < NA; ++k)
                        if (k < an) {
                            ck[k] = __ldg(J->colK + (a0 + k) * nx + cx);
                            cf[k] = __ldg(J->colF + (a0 + k) * nx + cx);
                            rk[k] = __ldg(J->rowK + (a0 + k) * nz + rz);
                            rf[k] = __ldg(J->rowF + (a0 + k) * nz + rz);
                        }
                    // integer parts relative to the tile's first pixel, per angle
#pragma unroll
                    for (int k = 0; k < NA; ++k) {
                        const int ref = __shfl_sync(0xffffffffu, ck[k] + rk[k], 0);
                        ck[k] -= ref;
                        kref = kq == k ? ref : kref;
                    }
                }
                if (s + 1 < steps)
                    record(s + 1);  // in flight while this step waits
                if (use > 0 && !mbar_wait(&sh.empty[st], (use - 1) & 1u, deadline, err))
                    return;  // the consumers' waits run out too
                if (g == 0) {
#pragma unroll
                    for (int k = 0; k < NA; ++k)
                        if (k < an) {
                            sh.tK[st][k][lane] = ck[k];
                            sh.tF[st][k][lane] = cf[k];
                            if (lane < TR) {
                                sh.tK[st][k][kTileCols + lane] = rk[k];
                                sh.tF[st][k][kTileCols + lane] = rf[k];
                            }
                        }
                    if (lane < TR)
                        sh.tZ[st][lane] = z;
                }
                unsigned char *base = stage_base(st);
                const uint32_t wins = smem_u32(base) + (uint32_t)(1 + amax) * table;
                if (lane < amax * runs)
                    for (int q = 0; q < run; ++q)
                        reinterpret_cast<int *>(&sh.ent[st][cq * run + q])[kq] =
                            (int)window_entry(
                                wins + (uint32_t)((kq * G + cq * run + q) * wmax * PB), w, kref, PB);
                if (lane < 2 * kWarps)
                    sh.mask[st][lane] = (uint32_t)m;
                const bool mine = lane < an * runs && w != kNoWindow;
                const unsigned nwin = __popc(__ballot_sync(0xffffffffu, mine));
                // the counted rows are read only for channels that count partly
                const bool parts = __any_sync(0xffffffffu, lane >= kWarps && m != 0);
                // everything written above is read by the consumers after the full barrier
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive_expect_tx(&sh.full[st], nwin * (unsigned)(run * wmax * PB) + table +
                                                            (parts ? table * (unsigned)amax : 0u));
                    tma_2d(base, J->dx2_map, tx * kTileCols, i0, &sh.full[st]);
                    if (parts)
                        tma_3d(base + table, J->valid_map, tx * kTileCols, i0, a0, &sh.full[st]);
                }
                __syncwarp();
                if (mine) {
                    unsigned char *dst = base + (size_t)(1 + amax) * table +
                                         (size_t)(kq * G + cq * run) * wmax * PB;
                    const int row = (a0 + kq) * ne + i0 + cq * run;
                    for (int off = 0; off < wmax; off += box)
                        tma_2d(dst + (size_t)off * PB, rf_map, w + off, row, &sh.full[st]);
                }
                if (++g == ngroups) {
                    g = 0;
                    ++ag;
                }
            }
        }
        return;
    }

    // ================= consumer warps
    wait_for_producer();  // so that their deadlines do not run while the pairs are made
    const int band = warp % BANDS, part = warp / BANDS;
    constexpr int NV = solo_sums(NA, DMAS, CF, PDAS);
    // sums handed over by warp part > 0 of this band: value v at ex(part) + 256 v
    auto ex = [&](int p) {
        return smem_u32(smem + kSoloHeaderBytes) +
               (uint32_t)((((p - 1) * BANDS + band) * NV * 32 + lane) * 8);
    };
    unsigned r = 0;
    for (int tg = blockIdx.x; tg < total_tiles; tg += gridDim.x) {
        const unsigned long long deadline = global_ns() + kWaitNs;
        const int jb = find_job(tile_prefix, njobs, tg);
        const BfJob *J = jobs + jb;
        const int tile = tg - __ldg(tile_prefix + jb);
        const int nx = J->nx, nz = J->nz, na = J->na, ne = J->ne, G = J->group, wmax = J->wmax;
        const int tx = tile % J->tiles_x, tz = tile / J->tiles_x;
        const int ngr = J->ang_groups, ngroups = (ne + G - 1) / G, steps = ngr * ngroups;
        const int amax = (na + ngr - 1) / ngr;
        // columns beyond the grid repeat its last one, so that their indices stay in
        // the windows too
        const int col = min(lane, nx - 1 - tx * kTileCols);
        const int r_first = tz * TR + 2 * band;
        const float pdas_p = J->pdas_p, inv_p = J->pdas_inv_p;
        const bool square = pdas_p == 2.0f;  // uniform over the job
        const uint32_t wbytes = (uint32_t)(wmax * PB), rstep = (uint32_t)(G * kTileCols * 4),
                       wstep = (uint32_t)G * wbytes;
        const f32x2_t zero2 = pk2(0.f, 0.f);
        SoloAcc<NA> A;
        A.Z = A.S1 = A.T2 = A.Su2 = A.Yd = A.Yp = zero2;
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            A.F[k] = A.M[k] = A.T1[k] = A.P1[k] = zero2;
        }
        bool dead = false;
        int g = 0, ag = 0;
#pragma unroll 1
        for (int s = 0; s < steps; ++s, ++r) {
            const int st = (int)(r % kSoloStages);
            const unsigned use = r / kSoloStages;
            const int an = NA == 1 ? 1 : (ag + 1) * na / ngr - ag * na / ngr;
            if (!dead)
                dead = !__all_sync(0xffffffffu, mbar_wait(&sh.full[st], use & 1u, deadline, err));
            if (dead && SPLIT == 1)
                return;  // warp-uniform: a bounded wait ran out (error bit set)
            if (!dead) {
                if (g == 0) {  // the angle group's delay tables
                    A.T2 = zero2;
                    A.Z = pk2(sh.tZ[st][2 * band], sh.tZ[st][2 * band + 1]);
#pragma unroll
                    for (int k = 0; k < NA; ++k)
                        if (k < an) {
                            const int ck = sh.tK[st][k][lane] + kRoundBits;
                            const float cf = sh.tF[st][k][lane];
                            const int *tk = &sh.tK[st][k][kTileCols + 2 * band];
                            const float *tf = &sh.tF[st][k][kTileCols + 2 * band];
                            A.M[k] = pk2(__int_as_float(ck + tk[0]), __int_as_float(ck + tk[1]));
                            A.F[k] = pk2(cf + tf[0] - 0.5f, cf + tf[1] - 0.5f);
                            A.T1[k] = A.P1[k] = zero2;
                        }
                }
                const uint32_t base = smem_u32(stage_base(st));
                const uint32_t d2b = base + (uint32_t)col * 4, wins = base + (uint32_t)(1 + amax) * rstep;
                const uint32_t entb = smem_u32(&sh.ent[st][0]);
                SoloCheck K{d2b + rstep, rstep, wins, wstep, wbytes - (uint32_t)PB, r_first};
                // the next run of adjacent channels of a mask: this warp's share of it
                auto next_run = [&](uint32_t &m, int &n) {
                    const int lo = __ffs(m) - 1, len = __ffs(~(m >> lo)) - 1;
                    m &= ~(((1u << len) - 1u) << lo);
                    const int a = len * part / SPLIT;
                    n = len * (part + 1) / SPLIT - a;
                    return lo + a;
                };
                auto walk = [&](auto an_c, auto nch_c) {
                    constexpr int AN = decltype(an_c)::value, NCH = decltype(nch_c)::value;
                    uint32_t m = sh.mask[st][band];
                    int n;
                    while (m) {
                        const int c = next_run(m, n);
                        uint32_t pe = entb + (uint32_t)c * 16u, pd = d2b + (uint32_t)c * (kTileCols * 4);
                        auto step = [&](auto nch) {
                            constexpr int N = decltype(nch)::value;
                            int4 E[N];
                            float D[N];
#pragma unroll
                            for (int q = 0; q < N; ++q) {
                                if (AN == 1)
                                    E[q] = make_int4(__float_as_int(lds_f32(pe + 16u * q)), 0, 0, 0);
                                else
                                    E[q] = lds_int4(pe + 16u * q);
                                D[q] = lds_f32(pd + (uint32_t)(kTileCols * 4 * q));
                            }
                            solo_channels<PREC, DMAS, CF, PDAS, NA, AN, N, false>(A, E, D, K, inv_p, square);
                            pe += 16u * N;
                            pd += (uint32_t)(kTileCols * 4 * N);
                        };
                        if constexpr (NCH > 1) {
#pragma unroll 1
                            for (; n >= NCH; n -= NCH)
                                step(nch_c);
#pragma unroll 1
                            for (; n > 0; --n)
                                step(std::integral_constant<int, 1>());
                        } else if (n > 0) {
                            // the next channel's entry and distance read ahead
                            int4 E[1] = {lds_int4(pe)};
                            float D[1] = {lds_f32(pd)};
#pragma unroll 1
                            for (; n > 0; --n) {
                                pe += 16u;
                                pd += (uint32_t)(kTileCols * 4);
                                const int4 e = lds_int4(pe);
                                const float d = lds_f32(pd);
                                solo_channels<PREC, DMAS, CF, PDAS, NA, AN, 1, false>(A, E, D, K, inv_p,
                                                                                      square);
                                E[0] = e;
                                D[0] = d;
                            }
                        }
                    }
                    m = sh.mask[st][kWarps + band];
                    while (m) {
                        int c = next_run(m, n);
#pragma unroll 1
                        for (; n > 0; --n, ++c) {
                            const int4 E[1] = {lds_int4(entb + (uint32_t)c * 16u)};
                            const float D[1] = {lds_f32(d2b + (uint32_t)c * (kTileCols * 4))};
                            SoloCheck Kc = K;
                            Kc.rows += (uint32_t)c * (kTileCols * 4);
                            Kc.win += (uint32_t)c * wbytes;
                            solo_channels<PREC, DMAS, CF, PDAS, NA, AN, 1, true>(A, E, D, Kc, inv_p,
                                                                                 square);
                        }
                    }
                };
                if constexpr (NA == 1) {
                    walk(std::integral_constant<int, 1>(), std::integral_constant<int, 4>());
                } else switch (an) {
                case 1: walk(std::integral_constant<int, 1>(), std::integral_constant<int, 4>()); break;
                case 2: walk(std::integral_constant<int, 2>(), std::integral_constant<int, 2>()); break;
                case 3: walk(std::integral_constant<int, 3>(), std::integral_constant<int, 1>()); break;
                default: walk(std::integral_constant<int, 4>(), std::integral_constant<int, 1>()); break;
                }
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(&sh.empty[st]);
            }
            if (++g < ngroups)
                continue;
            g = 0;
            ++ag;
            if constexpr (SPLIT > 1) {
                // the band's sums of this angle group (and of the tile) into part 0
                const bool last = ag == ngr;
                if (DMAS || PDAS || last) {
                    if (part > 0 && !dead) {
                        uint32_t o = ex(part);
                        auto put = [&](f32x2_t v) {
                            sts_b64(o, v);
                            o += 256;
                        };
#pragma unroll
                        for (int k = 0; k < NA; ++k) {
                            if (DMAS)
                                put(A.T1[k]);
                            if (PDAS)
                                put(A.P1[k]);
                        }
                        if (DMAS)
                            put(A.T2);
                        put(A.S1);
                        if (CF)
                            put(A.Su2);
                    }
                    // every warp of the band learns of a wait that ran out in one of them
                    if (bar_or(1 + band, 32 * SPLIT, dead))
                        return;
                    if (part == 0) {
#pragma unroll
                        for (int p = 1; p < SPLIT; ++p) {
                            uint32_t o = ex(p);
                            auto get = [&](f32x2_t &v) {
                                v = add2(v, lds_b64(o));
                                o += 256;
                            };
#pragma unroll
                            for (int k = 0; k < NA; ++k) {
                                if (DMAS)
                                    get(A.T1[k]);
                                if (PDAS)
                                    get(A.P1[k]);
                            }
                            if (DMAS)
                                get(A.T2);
                            if (last) {
                                get(A.S1);
                                if (CF)
                                    get(A.Su2);
                            }
                        }
                    }
                    bar_or(1 + band, 32 * SPLIT, false);  // the area is free again
                }
            }
            if (DMAS) {
                A.Yd = fma2(pk2(-0.5f, -0.5f), A.T2, A.Yd);
#pragma unroll
                for (int k = 0; k < NA; ++k)
                    if (k < an)
                        A.Yd = fma2(mul2(pk2(0.5f, 0.5f), A.T1[k]), A.T1[k], A.Yd);
            }
            if (PDAS) {  // Eq. (3) per angle, then the coherent sum
#pragma unroll
                for (int k = 0; k < NA; ++k)
                    if (k < an) {
                        float a, b;
                        upk2(A.P1[k], a, b);
                        A.Yp = add2(A.Yp, pk2(copysignf(powf(fabsf(a), pdas_p), a),
                                              copysignf(powf(fabsf(b), pdas_p), b)));
                    }
            }
        }
        const int ix = tx * kTileCols + lane;
        if (ix >= nx || r_first >= nz || part > 0)
            continue;
        const int modes = J->modes;
        const float scale = J->out_scale;
        const size_t plane = (size_t)nx * nz, o = (size_t)ix * nz + r_first;
        float *__restrict__ y = J->y;
        const bool two = r_first + 1 < nz;
        auto store = [&](float a, float b) {
            if (two && (reinterpret_cast<unsigned long long>(y + o) & 7) == 0) {
                *reinterpret_cast<float2 *>(y + o) = make_float2(a, b);
            } else {
                y[o] = a;
                if (two)
                    y[o + 1] = b;
            }
            y += plane;
        };
        float s0, s1, a, b;
        upk2(A.S1, s0, s1);
        if (modes & BF_DAS)
            store(s0 * scale, s1 * scale);
        if (modes & BF_DMAS) {
            upk2(A.Yd, a, b);
            store(a * scale, b * scale);
        }
        if (modes & BF_CF) {
            upk2(A.Su2, a, b);
            const float d0 = (float)na * (float)__ldg(J->apcnt + o) * a;
            const float d1 = (float)na * (float)__ldg(J->apcnt + o + (two ? 1 : 0)) * b;
            store(d0 > 0.f ? (s0 * s0 / d0) * s0 * scale : 0.f,
                  d1 > 0.f ? (s1 * s1 / d1) * s1 * scale : 0.f);
        }
        if (modes & BF_PDAS) {
            upk2(A.Yp, a, b);
            store(a * scale, b * scale);
        }
    }
}

template <int PREC, bool DMAS, bool CF, bool PDAS, int SPLIT, int NA>
cudaError_t launch_t(const BfJob *jobs, const int *prefix, int njobs, int tiles, size_t smem, int *err,
                     cudaStream_t st)
{
    auto k = solo_kernel<PREC, DMAS, CF, PDAS, SPLIT, NA>;
    int sms = 0, occ = 0;
    cudaError_t e = kernel_setup((const void *)k, smem, kThreads + 32, true, &sms, &occ);
    if (e != cudaSuccess)
        return e;
    const int grid = std::max(1, std::min(tiles, std::max(occ, 1) * sms));
    const int stride = (int)((smem - kSoloHeaderBytes - solo_exchange_bytes(SPLIT, NA, DMAS, CF, PDAS)) /
                             kSoloStages);
    // a launch of one wave starts under the ingest kernel's last CTAs (in larger ones
    // the early CTAs would take the SMs from the kernel they wait for)
    const bool dependent = tiles <= std::max(occ, 1) * sms;
    if (dependent) {
        smem = spread_smem(smem, grid, sms);
        e = kernel_setup((const void *)k, smem, kThreads + 32, true, &sms, nullptr);
        if (e != cudaSuccess)
            return e;
    }
    return launch_kernel(k, dim3((unsigned)grid), kThreads + 32, smem, dependent, st, jobs, prefix, njobs,
                         tiles, stride, err);
}

template <int PREC, int SPLIT, int NA>
cudaError_t launch_v(const BfJob *j, const int *pf, int njobs, int tiles, size_t smem, int variant,
                     int *err, cudaStream_t st)
{
    switch (variant & (BF_DMAS | BF_CF | BF_PDAS)) {
    case 0: return launch_t<PREC, false, false, false, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    case BF_DMAS: return launch_t<PREC, true, false, false, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    case BF_CF: return launch_t<PREC, false, true, false, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    case BF_DMAS | BF_CF:
        return launch_t<PREC, true, true, false, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    case BF_PDAS: return launch_t<PREC, false, false, true, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    case BF_DMAS | BF_PDAS:
        return launch_t<PREC, true, false, true, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    case BF_CF | BF_PDAS:
        return launch_t<PREC, false, true, true, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    default: return launch_t<PREC, true, true, true, SPLIT, NA>(j, pf, njobs, tiles, smem, err, st);
    }
}

template <int PREC, int NA>
cudaError_t launch_p(const BfJob *j, const int *pf, int njobs, int tiles, size_t smem, int variant,
                     int split, int *err, cudaStream_t st)
{
    if (split == 4)
        return launch_v<PREC, 4, NA>(j, pf, njobs, tiles, smem, variant, err, st);
    if (split == 2)
        return launch_v<PREC, 2, NA>(j, pf, njobs, tiles, smem, variant, err, st);
    return launch_v<PREC, 1, NA>(j, pf, njobs, tiles, smem, variant, err, st);
}

}  // namespace

// One translation unit per storage precision instantiates these.
#define BF_SOLO_INSTANTIATE(NAME, PREC)                                                             \
    cudaError_t NAME(const BfJob *jobs_dev, const int *tile_prefix_dev, int njobs, int total_tiles, \
                     size_t smem_bytes, int variant, int split, int ang, int *err_dev,              \
                     cudaStream_t stream)                                                           \
    {                                                                                               \
        return ang == 1 ? launch_p<PREC, 1>(jobs_dev, tile_prefix_dev, njobs, total_tiles,          \
                                            smem_bytes, variant, split, err_dev, stream)            \
                        : launch_p<PREC, kSoloAngles>(jobs_dev, tile_prefix_dev, njobs,             \
                                                      total_tiles, smem_bytes, variant, split,      \
                                                      err_dev, stream);                             \
    }

}  // namespace bfi
