// Envelopes of image columns, two columns per transform of sixteen points per
// thread (bf_fft16.cuh); shared by the envelope kernel and the allocation-free stage.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bf_fft16.cuh"
#include "bf_internal.h"

namespace bfi {
namespace {

__device__ __forceinline__ void red_max_global(unsigned *p, unsigned v)
{
    asm volatile("red.global.max.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Spectral factors from a plan's tables ([q][u], see EnvJob).
template <int T>
struct TableFactors {
    const float *__restrict__ gr, *__restrict__ gh;
    __device__ __forceinline__ float real(int u, int q) const { return __ldg(gr + q * T + u); }
    __device__ __forceinline__ float imag(int u, int q) const { return __ldg(gh + q * T + u); }
};

// The same for a power-of-two depth from the bin number: 1 / M inside the band lo ..
// hi of |k| (all bins without one), times -sgn(k) for the Hilbert transform.
template <int LG>
struct MaskFactors {
    int lo, hi;
    bool band;
    __device__ __forceinline__ float real(int u, int q) const
    {
        const int k = fft16_bin(LG, u, q), ka = 2 * k <= (1 << LG) ? k : (1 << LG) - k;
        return !band || (ka >= lo && ka <= hi) ? 1.f / (float)(1 << LG) : 0.f;
    }
    __device__ __forceinline__ float imag(int u, int q) const
    {
        const int k = fft16_bin(LG, u, q);
        const float r = real(u, q);
        return k == 0 || 2 * k == (1 << LG) ? 0.f : 2 * k < (1 << LG) ? -r : r;
    }
};

// Magnitude where the sum of squares leaves the range it can be formed in.
__device__ __noinline__ float hypot_far(float a, float b) { return hypotf(a, b); }

// The root of the sum of squares: the special-function unit's reciprocal root and one
// Newton step with the residual in a fused multiply-add, about half a unit in the last place.
__device__ __forceinline__ float magnitude(float q, float a, float b)
{
    if (!(q > 1e-36f && q < 3e38f))
        return hypot_far(a, b);
    const float y = rsqrtf(q), s = q * y;
    return fmaf(fmaf(-s, s, q), 0.5f * y, s);
}

// Envelopes of the column pairs pair0, pair0 + 1, ... of one image, one pair per
// T threads (C = THREADS / T pairs per CTA), as one complex column a + i b; returns
// this thread's largest envelope.
// Depths that are a power of two are transformed as they are (M = nz); any other
// depth nz convolves the column with the mask's impulse response of period nz,
// unrolled to 2 nz - 1 lags, in a transform of length M >= 2 nz - 1.  Either
// way the spectrum is multiplied by real tables (gr: the band-passed column, a
// real even response; gh: i gh its Hilbert transform, a real odd one), with the
// inverse's 1 / M in them: one forward transform and one inverse, or two for the
// band-passed image, serve two columns.  Convolved columns are brought to one magnitude
// first (pair_down), so that a quiet column keeps its own precision beside a loud one;
// power-of-two depths share as they are, like the warp kernel.  (Bluestein's four transforms per single
// column, which this replaced: 39.4 us of a 64 x 1750 image's pass, 732 us of the
// pass of 32 uneven images of 64-1024 rows; by the whole passes 47.7 -> 30.7 us
// and 3345 -> 2712 us.)  Bound: latency of the exchanges at small
// image counts, shared-memory traffic and FP32 issue about equally at large ones.
template <int LG, bool CONV, int THREADS, Twiddles TW, class Factors>
__device__ __forceinline__ float envelope_pairs(const float *__restrict__ y, float *__restrict__ env,
                                                int nx, int nz_in, int pair0, bool band,
                                                const float2 *tab, const Factors &G, uint32_t bufs,
                                                uint32_t hold)
{
    using F = Fft16<LG, TW>;
    constexpr int T = F::T;
    const int grp = threadIdx.x / T;
    const F f{bufs + (uint32_t)(grp * fft16_buf_bytes(LG)), tab, (int)threadIdx.x % T, 1 + grp};
    const uint32_t slot = hold + 8u * threadIdx.x;  // value r at slot + 8 THREADS r
    const int nz = CONV ? nz_in : F::M;
    const int ca = 2 * (pair0 + grp), cb = ca + 1;
    const bool has_a = ca < nx, has_b = cb < nx;
    const float *__restrict__ ya = y + (size_t)ca * nz;
    const float *__restrict__ yb = ya + nz;
    float2 v[16];
    constexpr int JN = CONV ? 8 : 16;  // M >= 2 nz - 1: nothing from M / 2 on
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        v[j] = make_float2(0.f, 0.f);
        if (j < JN) {
            const int n = f.u + j * T;
            const bool in = !CONV || n < nz;
            if (in && has_a)
                v[j].x = __ldcs(ya + n);
            if (in && has_b)
                v[j].y = __ldcs(yb + n);
        }
    }
    uint2 top = make_uint2(0u, 0u);
    if constexpr (CONV) {
#pragma unroll
        for (int j = 0; j < JN; ++j) {
            top.x = max(top.x, __float_as_uint(fabsf(v[j].x)));
            top.y = max(top.y, __float_as_uint(fabsf(v[j].y)));
        }
        top = f.pair_max(top.x, top.y);
        const float da = pair_down(top.x), db = pair_down(top.y);
#pragma unroll
        for (int j = 0; j < JN; ++j)
            v[j] = make_float2(v[j].x * da, v[j].y * db);
    }
    const float ua = CONV ? pair_up(top.x) : 1.f, ub = CONV ? pair_up(top.y) : 1.f;
    // a column with infinities or NaNs has no transform, and takes no part in its neighbour's
    const bool bad_a = CONV && top.x >= 0x7f800000u, bad_b = CONV && top.y >= 0x7f800000u;
    if (!band) {
#pragma unroll
        for (int j = 0; j < JN; ++j)
            sts2(slot + 8u * THREADS * j, v[j]);  // the columns themselves
    }
    if (bad_a || bad_b) {
#pragma unroll
        for (int j = 0; j < JN; ++j)
            v[j] = make_float2(bad_a ? 0.f : v[j].x, bad_b ? 0.f : v[j].y);
    }
    f.template forward<CONV>(v);
#pragma unroll 1
    for (int it = band ? 0 : 1; it < 2; ++it) {
        if (it == 0) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float r = G.real(f.u, q), h = G.imag(f.u, q);
                sts2(slot + 8u * THREADS * q, make_float2(-v[q].y * h, v[q].x * h));
                v[q] = make_float2(v[q].x * r, v[q].y * r);
            }
        } else if (!band) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float h = G.imag(f.u, q);
                v[q] = make_float2(-v[q].y * h, v[q].x * h);
            }
        }
        f.inverse(v);
        if (it == 0) {  // the band-passed columns kept, their Hilbert spectrum next
            // the second inverse writes its first level's addresses, which other threads
            // read in the last level of this one
            f.sync();
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const float2 t = lds2(slot + 8u * THREADS * q);
                sts2(slot + 8u * THREADS * q, v[q]);
                v[q] = t;
            }
        }
    }
    if (bad_a || bad_b) {
        const float nan = __int_as_float(0x7fffffff);
#pragma unroll
        for (int j = 0; j < JN; ++j)
            v[j] = make_float2(bad_a ? nan : v[j].x, bad_b ? nan : v[j].y);
    }
    float lmax = 0.f;
    float *__restrict__ oa = env + (size_t)ca * nz;
    float *__restrict__ ob = oa + nz;
#pragma unroll
    for (int j = 0; j < JN; ++j) {
        const int n = f.u + j * T;
        const float2 r = lds2(slot + 8u * THREADS * j);
        const float2 q = c_sqsum(r, v[j]);
        if (CONV && n >= nz)
            continue;
        if (has_a) {
            const float e = magnitude(q.x, r.x, v[j].x) * ua;
            __stcg(oa + n, e);
            lmax = fmaxf(lmax, e);
        }
        if (has_b) {
            const float e = magnitude(q.y, r.y, v[j].y) * ub;
            __stcg(ob + n, e);
            lmax = fmaxf(lmax, e);
        }
    }
    return lmax;
}

}  // namespace
}  // namespace bfi
