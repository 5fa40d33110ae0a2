// Transforms of length 2^LG, 32 <= 2^LG <= 8192, with sixteen points per thread
// held in registers: the building block of the envelope kernels.
//
// A transform of M = 2^LG points is run by T = M / 16 threads.  Thread u starts
// with x[u + j T], j < 16.  Forward, a level of (sub-)length 2^L takes 16-point
// DFTs across the stride S = 2^(L-4), multiplies output k by W_(2^L)^(t k)
// (t = u mod S) and leaves sixteen independent sub-sequences of length 2^(L-4);
// the last level (2, 4, 8 or 16 points, contiguous) ends it.  The spectrum stays
// in that digit-reversed order: register q of thread u holds bin
// fft16_bin(LG, u, q).  The inverse runs the levels backwards from there and
// ends with x[u + j T] again, so no pass only reorders.
//
// Between two levels the sixteen values go through shared memory once: every
// level writes the addresses its thread read, so one barrier per exchange is
// enough and one buffer serves both directions.  That holds from a transform to
// the next one, too, if the next runs the other way (it starts at the level the
// first ended with); two transforms one after the other in the same direction, or
// anything else stored in the buffer, need a barrier (sync) between them.  Element
// p lies at p + p / 16 (float2): every level's accesses of a half warp then fall on distinct banks.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bf_fft.cuh"
#include "bf_internal.h"

namespace bfi {

// cos, sin of 2 pi e / 32 for e < 16
static __device__ __constant__ float2 kW32[16] = {
    {1.000000000e+00f, 0.000000000e+00f},  {9.807852804e-01f, 1.950903220e-01f},
    {9.238795325e-01f, 3.826834324e-01f},  {8.314696123e-01f, 5.555702330e-01f},
    {7.071067812e-01f, 7.071067812e-01f},  {5.555702330e-01f, 8.314696123e-01f},
    {3.826834324e-01f, 9.238795325e-01f},  {1.950903220e-01f, 9.807852804e-01f},
    {0.000000000e+00f, 1.000000000e+00f},  {-1.950903220e-01f, 9.807852804e-01f},
    {-3.826834324e-01f, 9.238795325e-01f}, {-5.555702330e-01f, 8.314696123e-01f},
    {-7.071067812e-01f, 7.071067812e-01f}, {-8.314696123e-01f, 5.555702330e-01f},
    {-9.238795325e-01f, 3.826834324e-01f}, {-9.807852804e-01f, 1.950903220e-01f}};

// What rounding took from them.
static __device__ __constant__ float2 kW32Lo[16] = {
    {0.000000000e+00f, 0.000000000e+00f}, {2.973947311e-08f, -1.670471539e-09f},
    {2.830748969e-08f, 6.223350724e-09f}, {1.687026341e-08f, -1.176952136e-08f},
    {1.210161749e-08f, 1.210161749e-08f}, {-1.176952136e-08f, 1.687026341e-08f},
    {6.223350724e-09f, 2.830748969e-08f}, {-1.670471428e-09f, 2.973947311e-08f},
    {0.000000000e+00f, 0.000000000e+00f}, {1.670471539e-09f, 2.973947311e-08f},
    {-6.223350724e-09f, 2.830748969e-08f}, {1.176952136e-08f, 1.687026341e-08f},
    {-1.210161749e-08f, 1.210161749e-08f}, {-1.687026341e-08f, -1.176952136e-08f},
    {-2.830748969e-08f, 6.223351168e-09f}, {-2.973947311e-08f, -1.670471095e-09f}};

// Complex add / subtract as one paired FP32 instruction (Blackwell f32x2):
// the real and imaginary parts of a float2 sit in a register pair.
static __device__ __forceinline__ float2 c_add(float2 a, float2 b)
{
    unsigned long long ra, rb, rc;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rc) : "l"(ra), "l"(rb));
    float2 c;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c.x), "=f"(c.y) : "l"(rc));
    return c;
}

static __device__ __forceinline__ float2 c_sub(float2 a, float2 b)
{
    unsigned long long ra, rb, rc;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(rc) : "l"(ra), "l"(rb));
    float2 c;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c.x), "=f"(c.y) : "l"(rc));
    return c;
}

// (a.x^2 + b.x^2, a.y^2 + b.y^2): per half b^2 rounded, then one FMA.
static __device__ __forceinline__ float2 c_sqsum(float2 a, float2 b)
{
    unsigned long long ra, rb, rc;
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("mul.rn.f32x2 %0, %1, %1;" : "=l"(rc) : "l"(rb));
    asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(rc) : "l"(ra), "l"(rc));
    float2 c;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c.x), "=f"(c.y) : "l"(rc));
    return c;
}

// Square root on the special-function unit (relative error about one unit in
// the last place, far inside the envelope's tolerance).
static __device__ __forceinline__ float sqrt_fast(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// s * a + b with s a scalar (both halves), as one paired FMA.
static __device__ __forceinline__ float2 c_sfma(float s, float2 a, float2 b)
{
    unsigned long long rs, ra, rb, rc;
    asm("mov.b64 %0, {%1, %1};" : "=l"(rs) : "f"(s));
    asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rc) : "l"(rs), "l"(ra), "l"(rb));
    float2 c;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(c.x), "=f"(c.y) : "l"(rc));
    return c;
}

// a * (w + l): a twiddle in two parts, w rounded to FP32 and l what the rounding took.
// The rounding of the twiddles is half of a transform's error; with l the product keeps
// only its own.
static __device__ __forceinline__ float2 cmul_fine(float2 a, float2 w, float2 l)
{
    const float cr = fmaf(a.x, l.x, -a.y * l.y), ci = fmaf(a.x, l.y, a.y * l.x);
    return make_float2(fmaf(a.x, w.x, fmaf(-a.y, w.y, cr)), fmaf(a.x, w.y, fmaf(a.y, w.x, ci)));
}

// b * W_32^e (INV: conjugate), W_32 = exp(-2 pi i / 32), 0 <= e < 32; e is a
// compile-time constant wherever this is used (quarter turns are swaps).  FINE: the
// factor in two parts.
template <bool INV, bool FINE = false>
static __device__ __forceinline__ float2 w32mul(float2 b, int e)
{
    if (e >= 16) {  // W_32^16 = -1
        b = make_float2(-b.x, -b.y);
        e -= 16;
    }
    if (e == 0)
        return b;
    if (e == 8)
        return INV ? make_float2(-b.y, b.x) : make_float2(b.y, -b.x);
    const float2 w = kW32[e];
    const float s = INV ? w.y : -w.y;
    if constexpr (FINE)
        return cmul_fine(b, make_float2(w.x, s),
                         make_float2(kW32Lo[e].x, INV ? kW32Lo[e].y : -kW32Lo[e].y));
    return make_float2(b.x * w.x - b.y * s, b.x * s + b.y * w.x);
}

// 4-point DFT in place: y_k = sum_n x_n W_4^(n k), W_4 = -i (INV: +i).
template <bool INV>
static __device__ __forceinline__ void dft4(float2 &a, float2 &b, float2 &c, float2 &d)
{
    const float2 t0 = c_add(a, c), t1 = c_sub(a, c), t2 = c_add(b, d), u = c_sub(b, d);
    a = c_add(t0, t2);
    c = c_sub(t0, t2);
    // t1 +- u W_4 (W_4 = -i, INV: +i): the swapped halves in scalar operations
    if (INV) {
        b = make_float2(t1.x - u.y, t1.y + u.x);
        d = make_float2(t1.x + u.y, t1.y - u.x);
    } else {
        b = make_float2(t1.x + u.y, t1.y - u.x);
        d = make_float2(t1.x - u.y, t1.y + u.x);
    }
}

// The same with c = d = 0 on entry (forward).
static __device__ __forceinline__ void dft4_half(float2 &a, float2 &b, float2 &c, float2 &d)
{
    const float2 x = a, y = b;
    a = c_add(x, y);
    c = c_sub(x, y);
    b = make_float2(x.x + y.y, x.y - y.x);
    d = make_float2(x.x - y.y, x.y + y.x);
}

// In-register 16-point DFT, natural order in and out: x[k] <- sum_n x[n]
// W_16^(n k) (INV: conjugate exponent, no scaling), as 4 x 4 with n = n1 + 4 n2
// and k = 4 k1 + k2: DFTs over n2, twiddles W_16^(n1 k2), DFTs over n1, and a
// transposed read-out (register renaming only).  HALF: x[8 .. 15] are zero.
template <bool INV, bool HALF = false, bool FINE = false>
static __device__ __forceinline__ void dft16(float2 (&x)[16])
{
    if constexpr (HALF) {
        static_assert(!INV, "only forward transforms start from zero-padded data");
        dft4_half(x[0], x[4], x[8], x[12]);
        dft4_half(x[1], x[5], x[9], x[13]);
        dft4_half(x[2], x[6], x[10], x[14]);
        dft4_half(x[3], x[7], x[11], x[15]);
    } else {
        dft4<INV>(x[0], x[4], x[8], x[12]);  // -> B[n1][k2] at n1 + 4 k2
        dft4<INV>(x[1], x[5], x[9], x[13]);
        dft4<INV>(x[2], x[6], x[10], x[14]);
        dft4<INV>(x[3], x[7], x[11], x[15]);
    }
    x[5] = w32mul<INV, FINE>(x[5], 2);  // W_16^(n1 k2) = W_32^(2 n1 k2)
    x[9] = w32mul<INV, FINE>(x[9], 4);
    x[13] = w32mul<INV, FINE>(x[13], 6);
    x[6] = w32mul<INV, FINE>(x[6], 4);
    x[10] = w32mul<INV, FINE>(x[10], 8);
    x[14] = w32mul<INV, FINE>(x[14], 12);
    x[7] = w32mul<INV, FINE>(x[7], 6);
    x[11] = w32mul<INV, FINE>(x[11], 12);
    x[15] = w32mul<INV, FINE>(x[15], 18);
    dft4<INV>(x[0], x[1], x[2], x[3]);  // -> X[4 k1 + k2] at 4 k2 + k1
    dft4<INV>(x[4], x[5], x[6], x[7]);
    dft4<INV>(x[8], x[9], x[10], x[11]);
    dft4<INV>(x[12], x[13], x[14], x[15]);
    float2 t;
    t = x[1], x[1] = x[4], x[4] = t;
    t = x[2], x[2] = x[8], x[8] = t;
    t = x[3], x[3] = x[12], x[12] = t;
    t = x[6], x[6] = x[9], x[9] = t;
    t = x[7], x[7] = x[13], x[13] = t;
    t = x[11], x[11] = x[14], x[14] = t;
}

// R-point DFTs (R = 2, 4, 8) of consecutive registers, natural order in and out.
template <int R, bool INV, bool FINE>
static __device__ __forceinline__ void dft_runs(float2 (&v)[16])
{
#pragma unroll
    for (int s = 0; s < 16; s += R) {
        if constexpr (R == 2) {
            const float2 a = v[s], b = v[s + 1];
            v[s] = c_add(a, b);
            v[s + 1] = c_sub(a, b);
        } else if constexpr (R == 4) {
            dft4<INV>(v[s], v[s + 1], v[s + 2], v[s + 3]);
        } else {  // even and odd inputs, then W_8 twiddles and one radix-2 step
            dft4<INV>(v[s], v[s + 2], v[s + 4], v[s + 6]);
            dft4<INV>(v[s + 1], v[s + 3], v[s + 5], v[s + 7]);
            float2 e[4], o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                e[k] = v[s + 2 * k];
                o[k] = w32mul<INV, FINE>(v[s + 2 * k + 1], 4 * k);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                v[s + k] = c_add(e[k], o[k]);
                v[s + k + 4] = c_sub(e[k], o[k]);
            }
        }
    }
}

// Shared-memory accesses through 32-bit shared-window addresses: generic
// accesses through pointers the compiler cannot place would keep the
// transforms' register arrays in local memory.
static __device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

static __device__ __forceinline__ float2 lds2(uint32_t a)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}

static __device__ __forceinline__ void sts2(uint32_t a, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

// Two real sequences that share a complex transform leak each other's rounding errors:
// both are scaled to one magnitude first, by powers of two (exact), so that each keeps
// an error relative to its own.  m: the bits of a sequence's largest magnitude (finite);
// a sequence of zeros comes back as zeros.
static __device__ __forceinline__ unsigned pair_exponent(unsigned m)
{
    return min(max(m >> 23, 1u), 253u);
}

static __device__ __forceinline__ float pair_down(unsigned m)  // to [1, 2)
{
    return __uint_as_float((254u - pair_exponent(m)) << 23);
}

static __device__ __forceinline__ float pair_up(unsigned m)  // and back
{
    return m ? __uint_as_float(pair_exponent(m) << 23) : 0.f;
}

// buf: the transform's exchange buffer; tab: the twiddle table (fft16_tw_at's layout; what
// the rounding took from the entries lies kFft16TwLo entries on); bar: a named barrier
// (1 .. 15) of the transform's T threads, used where T > 32.
//
// How a level's fifteen twiddles come about: six entries and nine products of two (the
// envelopes and the demodulation, whose launches wait for these loads: with fifteen
// entries sixteen served frames took 1346 us instead of 1300); an entry each; or an entry
// and what its rounding took (two parts), where the transform's error shows.
enum class Twiddles { kProducts, kEntries, kTwoParts };

template <int LG, Twiddles TW = Twiddles::kProducts>
struct Fft16 {
    static constexpr bool FINE = TW == Twiddles::kTwoParts;
    static constexpr int M = 1 << LG, T = M / 16;
    static constexpr int kLast = (LG - 1) % 4 + 1;  // log2 length of the last level
    uint32_t buf;
    const float2 *__restrict__ tab;
    int u, bar;

    __device__ __forceinline__ void sync() const
    {
        if constexpr (T <= 32)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(T) : "memory");
    }
    // Largest of the T threads' ma and mb (magnitudes, as their bits).  The warps' results
    // go through elements of the buffer that no exchange uses (every seventeenth), so no
    // barrier stands before the transform that follows.  Once per kernel.
    __device__ __forceinline__ uint2 pair_max(unsigned ma, unsigned mb) const
    {
        if constexpr (T < 32) {
#pragma unroll
            for (int off = 1; off < T; off <<= 1) {
                ma = max(ma, __shfl_xor_sync(0xffffffffu, ma, off));
                mb = max(mb, __shfl_xor_sync(0xffffffffu, mb, off));
            }
        } else {
            ma = __reduce_max_sync(0xffffffffu, ma);
            mb = __reduce_max_sync(0xffffffffu, mb);
            if constexpr (T > 32) {
                auto at = [&](int w) { return buf + 8u * (uint32_t)(17 * w + 16); };
                if (u % 32 == 0)
                    sts2(at(u / 32), make_float2(__uint_as_float(ma), __uint_as_float(mb)));
                sync();
#pragma unroll
                for (int w = 0; w < T / 32; ++w) {
                    const float2 m = lds2(at(w));
                    ma = max(ma, __float_as_uint(m.x));
                    mb = max(mb, __float_as_uint(m.y));
                }
            }
        }
        return make_uint2(ma, mb);
    }
    // Address of this thread's element 0 at a level, and element j's offset.
    template <int L>
    __device__ __forceinline__ uint32_t first() const
    {
        if constexpr (L < 4) {
            return buf + 8u * (uint32_t)(17 * u);
        } else {
            constexpr int S = 1 << (L - 4);
            const int p = ((u >> (L - 4)) << L) + (u & (S - 1));
            return buf + 8u * (uint32_t)(p + (p >> 4));
        }
    }
    template <int L>
    __device__ static constexpr uint32_t step(int j)
    {
        return L < 4 ? 8u * (uint32_t)j
                     : 8u * (uint32_t)(j * (1 << (L < 4 ? 0 : L - 4)) +
                                       ((j * (1 << (L < 4 ? 0 : L - 4))) >> 4));
    }
    template <int L>
    __device__ __forceinline__ void put(const float2 (&v)[16]) const
    {
        const uint32_t a = first<L>();
#pragma unroll
        for (int j = 0; j < 16; ++j)
            sts2(a + step<L>(j), v[j]);
    }
    template <int L>
    __device__ __forceinline__ void get(float2 (&v)[16]) const
    {
        const uint32_t a = first<L>();
#pragma unroll
        for (int j = 0; j < 16; ++j)
            v[j] = lds2(a + step<L>(j));
    }
    template <int L, bool INV>
    __device__ __forceinline__ void twiddle(float2 (&v)[16]) const
    {
        constexpr int S = 1 << (L - 4);
        const float2 *__restrict__ t = tab + fft16_tw_at(L) + (u & (S - 1));
        auto entry = [&](int k) {
            const float2 w = __ldg(t + (k - 1) * S);
            return make_float2(w.x, INV ? -w.y : w.y);
        };
        if constexpr (TW == Twiddles::kProducts) {
            float2 w[16];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int e = k < 4 ? k + 1 : 4 * (k - 2);
                w[e] = entry(e);
            }
#pragma unroll
            for (int hi = 0; hi < 16; hi += 4)
#pragma unroll
                for (int lo = 0; lo < 4; ++lo) {
                    if (hi + lo == 0)
                        continue;
                    if (hi && lo)
                        w[hi + lo] = cmul(w[hi], w[lo]);
                    v[hi + lo] = cmul(v[hi + lo], w[hi + lo]);
                }
        } else {
#pragma unroll
            for (int k = 1; k < 16; ++k) {
                if constexpr (FINE) {
                    const float2 l = __ldg(t + kFft16TwLo + (k - 1) * S);
                    v[k] = cmul_fine(v[k], entry(k), make_float2(l.x, INV ? -l.y : l.y));
                } else {
                    v[k] = cmul(v[k], entry(k));
                }
            }
        }
    }
    template <int L, bool HALF>
    __device__ __forceinline__ void down(float2 (&v)[16]) const
    {
        if constexpr (L < 4) {
            dft_runs<(1 << L), false, FINE>(v);
        } else {
            dft16<false, HALF, FINE>(v);
            if constexpr (L > 4) {
                twiddle<L, false>(v);
                put<L>(v);
                sync();
                get<L - 4>(v);
                down<L - 4, false>(v);
            }
        }
    }
    template <int L>
    __device__ __forceinline__ void up(float2 (&v)[16]) const
    {
        if constexpr (L < LG) {
            put<L>(v);
            sync();
            get<L + 4>(v);
            twiddle<L + 4, true>(v);
            dft16<true, false, FINE>(v);
            up<L + 4>(v);
        }
    }
    // v[j] = x[u + j T] -> v[q] = X[fft16_bin(LG, u, q)].  HALF: x[M / 2 ..] = 0.
    template <bool HALF>
    __device__ __forceinline__ void forward(float2 (&v)[16]) const
    {
        down<LG, HALF>(v);
    }
    // The reverse with the conjugate exponent, without scaling.
    __device__ __forceinline__ void inverse(float2 (&v)[16]) const
    {
        if constexpr (kLast < 4)
            dft_runs<(1 << kLast), true, FINE>(v);
        else
            dft16<true, false, FINE>(v);
        up<kLast>(v);
    }
};

}  // namespace bfi
