// Device helpers of the beamforming kernels: mbarriers, tensor copies, the
// split delay, staged sample pairs and paired FP32 arithmetic.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "bf_internal.h"

namespace bfi {
namespace {

constexpr float kRoundMagic = 12582912.0f;  // 1.5 * 2^23: x + magic rounds x to an integer
constexpr int kRoundBits = 0x4B400000;      // bit pattern of kRoundMagic
constexpr unsigned long long kWaitNs = 4000000000ull;  // bounded wait per CTA (4 s)

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for a barrier phase until the CTA's deadline; false (and an error bit)
// if it passed.  Every wait of the CTA shares one deadline, so a stuck copy
// costs at most kWaitNs before the CTA gives up on all remaining steps.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity,
                                          unsigned long long deadline, int *err)
{
    if (mbar_try_wait(bar, parity))
        return true;
    while (global_ns() < deadline)
        if (mbar_try_wait(bar, parity))
            return true;
    atomicOr(err, kErrTimeout);
    return false;
}

// One 2-D tensor-map box into shared memory, completing on `bar`.
__device__ __forceinline__ void tma_2d(void *dst, const CUtensorMap *map, int x, int y,
                                       uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Before a job's first copies: a tensor map in global memory may lie where an earlier
// launch had another one (the job lists are rewritten, and a plan's maps may get the
// address of a destroyed handle's), so its descriptor is read again.
__device__ __forceinline__ void map_acquire(const CUtensorMap *map)
{
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(
                     reinterpret_cast<uint64_t>(map))
                 : "memory");
}

__device__ __forceinline__ void maps_acquire(const BfJob *J)
{
    map_acquire(J->rf_map);
    map_acquire(J->valid_map);
    map_acquire(J->dx2_map);
}

__device__ __forceinline__ float rsqrt_approx(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sqrt_approx(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// x^e for x >= 0, e > 0 as 2^(e log2 x) on the special-function unit
// (x = 0: log2 gives -inf, 2^-inf = 0).
__device__ __forceinline__ float pow_approx(float x, float e)
{
    float l, y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(l * e));
    return y;
}

// sign(v) |v|^(1/p) of one delayed sample; p = 2 takes the square root.
__device__ __forceinline__ float pdas_root(float v, float inv_p, bool square)
{
    const float av = fabsf(v);
    return copysignf(square ? sqrt_approx(av) : pow_approx(av, inv_p), v);
}

// Receive path length beyond the depth term, in samples:
//   q = sqrt(d2 + z^2) - z = d2 / (sqrt(d2 + z^2) + z),
// d2 = (kappa (x_p - x_i))^2, z = kappa z_p.  The large, pixel-only part of
// the delay (transmit leg + depth) comes from the host as an exact integer +
// remainder, so FP32 only has to carry this small term, formed without
// cancellation; its relative error (a few ulp) keeps the delay within ~1e-6
// samples (float32 emulation: 1e-6 rms, 1e-5 max over |x_p - x_i| <= z_p / 3).
// dx2 >= 1e-30 (host floor), so the square root never sees 0; dx2 + z^2 is
// formed with one rounding.
__device__ __forceinline__ float rx_excess(float dx2, float z)
{
    const float s = fmaf(z, z, dx2);
    const float r = s * rsqrt_approx(s);
    return dx2 * rcp_approx(r + z);
}

__device__ __forceinline__ int find_job(const int *__restrict__ prefix, int njobs, int bid)
{
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(prefix + mid) <= bid)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Sample pairs read from shared memory through 32-bit shared-window addresses.
template <int PREC>
struct PairIO;

template <>
struct PairIO<kPrecF32> {
    static constexpr int kBytes = 8;
    __device__ static __forceinline__ float interp(uint32_t addr, float al)
    {
        float mid, diff;
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(mid), "=f"(diff) : "r"(addr));
        return fmaf(al, diff, mid);
    }
};

template <>
struct PairIO<kPrecF16> {
    static constexpr int kBytes = 4;
    __device__ static __forceinline__ float interp(uint32_t addr, float al)
    {
        unsigned w;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w) : "r"(addr));
        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w));
        return fmaf(al + 0.5f, f.y - f.x, f.x);
    }
};

template <>
struct PairIO<kPrecBF16> {
    static constexpr int kBytes = 4;
    __device__ static __forceinline__ float interp(uint32_t addr, float al)
    {
        unsigned w;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w) : "r"(addr));
        const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xffff0000u);
        return fmaf(al + 0.5f, hi - lo, lo);
    }
};

// Loads through 32-bit shared-window addresses (the consumer loop's tables).
__device__ __forceinline__ float4 lds_f32x4(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr));
    return v;
}

__device__ __forceinline__ int2 lds_int2(uint32_t addr)
{
    int2 v;
    asm volatile("ld.shared.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}

// First and last counted row (two 16-bit halves).
__device__ __forceinline__ int2 lds_rows(uint32_t addr)
{
    int w;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w) : "r"(addr));
    return make_int2((int)(short)(w & 0xffff), w >> 16);
}

__device__ __forceinline__ float lds_f32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void sts_f32x2(uint32_t addr, float a, float b)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
}

// This thread's shared-memory writes, visible to the async proxy (bulk copies).
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Bulk copy shared -> global (16-byte aligned addresses, size a multiple of 16),
// tracked in this thread's bulk groups.
__device__ __forceinline__ void bulk_store(void *gdst, uint32_t ssrc, unsigned bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst),
                 "r"(ssrc), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

// Every committed bulk copy of this thread has read its shared-memory source.
__device__ __forceinline__ void bulk_wait_read()
{
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// Every committed bulk copy of this thread is complete.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ---- packed FP32 pairs (Blackwell f32x2 arithmetic): two rows' delays at once
typedef unsigned long long f32x2_t;

__device__ __forceinline__ f32x2_t pk2(float lo, float hi)
{
    f32x2_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void upk2(f32x2_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

__device__ __forceinline__ f32x2_t fma2(f32x2_t a, f32x2_t b, f32x2_t c)
{
    f32x2_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f32x2_t add2(f32x2_t a, f32x2_t b)
{
    f32x2_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f32x2_t sub2(f32x2_t a, f32x2_t b)
{
    f32x2_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f32x2_t mul2(f32x2_t a, f32x2_t b)
{
    f32x2_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Rounded delays of rows j and j + 1 for one channel (d2 packed twice): the
// rx_excess arithmetic of both rows in paired instructions, each half with
// exactly the scalar version's operations and roundings, plus the pixels'
// remainders.  M: the rounding constant plus the integer parts of the pixels'
// terms, so m holds the whole delay in its low bits (one addition rounds and adds
// the integer part; the bits times the pair size plus a channel's entry are a
// sample pair's address), al the offset in [-1/2, 1/2].
__device__ __forceinline__ void delay2(f32x2_t D2, f32x2_t Zp, f32x2_t Fp, f32x2_t M, float &ma,
                                       float &mb, float &ala, float &alb)
{
    const f32x2_t s = fma2(Zp, Zp, D2);
    float sa, sb;
    upk2(s, sa, sb);
    const f32x2_t r = mul2(s, pk2(rsqrt_approx(sa), rsqrt_approx(sb)));
    float da, db;
    upk2(add2(r, Zp), da, db);
    const f32x2_t x = fma2(D2, pk2(rcp_approx(da), rcp_approx(db)), Fp);
    const f32x2_t m = add2(x, M);
    upk2(m, ma, mb);
    upk2(sub2(x, sub2(m, M)), ala, alb);
}

// Address of the sample pair at rounded delay m: `step` bytes per pair, ent the
// channel's entry (the address of index zero).  CHECK: held inside the window
// [win, win + last], for pixels that do not count the channel.
template <uint32_t STEP, bool CHECK>
__device__ __forceinline__ uint32_t pair_at(float m, uint32_t ent, uint32_t win, uint32_t last)
{
    const uint32_t p = (uint32_t)__float_as_int(m) * STEP + ent;
    return CHECK ? win + min(p - win, last) : p;
}

// Entry of a window that starts at address win with staged pair w0 (ref: the tile's
// reference integer part, which the pixels' terms are relative to).
__device__ __forceinline__ uint32_t window_entry(uint32_t win, int w0, int ref, uint32_t step)
{
    return win - (uint32_t)(w0 + kRoundBits - ref - kPadL) * step;
}

}  // namespace
}  // namespace bfi
