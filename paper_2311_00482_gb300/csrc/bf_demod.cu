// Demodulation of channel records for the IQ combiners (Sec. II-B-1): complex
// interpolation pairs of the analytic signal, two records per transform.
//
// Two real records a, b go through one complex transform of a + i b.  Multiplied by
// -i sgn(k) its inverse is H{a} + i H{b}, and the analytic signals are a + i H{a} and
// b + i H{b}: one forward and one inverse transform serve both, and their real parts
// are the records themselves, exact.  (Splitting the spectrum and transforming each
// one-sided half back took three transforms for two records, or four; sixteen frames
// of 64 x 2048: 43.1 us.)  Sixteen points per thread in registers (bf_fft16.cuh); the
// Hilbert transforms then pass through the exchange buffer in natural order, because
// a pair needs its next sample.
#include <type_traits>

#include "bf_fft16.cuh"
#include "bf_internal.h"

namespace bfi {
namespace {

constexpr int kDemodThreads = 256, kDemodBigThreads = 512;

// Units of one job: the row pairs of a frame, or the rows of a frame pair.
template <int LG, int THREADS>
__device__ __forceinline__ void demod_units(const DemodJob &J, int unit0, uint32_t bufs)
{
    using F = Fft16<LG>;
    constexpr int T = F::T, M = F::M;
    const int grp = threadIdx.x / T;
    const F f{bufs + (uint32_t)(grp * fft16_buf_bytes(LG)), J.ptw, (int)threadIdx.x % T, 1 + grp};
    const int unit = unit0 + grp;
    const int rb = J.nf == 1 ? 2 * unit + 1 : unit;  // the second record's row
    const int ra = J.nf == 1 ? rb - 1 : rb;
    const bool has_a = ra < J.rows, has_b = rb < J.rows;
    const int16_t *__restrict__ ua = J.rf + (size_t)ra * M;
    const int16_t *__restrict__ ub = (J.nf == 1 ? J.rf : J.rf2) + (size_t)rb * M;
    float2 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j)
        v[j] = make_float2(has_a ? (float)__ldg(ua + f.u + j * T) : 0.f,
                           has_b ? (float)__ldg(ub + f.u + j * T) : 0.f);
    // Two rows of one frame each keep their own precision (a dead channel's stays zero);
    // the two frames of a pair share a row as they are.
    float ha = 1.f, hb = 1.f;
    if (J.nf == 1) {
        unsigned ma = 0u, mb = 0u;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            ma = max(ma, __float_as_uint(fabsf(v[j].x)));
            mb = max(mb, __float_as_uint(fabsf(v[j].y)));
        }
        const uint2 m = f.pair_max(ma, mb);
        const float da = pair_down(m.x), db = pair_down(m.y);
        ha = pair_up(m.x);
        hb = pair_up(m.y);
#pragma unroll
        for (int j = 0; j < 16; ++j)
            v[j] = make_float2(v[j].x * da, v[j].y * db);
    }
    f.template forward<false>(v);
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const int k = fft16_bin(LG, f.u, q);
        const float s = k == 0 || 2 * k == M ? 0.f : 2 * k < M ? 1.f / (float)M : -1.f / (float)M;
        v[q] = make_float2(v[q].y * s, -v[q].x * s);  // -i sgn(k) / M
    }
    f.inverse(v);
    // natural order at n + n / 16: the addresses this thread's last exchange read
    auto at = [&](int n) { return f.buf + 8u * (uint32_t)(n + (n >> 4)); };
#pragma unroll
    for (int j = 0; j < 16; ++j)
        sts2(at(f.u + j * T), make_float2(v[j].x * ha, v[j].y * hb));
    f.sync();
    // pair j: samples k = j - kPadL and k + 1, mid = (A + B) / 2 and diff = B - A with
    // A = a[k], B = a[k + 1] rot (zero outside the record)
    const float2 rot = J.rot;
    float4 *__restrict__ oa = J.pairs + (J.nf == 1 ? (size_t)ra * J.nsp
                                                   : (size_t)ra * J.nsp * J.nf + J.fi / 2 * 2);
    for (int j = f.u; j < J.nsp; j += T) {
        float2 h[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        float xa[2] = {0.f, 0.f}, xb[2] = {0.f, 0.f};
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int k = j - kPadL + s;
            if (k >= 0 && k < M) {
                h[s] = lds2(at(k));
                xa[s] = has_a ? (float)__ldg(ua + k) : 0.f;
                xb[s] = has_b ? (float)__ldg(ub + k) : 0.f;
            }
        }
        const float2 ba = cmul(make_float2(xa[1], h[1].x), rot), bb = cmul(make_float2(xb[1], h[1].y), rot);
        const float4 pa = make_float4(0.5f * (xa[0] + ba.x), 0.5f * (h[0].x + ba.y), ba.x - xa[0],
                                      ba.y - h[0].x);
        const float4 pb = make_float4(0.5f * (xb[0] + bb.x), 0.5f * (h[0].y + bb.y), bb.x - xb[0],
                                      bb.y - h[0].y);
        if (J.nf == 1) {
            if (has_a)
                oa[j] = pa;
            if (has_b)
                oa[(size_t)J.nsp + j] = pb;
        } else if (has_a) {
            // per pair index the frame pair's eight floats
            float4 *o = oa + (size_t)j * J.nf;
            o[0] = make_float4(pa.x, pb.x, pa.y, pb.y);
            o[1] = make_float4(pa.z, pb.z, pa.w, pb.w);
        }
    }
}

template <bool BIG>
__global__ void __launch_bounds__(BIG ? kDemodBigThreads : kDemodThreads, BIG ? 1 : 3)
    demod16_kernel(const DemodJob *__restrict__ jobs, const int *__restrict__ blk_prefix, int njobs)
{
    constexpr int THREADS = BIG ? kDemodBigThreads : kDemodThreads;
    extern __shared__ __align__(16) float2 dsm[];
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(blk_prefix + mid) <= (int)blockIdx.x)
            lo = mid;
        else
            hi = mid - 1;
    }
    const DemodJob &J = jobs[lo];
    const int first = blockIdx.x - __ldg(blk_prefix + lo);
    if (first == 0 && threadIdx.x < 4) {  // before any later kernel takes a maximum
        if (J.maxbits)
            J.maxbits[threadIdx.x] = 0u;
        if (J.maxbits2)
            J.maxbits2[threadIdx.x] = 0u;
    }
    const uint32_t bufs = smem_addr(dsm);
    auto run = [&](auto lg) {
        constexpr int LG = decltype(lg)::value;
        demod_units<LG, THREADS>(J, first * demod_units_per_block(LG), bufs);
    };
    if constexpr (BIG) {
        run(std::integral_constant<int, 13>());
    } else {
        switch (J.lgn) {
        case 5: run(std::integral_constant<int, 5>()); break;
        case 6: run(std::integral_constant<int, 6>()); break;
        case 7: run(std::integral_constant<int, 7>()); break;
        case 8: run(std::integral_constant<int, 8>()); break;
        case 9: run(std::integral_constant<int, 9>()); break;
        case 10: run(std::integral_constant<int, 10>()); break;
        case 11: run(std::integral_constant<int, 11>()); break;
        default: run(std::integral_constant<int, 12>()); break;
        }
    }
}

template <bool BIG>
cudaError_t launch_t(const DemodJob *jobs_dev, const int *blk_prefix_dev, int njobs, int total_blocks,
                     cudaStream_t stream)
{
    constexpr int threads = BIG ? kDemodBigThreads : kDemodThreads;
    const size_t smem = (size_t)threads * 17 * sizeof(float2);
    int sms = 0;
    cudaError_t e = kernel_setup((const void *)demod16_kernel<BIG>, smem, threads, true, &sms, nullptr);
    if (e != cudaSuccess)
        return e;
    demod16_kernel<BIG><<<total_blocks, threads, smem, stream>>>(jobs_dev, blk_prefix_dev, njobs);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_demod16(const DemodJob *jobs_dev, const int *blk_prefix_dev, int njobs,
                           int total_blocks, bool big, cudaStream_t stream)
{
    if (njobs <= 0 || total_blocks <= 0)
        return cudaSuccess;
    return big ? launch_t<true>(jobs_dev, blk_prefix_dev, njobs, total_blocks, stream)
               : launch_t<false>(jobs_dev, blk_prefix_dev, njobs, total_blocks, stream);
}

}  // namespace bfi
