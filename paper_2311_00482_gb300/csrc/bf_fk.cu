// Plane-wave f-k migration (Sec. II-B-3) with the register transforms (bf_fft16.cuh):
// records to per-angle spectra, lateral transforms, the wavenumber mapping with the
// inverse lateral transforms, and the inverse depth transforms.  Four launches (and
// the log stage), each a programmatic dependent of the one before.
//
//   fk_time16   two real records per complex transform; the spectra of both from its
//               Hermitian parts, the transmit's lateral delay removed
//   fk_rows16   lateral transforms
//   fk_map16    per migrated Kz bin the gathered, weighted and summed spectrum and its
//               inverse lateral transform, stored by image column
//   fk_depth16  inverse transform along depth, magnitude, image maximum
//
// A mapped point lies between two temporal bins, and its neighbour along Kz between the
// next two: the lateral transforms therefore leave the spectra transposed, [lateral
// bin][temporal bin], lateral bins in the transform's register order, and the gather
// runs along Kz (with temporal bins a row apart every point took two 32-byte sectors
// of its own).  Bound: the launches' latencies (a 64 x 2048 record of three angles has
// 96 to 193 CTAs of work per launch).  Five launches of shared-memory radix-8
// transforms and a synchronous upload took 59 us per call, these 31 us.
#include "bf_fft16.cuh"
#include "bf_internal.h"
#include "bf_launch.cuh"

namespace bfi {
namespace {

// Kz rows of one fk_map16 CTA.
__host__ __device__ constexpr int fk_map_rows(int lgk) { return lgk >= 11 ? 1 : 2048 >> lgk; }

template <int LG>
struct FkShape {
    static constexpr int T = (1 << LG) / 16;
    static constexpr int threads(int least) { return T > least ? T : least; }
};

// exp(i pi b t), t = turns.x + turns.y half turns a bin: the whole turns of b t drop out
// exactly, so the phase's error does not grow with the delay (as one product it is b t
// 2^-24 half turns, with a delay of 15 samples the largest error of the image).
__device__ __forceinline__ float2 delay_phase(int bin, float2 turns)
{
    const float b = (float)bin, p = __fmul_rn(b, turns.x);
    const float rest = fmaf(b, turns.x, -p) + b * turns.y;
    float s, c;
    sincospif((p - 2.f * rintf(0.5f * p)) + rest, &s, &c);
    return make_float2(c, s);
}

template <int LG, int THREADS>
__global__ void __launch_bounds__(THREADS) fk_time16_kernel(const FkJob J)
{
    extern __shared__ __align__(16) float2 fsm[];
    using F = Fft16<LG, Twiddles::kTwoParts>;
    constexpr int T = F::T, M = F::M;
    dependents_may_start();
    if (blockIdx.x == 0 && threadIdx.x == 0 && J.maxbits)
        *J.maxbits = 0u;  // before fk_depth16 takes the maximum
    const int grp = threadIdx.x / T, np = (J.ne + 1) / 2;
    const F f{smem_addr(fsm) + (uint32_t)(grp * fft16_buf_bytes(LG)), J.ptw, (int)threadIdx.x % T,
              1 + grp};
    const int unit = blockIdx.x * (THREADS / T) + grp, a = unit / np, i = 2 * (unit - a * np);
    const bool has_a = a < J.na, has_b = has_a && i + 1 < J.ne;
    const int16_t *__restrict__ ua = J.rf + (size_t)(a * J.ne + i) * J.ns;
    float2 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        v[j] = make_float2(0.f, 0.f);
        const int n = f.u + j * T;
        if (j < 8 && n < J.ns) {  // records fill at most half of the transform
            v[j].x = has_a ? (float)__ldg(ua + n) : 0.f;
            v[j].y = has_b ? (float)__ldg(ua + J.ns + n) : 0.f;
        }
    }
    f.template forward<true>(v);
    // natural order at k + k / 16 (other threads' last reads are done after the barrier)
    auto at = [&](int k) { return f.buf + 8u * (uint32_t)(k + (k >> 4)); };
    f.sync();
#pragma unroll
    for (int q = 0; q < 16; ++q)
        sts2(at(fft16_bin(LG, f.u, q)), v[q]);
    f.sync();
    if (!has_a)
        return;
    const int row = a * J.ne + i;
    const float2 *__restrict__ turns = reinterpret_cast<const float2 *>(J.beta) + row;
    const float2 ba = __ldg(turns), bb = has_b ? __ldg(turns + 1) : make_float2(0.f, 0.f);
    // D[a][b][i]: nk >= 2 ne leaves room for the odd channel's empty partner
    float2 *__restrict__ D = J.D + (size_t)a * (M / 2 + 1) * J.nk + i;
    for (int b = f.u; b <= M / 2; b += T) {
        const float2 z = lds2(at(b)), w = lds2(at((M - b) & (M - 1)));
        const float2 sa = make_float2(0.5f * (z.x + w.x), 0.5f * (z.y - w.y));
        const float2 sb = make_float2(0.5f * (z.y + w.y), 0.5f * (w.x - z.x));
        const float2 da = cmul(sa, delay_phase(b, ba)), db = cmul(sb, delay_phase(b, bb));
        *reinterpret_cast<float4 *>(D + (size_t)b * J.nk) = make_float4(da.x, da.y, db.x, db.y);
    }
}

// Rows of D (temporal bins of one angle): transforms over the elements (zero from ne
// on, at most half of nk), transposed to E[angle][q T + u][temporal bin].
template <int LG, int THREADS>
__global__ void __launch_bounds__(THREADS) fk_rows16_kernel(const FkJob J)
{
    extern __shared__ __align__(16) float2 fsm[];
    using F = Fft16<LG, Twiddles::kEntries>;
    constexpr int T = F::T, M = F::M;
    dependents_may_start();
    const int grp = threadIdx.x / T, nb = J.nt / 2 + 1, a = blockIdx.y;
    const F f{smem_addr(fsm) + (uint32_t)(grp * fft16_buf_bytes(LG)), J.ptw, (int)threadIdx.x % T,
              1 + grp};
    const int b = blockIdx.x * (THREADS / T) + grp;
    const float2 *__restrict__ D = J.D + ((size_t)a * nb + b) * M;
    wait_for_producer();
    float2 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int n = f.u + j * T;
        v[j] = j < 8 && b < nb && n < J.ne ? D[n] : make_float2(0.f, 0.f);
    }
    f.template forward<true>(v);
    const int pitch = fk_pitch(J.nt);
    float2 *__restrict__ E = J.E + ((size_t)a * M + f.u) * pitch + b;
    if (b < nb)
#pragma unroll
        for (int q = 0; q < 16; ++q)
            E[(size_t)(q * T) * pitch] = v[q];
}

// R = 2048 / nk Kz rows (q = r + 1): every angle's spectrum at its mapped position,
// interpolated between temporal bins i0 and i0 + 1 and weighted, summed, by all the
// CTA's threads (lanes along Kz); then the inverse over the elements, T threads a row.
template <int LG>
__global__ void __launch_bounds__(256) fk_map16_kernel(const FkJob J)
{
    extern __shared__ __align__(16) float2 fsm[];
    using F = Fft16<LG, Twiddles::kEntries>;
    constexpr int T = F::T, M = F::M, R = fk_map_rows(LG), STEP = 256 / R, NP = M / STEP;
    // rows' buffers one float2 apart modulo the banks: lanes along rows do not collide
    constexpr int ROW = fft16_buf_bytes(LG) + 8;
    constexpr int B = NP < 8 ? NP : 8;  // points of an angle loaded at a time
    dependents_may_start();
    const int half = J.nt / 2, pitch = fk_pitch(J.nt), r0 = blockIdx.x * R;
    {
        const int rr = threadIdx.x % R, p0 = threadIdx.x / R, r = min(r0 + rr, half - 1);
        const uint32_t o = smem_addr(fsm) + (uint32_t)(rr * ROW);
        wait_for_producer();
#pragma unroll 1
        for (int c = 0; c < NP; c += B) {
            float2 acc[B];
#pragma unroll
            for (int k = 0; k < B; ++k)
                acc[k] = make_float2(0.f, 0.f);
            for (int a = 0; a < J.na; ++a) {
                int i0[B];
                float2 aw[B], v0[B], v1[B];  // (alpha, weight); untaken points have weight 0
#pragma unroll
                for (int k = 0; k < B; ++k) {
                    const size_t t = ((size_t)a * M + p0 + (c + k) * STEP) * half + r;
                    i0[k] = max(__ldg(J.map_i0 + t), 0);
                    aw[k] = __ldg(J.map_aw + t);
                }
#pragma unroll
                for (int k = 0; k < B; ++k) {
                    const float2 *p = J.E + ((size_t)a * M + p0 + (c + k) * STEP) * pitch + i0[k];
                    v0[k] = p[0];
                    v1[k] = p[i0[k] < half ? 1 : 0];
                }
#pragma unroll
                for (int k = 0; k < B; ++k) {
                    acc[k].x = fmaf(aw[k].y, fmaf(aw[k].x, v1[k].x - v0[k].x, v0[k].x), acc[k].x);
                    acc[k].y = fmaf(aw[k].y, fmaf(aw[k].x, v1[k].y - v0[k].y, v0[k].y), acc[k].y);
                }
            }
            // register q of thread u lies at 17 u + q, where the inverse's first level reads
#pragma unroll
            for (int k = 0; k < B; ++k) {
                const int p = p0 + (c + k) * STEP;
                sts2(o + 8u * (uint32_t)(17 * (p % T) + p / T), acc[k]);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x >= R * T)
        return;
    const int grp = threadIdx.x / T, r = r0 + grp;
    const F f{smem_addr(fsm) + (uint32_t)(grp * ROW), J.ptw, (int)threadIdx.x % T, 1 + grp};
    float2 v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q)
        v[q] = lds2(f.buf + 8u * (uint32_t)(17 * f.u + q));
    f.inverse(v);
    if (r >= half)
        return;
#pragma unroll
    for (int j = 0; j < 8; ++j) {  // elements only: the first half at most
        const int n = f.u + j * T;
        if (n < J.ne)
            J.spec[(size_t)n * half + r] = v[j];
    }
}

// Image column n: inverse transform of its Kz bins (0 < bin <= nt / 2) as the conjugate
// of the forward transform of their conjugates (whose input order the bins have, and
// only the magnitude is wanted), then the first ns samples in natural order through
// the exchange buffer (the 1 / (nt nk) of both inverse transforms applied here).
template <int LG, int THREADS>
__global__ void __launch_bounds__(THREADS) fk_depth16_kernel(const FkJob J)
{
    extern __shared__ __align__(16) float2 fsm[];
    using F = Fft16<LG, Twiddles::kEntries>;
    constexpr int T = F::T, M = F::M;
    dependents_may_start();
    const int grp = threadIdx.x / T;
    const F f{smem_addr(fsm) + (uint32_t)(grp * fft16_buf_bytes(LG)), J.ptw, (int)threadIdx.x % T,
              1 + grp};
    const int col = blockIdx.x * (THREADS / T) + grp;
    wait_for_producer();
    const float2 *__restrict__ s = J.spec + (size_t)col * (M / 2) - 1;  // bin k at s[k]
    float2 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int k = f.u + j * T;
        v[j] = make_float2(0.f, 0.f);
        if (j <= 8 && k >= 1 && k <= M / 2 && col < J.ne) {
            v[j] = s[k];
            v[j].y = -v[j].y;
        }
    }
    f.template forward<false>(v);
    auto at = [&](int k) { return f.buf + 8u * (uint32_t)(k + (k >> 4)); };
    f.sync();
#pragma unroll
    for (int q = 0; q < 16; ++q)
        sts2(at(fft16_bin(LG, f.u, q)), v[q]);
    f.sync();
    const float inv = 1.f / ((float)M * (float)J.nk);
    float lmax = 0.f;
    if (col < J.ne) {
        float *__restrict__ out = J.img + (size_t)col * J.ns;
        for (int z = f.u; z < J.ns; z += T) {
            const float2 w = lds2(at(z));
            const float e = hypotf(w.x, w.y) * inv;
            out[z] = e;
            lmax = fmaxf(lmax, e);
        }
    }
    if (J.maxbits) {
        const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(lmax));  // e >= 0
        if ((threadIdx.x & 31) == 0)
            atomicMax(J.maxbits, w);
    }
}

template <class... Params, class... Args>
cudaError_t launch_after(void (*k)(Params...), dim3 blocks, int threads, size_t smem, bool dependent,
                         cudaStream_t st, Args... args)
{
    int sms = 0;
    cudaError_t e = kernel_setup((const void *)k, smem, threads, true, &sms, nullptr);
    if (e != cudaSuccess)
        return e;
    return launch_kernel(k, blocks, threads, smem, dependent, st, args...);
}

template <int LG>
cudaError_t time_t(const FkJob &J, cudaStream_t st)
{
    constexpr int T = FkShape<LG>::T, TH = FkShape<LG>::threads(128), C = TH / T;
    const int units = J.na * ((J.ne + 1) / 2);
    return launch_after(fk_time16_kernel<LG, TH>, dim3((unsigned)((units + C - 1) / C)), TH,
                        (size_t)C * fft16_buf_bytes(LG), false, st, J);
}

template <int LG>
cudaError_t rows_t(const FkJob &J, cudaStream_t st)
{
    constexpr int T = FkShape<LG>::T, TH = FkShape<LG>::threads(256), C = TH / T;
    const dim3 grid((unsigned)((J.nt / 2 + 1 + C - 1) / C), (unsigned)J.na);
    return launch_after(fk_rows16_kernel<LG, TH>, grid, TH, (size_t)C * fft16_buf_bytes(LG), true, st, J);
}

template <int LG>
cudaError_t map_t(const FkJob &J, cudaStream_t st)
{
    constexpr int R = fk_map_rows(LG);
    return launch_after(fk_map16_kernel<LG>, dim3((unsigned)((J.nt / 2 + R - 1) / R)), 256,
                        (size_t)R * (fft16_buf_bytes(LG) + 8), true, st, J);
}

template <int LG>
cudaError_t depth_t(const FkJob &J, cudaStream_t st)
{
    constexpr int T = FkShape<LG>::T, TH = FkShape<LG>::threads(64), C = TH / T;
    return launch_after(fk_depth16_kernel<LG, TH>, dim3((unsigned)((J.ne + C - 1) / C)), TH,
                        (size_t)C * fft16_buf_bytes(LG), true, st, J);
}

using Stage = cudaError_t (*)(const FkJob &, cudaStream_t);

}  // namespace

cudaError_t launch_fkmig16(const FkJob &J, cudaStream_t st)
{
    static const Stage time[] = {time_t<5>, time_t<6>, time_t<7>, time_t<8>, time_t<9>,
                                 time_t<10>, time_t<11>, time_t<12>, time_t<13>};
    static const Stage rows[] = {rows_t<5>, rows_t<6>, rows_t<7>, rows_t<8>,
                                 rows_t<9>, rows_t<10>, rows_t<11>, rows_t<12>};
    static const Stage map[] = {map_t<5>, map_t<6>, map_t<7>, map_t<8>,
                                map_t<9>, map_t<10>, map_t<11>, map_t<12>};
    static const Stage depth[] = {depth_t<5>, depth_t<6>, depth_t<7>, depth_t<8>, depth_t<9>,
                                  depth_t<10>, depth_t<11>, depth_t<12>, depth_t<13>};
    cudaError_t e = cudaSuccess;
    const int held = fk_angles(J.na, J.nt, J.nk);
    for (int a = 0; a < J.na && e == cudaSuccess; a += held) {  // D is written anew for each
        FkJob g = J;
        g.na = J.na - a < held ? J.na - a : held;
        g.rf += (size_t)a * J.ne * J.ns;
        g.beta += (size_t)a * J.ne * 2;
        g.E += (size_t)a * J.nk * fk_pitch(J.nt);
        e = time[J.lgt - 5](g, st);
        if (e == cudaSuccess)
            e = rows[J.lgk - 5](g, st);
    }
    if (e == cudaSuccess)
        e = map[J.lgk - 5](J, st);
    if (e == cudaSuccess)
        e = depth[J.lgt - 5](J, st);
    return e;
}

}  // namespace bfi
