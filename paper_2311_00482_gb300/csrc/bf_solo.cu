// Solo beamforming: the planner, the launch by precision, and the kernels of FP32
// records (those of FP16 and BF16 records: bf_solo_f16.cu, bf_solo_bf16.cu).
#include "bf_solo.cuh"

namespace bfi {

cudaError_t launch_solo_f16(const BfJob *jobs_dev, const int *tile_prefix_dev, int njobs,
                            int total_tiles, size_t smem_bytes, int variant, int split, int ang,
                            int *err_dev, cudaStream_t stream);
cudaError_t launch_solo_bf16(const BfJob *jobs_dev, const int *tile_prefix_dev, int njobs,
                            int total_tiles, size_t smem_bytes, int variant, int split, int ang,
                            int *err_dev, cudaStream_t stream);
static BF_SOLO_INSTANTIATE(launch_solo_f32, kPrecF32)

namespace {

// Records of a solo plan: one CTA per (tile, angle group, channel group), one thread
// per (angle, channel).  Per step: for every row band the channels that
// all its pixels count for all the group's angles, and those that only some do;
// per (angle, run of channels) the first staged pair of the run's windows.
__global__ void __launch_bounds__(128) solo_plan_kernel(const PlanJob J, int *__restrict__ err)
{
    __shared__ int kmin[kSoloAngles][kMaxGroup], kmax[kSoloAngles][kMaxGroup];
    __shared__ unsigned flags[kSoloAngles][kMaxGroup];
    const int tile = blockIdx.x, ag = blockIdx.y;
    const int tx = tile % J.tiles_x, tz = tile / J.tiles_x, ntiles = J.tiles_x * J.tiles_z;
    const int th = J.bands * J.rows, tz0 = tz * th, tz_last = min(tz0 + th - 1, J.nz - 1);
    const int a0 = ag * J.na / J.ang_groups, an = (ag + 1) * J.na / J.ang_groups - a0;
    const int amax = (J.na + J.ang_groups - 1) / J.ang_groups;
    const int G = J.group, ngroups = (J.ne + G - 1) / G, runs = G / J.run;
    const int words = solo_record_words(amax, runs);
    const int g = blockIdx.z;
    const int k = threadIdx.x / G, c = threadIdx.x - k * G, i = g * G + c;
    if (k < an) {
        int lo = INT_MAX, hi = INT_MIN;
        unsigned any = 0, full = (1u << J.bands) - 1;
        const int a = a0 + k;
        for (int w = 0; w < kTileCols && i < J.ne; ++w) {
            const int ix = tx * kTileCols + w;
            if (ix >= J.nx)
                break;
            const short2 vr = J.valid[((size_t)a * J.ne + i) * J.nxp + ix];
            for (int b = 0; b < J.bands; ++b) {
                const int b0 = tz0 + b * J.rows, b1 = min(b0 + J.rows - 1, J.nz - 1);
                if (b0 > b1)
                    continue;  // band below the grid: nothing to store there
                if (vr.x <= b1 && vr.y >= b0)
                    any |= 1u << b;
                if (!(vr.x <= b0 && vr.y >= b1))
                    full &= ~(1u << b);
            }
            const int r0 = max((int)vr.x, tz0), r1 = min((int)vr.y, tz_last);
            if (r0 > r1)
                continue;
            const float d2 = J.dx2[(size_t)i * J.nxp + ix];
            const int kb = J.colK[a * J.nx + ix];
            const float fb = J.colF[a * J.nx + ix];
            const int k0 = kb + J.rowK[a * J.nz + r0] +
                           __float2int_rd(fb + J.rowF[a * J.nz + r0] + rx_excess(d2, J.rowZ[r0]));
            const int k1 = kb + J.rowK[a * J.nz + r1] +
                           __float2int_rd(fb + J.rowF[a * J.nz + r1] + rx_excess(d2, J.rowZ[r1]));
            lo = min(lo, min(k0, k1));
            hi = max(hi, max(k0, k1));
        }
        kmin[k][c] = lo;
        kmax[k][c] = hi;
        flags[k][c] = lo > hi ? 0u : any | ((full & any) << 8);
    }
    __syncthreads();
    int *rec = J.wtab + ((size_t)(ag * ngroups + g) * ntiles + tile) * words;
    if (threadIdx.x < kWarps) {
        const int b = threadIdx.x;
        unsigned mf = 0, mp = 0;
        for (int ch = 0; ch < G; ++ch) {
            bool all = true, some = false;
            for (int q = 0; q < an; ++q) {
                all = all && ((flags[q][ch] >> (8 + b)) & 1u);
                some = some || ((flags[q][ch] >> b) & 1u);
            }
            if (all)
                mf |= 1u << ch;
            else if (some)
                mp |= 1u << ch;
        }
        rec[b] = (int)mf;
        rec[kWarps + b] = (int)mp;
    } else if (threadIdx.x >= 32 && threadIdx.x < 32 + amax * runs) {
        const int q = (threadIdx.x - 32) / runs, c0 = (threadIdx.x - 32 - q * runs) * J.run;
        int lo = INT_MAX, hi = INT_MIN;
        for (int ch = c0; ch < c0 + J.run && q < an; ++ch) {
            lo = min(lo, kmin[q][ch]);
            hi = max(hi, kmax[q][ch]);
        }
        int w0 = kNoWindow;
        if (lo <= hi) {
            // pairs lo + kPadL .. hi + kPadL, two pairs of margin on either side
            w0 = (lo + kPadL - 2) & ~(J.align - 1);
            if (hi + kPadL + 2 - w0 + 1 > J.wmax)
                atomicOr(err, kErrWindow);
        }
        rec[2 * kWarps + threadIdx.x - 32] = w0;
    }
}

}  // namespace

size_t solo_smem_bytes(int wmax, int group, int prec, int ang, int split, int variant)
{
    return (size_t)kSoloHeaderBytes +
           solo_exchange_bytes(split, ang == 1 ? 1 : kSoloAngles, variant & BF_DMAS, variant & BF_CF,
                               variant & BF_PDAS) +
           (size_t)kSoloStages * group *
               (kTileCols * 4 * (1 + ang) + (size_t)ang * wmax * pair_bytes(prec));
}

cudaError_t launch_solo_plan(const PlanJob &job, int *err_dev, cudaStream_t stream)
{
    const dim3 grid(job.tiles_x * job.tiles_z, job.ang_groups, (job.ne + job.group - 1) / job.group);
    solo_plan_kernel<<<grid, 128, 0, stream>>>(job, err_dev);
    return cudaGetLastError();
}

cudaError_t launch_solo(const BfJob *jobs_dev, const int *tile_prefix_dev, int njobs, int total_tiles,
                        size_t smem_bytes, int prec, int variant, int split, int ang, int *err_dev,
                        cudaStream_t stream)
{
    if (njobs <= 0 || total_tiles <= 0)
        return cudaSuccess;
    auto *f = prec == kPrecF32    ? launch_solo_f32
              : prec == kPrecF16  ? launch_solo_f16
              : prec == kPrecBF16 ? launch_solo_bf16
                                  : nullptr;
    return f ? f(jobs_dev, tile_prefix_dev, njobs, total_tiles, smem_bytes, variant, split, ang, err_dev,
                 stream)
             : cudaErrorInvalidValue;
}

}  // namespace bfi
