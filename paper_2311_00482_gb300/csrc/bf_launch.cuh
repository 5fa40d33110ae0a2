// Kernel launches, plain or as a programmatic dependent of the launch before.
#pragma once

#include <cuda_runtime.h>

namespace bfi {

// Lets the next launch's blocks be scheduled (a dependent one's; they wait for this
// grid's completion before they read its results).
static __device__ __forceinline__ void dependents_may_start()
{
    asm volatile("griddepcontrol.launch_dependents;");
}

// Waits until the launch before has completed and its results are visible (returns at
// once in a plain launch).
static __device__ __forceinline__ void wait_for_producer()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Dynamic shared memory that keeps a grid of `blocks` spread over `sms` SMs: as much as
// ceil(blocks / sms) CTAs per SM leave each.  A dependent launch's blocks are placed
// while the kernel before still holds most SMs, and without this pile up on the few
// that are free first (a 300 x 384 pDAS frame: 45.6 us plain, 54.6 us piled up).
static inline size_t spread_smem(size_t smem, int blocks, int sms)
{
    const size_t per = (size_t)((blocks + sms - 1) / sms);
    const size_t most = ((size_t)228 << 10) / (per > 0 ? per : 1) - 2048;  // 1 KB reserved per CTA, static arrays
    return smem > most ? smem : most;
}

template <class... Params, class... Args>
static cudaError_t launch_kernel(void (*k)(Params...), dim3 blocks, int threads, size_t smem,
                                 bool dependent, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = blocks;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace bfi
