// Launches of gate kernels one behind the other on a stream (programmatic dependent launch).
//
// A circuit is a chain of kernels that each read what the one before wrote.  Launched this way, a
// kernel's CTAs may start while the one before drains: they set up (barriers, tables, matrix images,
// which no kernel writes) and then wait for its end.  From launch to launch of small kernels this
// takes 1.8 us instead of 3.1.
#pragma once

#include "sv_internal.h"

namespace svg {

#ifdef __CUDACC__
// Once every CTA of this grid has called it (or ended), the next kernel's CTAs may start.
__device__ __forceinline__ void next_may_start() { asm volatile("griddepcontrol.launch_dependents;"); }
// Waits until the kernel before has ended and its writes are visible.  Every thread calls it before
// its first access to the state (at once when the launch before was not of this kind or has ended).
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// chained = false: an ordinary launch (the kernel starts when the one before has ended).
template <typename... P, typename... A>
int launch_chained(bool chained, void (*kern)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t stream, A &&...args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    SV_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...));
    return SV_OK;
}
#endif

}  // namespace svg
