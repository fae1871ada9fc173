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

// Whether chaining a one-gate kernel pays at this size: `ctas` of its CTAs, `resident` of which the GPU
// holds at once.  The next kernel's CTAs take the room that is left, all of it on the SMs with least to
// do; between a seventh and half of a full GPU they then crowd there while other SMs run dry.  Measured
// (us a gate in chains of ten, plain / chained), gates of 4: high targets, 19 qubits (64 of 304) 6.2 / 7.0, 18
// qubits (32) 6.2 / 4.8, 21 qubits (256) 8.7 / 7.7; mixed, 19 qubits (256 of 912) 6.2 / 9.0, 18 qubits
// (128) 6.2 / 5.0, 20 qubits (512) 8.2 / 7.6; gates of 6, mixed: 19 and 20 qubits (64 and 128 of 304) 24.6 / 30.5
// and 24.6 / 30.8, 18 qubits (32) 24.6 / 22.2, 21 qubits (256) 34.8 / 31.1.
inline bool chain_pays(long long ctas, long long resident) { return 7 * ctas <= resident || 2 * ctas >= resident; }

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
