// Programmatic dependent launch: a kernel launched with launch_pdl may be scheduled
// while the stream's previous kernel still runs (if that kernel lets it, or drains).
// Its blocks call pdl_wait() before they read or write anything another kernel may
// touch: it returns once the previous kernel has completed and its writes are visible.
// (Loads of such data go through L2 or the ordinary path, never the read-only one.)
// Before the wait a block touches only what no kernel writes.  Where a kernel calls
// pdl_launch_dependents() after its own wait instead of first, its successor may also
// rely on everything before it in the stream (the update of the predictor's training).
#pragma once

#include <cuda_runtime.h>

#include <utility>

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// overlap = false: an ordinary launch, which starts when its predecessor is complete (its
// pdl_wait() returns at once).
template <typename... P, typename... A>
inline cudaError_t launch_pdl_if(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
}
template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
    return launch_pdl_if(true, kernel, grid, block, smem, st, std::forward<A>(args)...);
}
