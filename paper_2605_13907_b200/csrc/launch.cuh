// Launching with programmatic dependent launch: every kernel of the library may start while the kernel before it in the
// stream still runs, and waits (pdl_wait) before it touches global memory.  The steps of a small batch are a chain of
// kernels of 2 to 8 us, and an ordinary launch adds 1 to 3 us between two of them.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace ais {

// Blocks until every kernel this launch depends on has completed and its writes are visible.  Every thread of a kernel
// launched with launch_pdl executes it before its first access to global memory (and before it may return), so that a
// kernel's completion implies the completion of everything before it in the stream.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the stream be scheduled once all CTAs of this one have got here (it still waits for our end).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// The usual opening of a kernel.
__device__ __forceinline__ void pdl_enter() {
    pdl_wait();
    pdl_trigger();
}

template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(std::forward<Args>(args))...);
}

}  // namespace ais
