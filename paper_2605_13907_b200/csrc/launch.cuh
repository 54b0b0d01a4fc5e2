// Launching with programmatic dependent launch: every kernel of the library may start while the kernel before it in the
// stream still runs.  The steps of a small batch are a chain of kernels of 2 to 8 us, and an ordinary launch adds 1 to 3 us
// between two of them.  What a kernel may rely on, and what it owes the next one:
//  - Every kernel triggers (pdl_trigger) only after its own wait.  So when a kernel starts, everything older than the kernel
//    before it is complete, and it may read that before its wait (the moments and rectification kernels read row offsets,
//    masks and log-probs so early); it may write nothing to global memory before it.  The one exception is a pass that runs
//    beside the other pass of its call (LmheadArgs::overlap): it triggers at once and waits at its end, and the merge behind
//    it reads nothing early.
//  - What the kernel before it writes it reads after the wait, and not through pointers that promise the data constant for as
//    long as the kernel runs (const together with __restrict__, __ldg): the writer may run beside it.
//  - Every thread waits before it returns, so that a kernel's completion implies the completion of everything before it.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace ais {

// Blocks until every kernel this launch depends on has completed and its writes are visible.
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
