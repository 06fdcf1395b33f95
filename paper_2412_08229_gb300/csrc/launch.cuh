// launch.cuh - kernel launches that overlap the end of the launch before them.
//
// A kernel launched with `overlap` on a stream (or captured into a graph) right behind
// another starts as soon as every block of that one has begun, and waits in overlap_wait()
// for its results; nothing that an earlier kernel writes may be read, and nothing that it
// reads may be written, before that. What an earlier kernel writes is read by plain loads:
// the compiler and the caches may take a __ldg as good at any time of the kernel's life. The
// wait covers all launches before, because the launch waited for has itself waited for its own
// predecessor.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

// At the start of a kernel: lets a next launch made with `overlap` begin, however this one was
// made, then waits for the one before (nothing to wait for in a kernel launched plainly).
__device__ __forceinline__ void overlap_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_kernel(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                                 bool overlap, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace lbm
