// Programmatic dependent launches: the kernels of a chain on one stream, each of which may start while
// the one before it ends.
#pragma once

#include <cuda_runtime.h>

namespace mk {

// Start of a kernel of the chain: the next kernel's blocks may be scheduled as soon as all of this
// one's run, do their own start (the geometry) and wait in wait_for_last_kernel until this kernel has
// finished and its writes are visible.  Every kernel of a chain waits before it reads or writes what
// another one does, so that each also orders the kernels before its predecessor.
__device__ __forceinline__ void next_kernel_may_start() { cudaTriggerProgrammaticLaunchCompletion(); }
__device__ __forceinline__ void wait_for_last_kernel() { cudaGridDependencySynchronize(); }

// Launch of a kernel of the chain behind its predecessor on st (not the first one).  early: before the
// predecessor has ended, as above; else behind it.
template <class... Args>
void launch_next(void (*kernel)(Args...), int grid, int threads, cudaStream_t st, bool early, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace mk
