// launch_next.cuh -- kernels launched while the one before them in the stream still runs
// (programmatic dependent launch): only the launch and what a kernel does before
// grid_dependency_wait, which must not touch global memory, overlap.
#pragma once

#include <cuda_runtime.h>

namespace rsv {

// Lets the next kernel of the stream be launched, and waits until the one before it has
// finished and its writes are seen (both at once if it was launched as an ordinary kernel).
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_next(void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, const A&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, P(args)...);
}

}  // namespace rsv
