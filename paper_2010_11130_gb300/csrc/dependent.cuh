// Launches with programmatic dependence: a grid may start while the one before
// it on the stream still runs, reads what none of them writes (the matrix, row
// lists, 1 / a_ii) and only then waits for it.  Between kernels of a few
// microseconds that hides the launch and the first load latencies.  A kernel
// reads vectors and writes only after dep_wait, which at least one thread of
// every grid reaches, so the end of a grid also is the end of all before it.
#pragma once

#include "air_internal.cuh"

__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
void launch_dependent(void (*kernel)(P...), unsigned grid, unsigned threads, cudaStream_t s, const A &...args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = air_counted(grid);
    cfg.blockDim = dim3(threads);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
