// Programmatic launches: the blocks of a kernel may start before the preceding
// kernel of the stream has ended.  Every kernel launched by launch_early calls
// grid_wait before it touches anything that an earlier launch writes or reads,
// and loads such data with ordinary loads: a read-only load (__ldg, or what the
// compiler makes of a const __restrict__ argument) may be moved above the wait.
#pragma once

#include <cuda_runtime.h>

namespace sg {

// lets the successor's blocks start; waits for the predecessor (whose writes are
// then seen).  Both do nothing in a plain launch.
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_early(void (*k)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k, args...);
}

}  // namespace sg
