// npp_launch.cuh -- programmatic dependent launch: a kernel queued with
// launch_dependent may start while the kernel before it in the stream drains
// (its launch and its set-up overlap that kernel's tail); it calls
// wait_for_previous before it touches anything that kernel reads or writes.
// An event wait queued in between makes it an ordinary launch.
// GB300: a plan step of 512 samples, T = 20, 37 -> 34 us, a sampling time of
// a road mission 135 -> 133 (with its two advance launches in one).
#pragma once

#include <cuda_runtime.h>

namespace npp {

// returns once the grids this one depends on have completed and their writes
// are visible (at once in an ordinary launch)
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// lets the next launch_dependent kernel of the stream start once every block of
// this grid has called it (or ended)
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*fn)(P...), int grid, int block, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, fn, P(args)...);
}

}  // namespace npp
