// Launches that overlap the previous kernel's end (programmatic dependent launch).
//
// A kernel launched by launch_dependent may be set up, its blocks placed, while the
// kernel before it in the stream still runs; it begins with grid_begin, which lets the
// next such kernel be set up and then waits until every kernel before it has completed
// and its writes are visible.  Nothing of the previous kernels' memory is touched
// before that, so the order is the stream's; what is saved is the launch and the
// prologue between two kernels, about 1.5 us each, which is what short solves are
// made of.  After anything else in the stream (another launch, a copy) it is an
// ordinary launch.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace tma {

__device__ __forceinline__ void grid_begin()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
}

}  // namespace tma
