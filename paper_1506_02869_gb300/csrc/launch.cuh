// Launches that overlap the previous kernel's end (programmatic dependent launch).
//
// A kernel launched by launch_dependent may be set up, its blocks placed, while the
// kernel before it in the stream still runs; it begins with grid_begin, which waits
// until every kernel before it has completed and its writes are visible, and then lets
// the next such kernel be set up.  Nothing of the previous kernels' memory is touched
// before that, so the order is the stream's; what is saved is the launch and the
// prologue between two kernels, about 1.5 us each, which is what short solves are
// made of.  After anything else in the stream (another launch, a copy) it is an
// ordinary launch.
//
// The next kernel is let in after the wait and not before it: with a queue of passes,
// kernels let in before it were placed three and four ahead, wherever the running ones
// left room first, and then ran crowded on those SMs.  Calls one after the other, before
// -> after: gradient of 8 aircraft, 60 steps, 1024 particles, one sample 238 -> 216 us,
// of 2 aircraft, 30 steps, 4096 particles, 12 samples 198 -> 182 us; solve of 4 aircraft
// with Langevin moves 560 -> 510 us, of 2 aircraft 459 -> 438 us.
//
// grid_begin_early lets it in before the wait: the short kernels between two rollouts
// (sample means, normalisation, resampling) and the last one of the selection, which
// are set up while a long rollout ends and behind which nothing crowds.  Without it for
// them: solve of 8 aircraft, 60 steps, 4096 particles, 16 samples 2925 -> 3045 us, with
// random-walk moves of 6 aircraft 1387 -> 1432 us, weights of 3 x 100000 particles 26.0
// -> 33.5 us; in the moves and the two rollout kernels too it gained nothing.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace tma {

__device__ __forceinline__ void grid_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void grid_begin_early()
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
