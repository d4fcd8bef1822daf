// launch.cuh -- grid sizing of the grid-stride kernels, and launches that may
// start before the kernel ahead of them on the stream has ended.
#pragma once

#include <utility>

#include "common.cuh"

namespace qed {

int sm_count();

// CTAs of `threads` for a grid-stride kernel over `items` work items: at most
// as many as stay resident on the GPU at once (computed once per kernel), since
// a CTA left for a second wave only lengthens the launch
template <auto Kernel>
int resident_grid(int threads, size_t dyn, int64_t items)
{
    static int per_sm = 0;
    if (per_sm == 0) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, Kernel, threads, dyn);
        if (per_sm <= 0) per_sm = 1;
    }
    const int64_t want = (items + threads - 1) / threads;
    const int64_t cap = (int64_t)sm_count() * per_sm;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

// A launch, with `early` a programmatic dependent one: the kernel may be scheduled
// once every CTA of the kernel ahead of it on the stream has called allow_next()
// (or exited), so that its launch and whatever it does before wait_previous()
// overlap that kernel's tail.  wait_previous() returns when the kernel ahead has
// ended and its writes are visible; a kernel launched this way calls it, in every
// thread, before it touches anything that an earlier launch writes (one that is never
// launched early -- the bulk copies, the fused push -- starts after it and has none).  Used where
// the launches are most of a step (kSmallPerSm): the substep of 1e4 electrons
// takes 13.6 us instead of 18.5; at 2e6 particles it changes nothing, and the bulk
// pipeline loses 2 % to the waiting CTAs.
template <typename... P, typename... A>
cudaError_t launch_next(bool early, void (*kernel)(P...), int grid, int threads, size_t dyn, cudaStream_t st,
                        A &&...args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = dyn;
    c.stream = st;
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}

__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace qed
