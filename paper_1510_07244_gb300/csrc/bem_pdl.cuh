// Programmatic dependent launch: chains of short kernels in one stream that may
// overlap.
//
// A kernel launched with launch_chain(chained = true) starts as soon as every CTA
// of the kernel before it has called pdl_launch() (or exited), not when that
// kernel has finished.  A kernel of a chain calls pdl_wait() before it touches
// anything that an earlier kernel of the chain writes, and takes it through plain
// pointers: const __restrict__ would promise that nothing changes while the kernel is
// resident, and allow non-coherent loads.  A kernel that depends on none of
// them calls pdl_end() last, so that its own completion implies theirs (one warp
// of the grid: a wait is an acquire, and one at the end of every warp cost the
// touching kernels 7%).  The first kernel of a chain is launched with chained = false and waits
// for all earlier work of the stream.  Both calls do nothing in a plain launch.
#pragma once

#include <cuda_runtime.h>

namespace bem {

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;"); }
// called by warp 0 of CTA 0 at least
__device__ __forceinline__ void pdl_end()
{
    if (blockIdx.x == 0 && threadIdx.x < 32) pdl_wait();
}
#endif

template <class... P, class... A>
cudaError_t launch_chain(bool chained, unsigned grid, unsigned block, cudaStream_t st, void (*k)(P...),
                         A... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&c, k, static_cast<P>(args)...);
}

}  // namespace bem
