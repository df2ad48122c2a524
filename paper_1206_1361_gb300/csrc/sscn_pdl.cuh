// sscn_pdl.cuh -- programmatic dependent launch of the kernels of a step.  A
// kernel launched with launch_after is scheduled as the blocks of the kernel
// before it in the stream end, not after that one's completion has been flushed
// and signalled: its set-up (coefficient tables, the search for a block's
// instance) runs in the other's tail.  pdl_wait() returns when all earlier
// kernels have completed and their writes are visible; every thread calls it
// before it touches psi or anything else that a kernel writes.
//
// No kernel lets its dependents start earlier (griddepcontrol.launch_dependents):
// their resident blocks then take shared memory and issue slots from the last
// wave.  Measured us a step, ordinary launches / this / a trigger at the top:
// 64^3 FP64 36.8 / 36.0 / 33.8, but 2D 500x384 33.3 / 32.5 / 39.2; complex64
// 64^3 15.7 / 14.9 / 14.7; 256^3 FP64 868 / 868 / 862; a lone 128x128x32 of a
// batch 40.3 / 30.4 / 30.3.  The bandwidth-bound sweeps on long lines (TMA,
// float-float) gained nothing and are launched plainly.
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace gp {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// overlap = false: an ordinary launch.
template <typename... P, typename... A>
cudaError_t launch_after(bool overlap, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                         A &&...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(std::forward<A>(args))...);
}

}  // namespace gp
