// launch.cuh -- dependent launches: a kernel of a chain of short steps may start while the one
// before it drains (programmatic dependent launch), and waits for it itself.  Empty kernels of 152
// CTAs follow one another every 1.35 us so, 2.06 us launched the plain way, and what does not depend
// on the step before (barriers, the copies of W) runs ahead: 48^3, one slice, 3 vectors 12.3 -> 9.3
// us per step, 14^3 x 24, 5 FP16 vectors 14.4 -> 12.5, 16^3 x 32, one vector 7.5 -> 6.5; nothing from
// about 30 us up.
#pragma once

#include <cuda_runtime.h>

namespace tls {

// Waits until the grids this one depends on have finished and their writes are visible.  Every
// thread that reads what they wrote, or writes what they read, comes after it; a CTA does not
// return without it (the grid's own completion is what the next grid waits for).  Returns at once
// in a kernel launched the plain way.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next grid of the chain start as soon as every CTA of this one has come here.
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;"); }

// dep: the kernel starts with grid_dep_wait() and may overlap the end of its predecessor.
template <typename... P, typename... A>
inline cudaError_t launch_dep(bool dep, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = dep ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace tls
