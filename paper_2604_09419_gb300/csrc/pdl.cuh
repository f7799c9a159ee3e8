// Programmatic dependent launch: a kernel may start while the one before it on
// its stream is still running, and waits for it where it needs its results.
// A kernel that is launched so waits (pdl_wait) at some point in every block
// that the next kernel relies on, so that each kernel's end comes after the
// end of all before it.
#pragma once

#include <cuda_runtime.h>

namespace line {

// Let the next kernel of the stream start; wait until the previous kernel's
// writes are visible.  (No effect in a kernel that was launched plainly.)
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... Args, typename... Vals>
cudaError_t launch_pdl(void (*kern)(Args...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              bool pdl, Vals... vals) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, vals...);
}

}  // namespace line
