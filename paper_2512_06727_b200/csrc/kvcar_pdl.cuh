// Programmatic dependent launches: a kernel starts while its predecessor in the stream ends, and waits for it where it needs what
// came before.  Every kernel launched this way waits in each of its blocks, so that a kernel's end implies the end of all before it.
#pragma once
#include <cuda_runtime.h>

namespace kvcar {

__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Formal, typename... Args>
cudaError_t launch_pdl(void (*k)(Formal...), dim3 grid, int threads, size_t smem, cudaStream_t st, const Args &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace kvcar
