// Programmatic dependent launches: a kernel starts while its predecessor in the stream ends, and waits for it where it needs what
// came before.  Every kernel launched this way waits in each of its blocks, so that a kernel's end implies the end of all before it.
//
// What a kernel may read before its own wait.  The wait is what makes its predecessor's writes visible; launch_dependents is no
// release.  decode_latent_kernel and fma_hidden_kernel start on page table, cached rows and (int8) widened rows before they wait.
// Their predecessors in the stream (latent_front_kernel, fma_query_kernel) let them start only after a wait of their own, so whatever
// was enqueued before those is complete and written back to L2 by then, and that is where these reads go: tensor loads (which know no
// other cache) and __ldcg for the table and the row parameters, whose addresses are written again from call to call.  Cached rows
// that fma_hidden_kernel reads through the first-level cache lie below the sequences' lengths: a row gets there by kvcar_advance,
// whose table update is an ordinary launch, behind everything before it and in front of everything after it.
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
