// Programmatic dependent launches: a kernel starts while its predecessor in the stream ends, and waits for it where it needs what
// came before.  Every kernel launched this way waits in each of its blocks, so that a kernel's end implies the end of all before it.
//
// What a kernel may read before its own wait.  The wait is what makes its predecessor's writes visible; launch_dependents is no
// release.  decode_latent_kernel and fma_hidden_kernel start on page table, cached rows and (int8) widened rows before they wait.
// Their predecessors in the stream (latent_front_kernel, fma_query_kernel) let them start only after a wait of their own, so whatever
// was enqueued before those is complete and written back to L2 by then.  What is left is an older line in an SM's first-level cache.
//   - Page table and cached rows below the sequences' lengths are written, or counted in (kvcar_advance), by the table update, an
//     ordinary launch: behind everything before it and in front of everything after it, so no kernel after it meets older lines.
//   - The widened int8 rows and their parameters are written again by every layer of a step with dependent launches all the way, so
//     they are read where no first-level cache stands between: tensor loads, and __ldcg for the parameters.
// (The table past that cache as well: 12-layer step of GPT-2's shape, 1 x 200 tokens, 337 -> 341 us, TinyLLaMA 4 x 32768 1653 -> 1669.)
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
