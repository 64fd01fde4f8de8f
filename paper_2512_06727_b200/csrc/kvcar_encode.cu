// Decode-time encoder + append (one new token per sequence).
//
// A batch of B rows meets weights that are far larger than the rows (GPT-2 shape:
// 0.9 MB per K or V encoder), so the cost is streaming the weights once, and that
// needs the whole machine: each of the two fully connected layers is its own launch
// whose grid spreads the layer's output features over all SMs (one warp per feature:
// the lanes stream that feature's weight row in 16-byte loads and hold it against a
// block of up to 16 input rows staged in shared memory).  The hidden activations
// travel between the two launches through a small fp32 scratch in the workspace.
// Both launches use programmatic dependent launch: a kernel starts while its
// predecessor in the stream drains, fetches its first weights, and only then waits
// for the predecessor's results.
#include <algorithm>

#include "kvcar_encode.cuh"

namespace kvcar {

using namespace enc;

namespace {

constexpr int NW = 8;  // warps (= output features) per CTA

// grid = (ceil(features / NW), ceil(rows / RB), 2 [K, V]); block = NW warps.
template <typename T, int STAGE>
__global__ void __launch_bounds__(NW * 32)
    encode_fc_kernel(const __grid_constant__ EncodeArgs a, const __grid_constant__ SeqList seqs, float *hid, int hid_pitch,
                     int max_batch) {
    extern __shared__ __align__(16) float xs[];  // [RB][n_in]
    encode_fc_block<T, STAGE, true, 1>(a, seqs.id, seqs.n, hid, hid_pitch, max_batch, xs, blockIdx.x, blockIdx.y, blockIdx.z, gridDim.x);
}

template <typename T, int STAGE>
cudaError_t launch_stage(const EncodeArgs &a, const SeqList &seqs, float *hid, int hid_pitch, int max_batch, int n_out_max,
                         int n_in_max, cudaStream_t st) {
    const size_t smem = (size_t)RB * n_in_max * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(encode_fc_kernel<T, STAGE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((n_out_max + NW - 1) / NW, (seqs.n + RB - 1) / RB, 2);
    cfg.blockDim = dim3(NW * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, encode_fc_kernel<T, STAGE>, a, seqs, hid, hid_pitch, max_batch);
}

}  // namespace

size_t encode_split_smem(int max_in, int max_m) { return (size_t)RB * std::max(max_in, max_m) * sizeof(float); }

cudaError_t launch_encode_split(const EncodeArgs &a, const SeqList &seqs, int dtype, int max_in, int max_m, int max_d,
                                float *hid, int max_batch, cudaStream_t st) {
    cudaError_t e;
    const int n_hidden = std::max(max_m, NW);  // raw layers still need one block column for the copy
    if (dtype == KVCAR_F32) {
        e = launch_stage<float, 1>(a, seqs, hid, max_m, max_batch, n_hidden, max_in, st);
        if (e == cudaSuccess && max_m > 0) e = launch_stage<float, 2>(a, seqs, hid, max_m, max_batch, max_d, max_m, st);
    } else {
        e = launch_stage<__nv_bfloat16, 1>(a, seqs, hid, max_m, max_batch, n_hidden, max_in, st);
        if (e == cudaSuccess && max_m > 0)
            e = launch_stage<__nv_bfloat16, 2>(a, seqs, hid, max_m, max_batch, max_d, max_m, st);
    }
    return e;
}

}  // namespace kvcar
