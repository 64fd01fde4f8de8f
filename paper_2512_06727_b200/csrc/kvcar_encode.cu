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
    return launch_pdl(encode_fc_kernel<T, STAGE>, dim3((n_out_max + NW - 1) / NW, (seqs.n + RB - 1) / RB, 2), NW * 32, smem, st, a, seqs, hid,
                      hid_pitch, max_batch);
}

// Eq. 4 per cached row, as the tail of encode_generic_kernel: scale = 255/(max-min), zero-point = -round(scale*min) - 128,
// code = round(scale*x + zero-point) kept inside int8.  grid = ceil(2 * rows / 8), one warp per (K or V, row).
__global__ void __launch_bounds__(256) encode_quant_kernel(const __grid_constant__ EncodeArgs a, const __grid_constant__ SeqList seqs,
                                                           int max_batch) {
    grid_dependency_wait();
    launch_dependents();
    const int item = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int which = item / seqs.n, r = item % seqs.n;
    if (which > 1) return;
    const EncPlan &pl = a.plan[which];
    if (!pl.qparam) return;
    const float *z = a.z + ((int64_t)which * max_batch + r) * a.z_pitch;
    const int seq = seqs.id[r], t = a.seq_len[seq], d = pl.d;
    const int page = a.block_table[(int64_t)seq * a.max_pages_per_seq + t / a.page_tokens];
    const int64_t row = (int64_t)page * a.page_tokens + t % a.page_tokens;
    float lo = INFINITY, hi = -INFINITY;
    for (int j = lane; j < d; j += 32) {
        lo = fminf(lo, z[j]);
        hi = fmaxf(hi, z[j]);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    float scale = 1.f, zp = -lo;  // a row of equal values has no range: code 0 with zero-point -x restores it exactly
    if (hi > lo) {
        scale = 255.f / (hi - lo);
        zp = -rintf(scale * lo) - 128.f;
    }
    int8_t *codes = reinterpret_cast<int8_t *>(pl.pool) + row * pl.width;
    for (int j = lane; j < d; j += 32)
        codes[j] = (int8_t)(int)(hi > lo ? fminf(fmaxf(rintf(fmaf(scale, z[j], zp)), -128.f), 127.f) : 0.f);
    if (lane == 0) {
        pl.qparam[row * 2] = scale;
        pl.qparam[row * 2 + 1] = zp;
    }
}

}  // namespace

cudaError_t launch_encode_quant(const EncodeArgs &a, const SeqList &seqs, int max_batch, cudaStream_t st) {
    return launch_pdl(encode_quant_kernel, dim3((2 * seqs.n + 7) / 8), 256, 0, st, a, seqs, max_batch);
}

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
        if (e == cudaSuccess && a.z) e = launch_encode_quant(a, seqs, max_batch, st);
    }
    return e;
}

}  // namespace kvcar
