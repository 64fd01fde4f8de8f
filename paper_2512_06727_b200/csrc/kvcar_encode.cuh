// One block of the decode-time encoder (kvcar_encode.cu): a fully connected layer for up to 16 input rows, one warp per output
// feature.  Device code only; shared by the encoder's own launches and by those that carry it beside other work.
#pragma once
#include "kvcar_internal.h"
#include "kvcar_pdl.cuh"

namespace kvcar {
namespace enc {

constexpr int RB = 16;  // input rows per CTA

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ uint4 load(const float *p) { return __ldg(reinterpret_cast<const uint4 *>(p)); }
    static __device__ __forceinline__ void unpack(const uint4 &v, float *w) {
        w[0] = __uint_as_float(v.x); w[1] = __uint_as_float(v.y); w[2] = __uint_as_float(v.z); w[3] = __uint_as_float(v.w);
    }
    static __device__ __forceinline__ float one(const float *p) { return __ldg(p); }
    static __device__ __forceinline__ void store(float *p, float v) { *p = v; }
};
template <>
struct Vec16<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ uint4 load(const __nv_bfloat16 *p) {
        return __ldg(reinterpret_cast<const uint4 *>(p));
    }
    static __device__ __forceinline__ void unpack(const uint4 &v, float *w) {
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[2 * i] = __uint_as_float(u[i] << 16);
            w[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
        }
    }
    static __device__ __forceinline__ float one(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};

// acc[f][r] += sum over this lane's share of w_f[0..n) * x[r][0..n); `pre` holds the lane's first vector of each row already
template <typename T, int NF>
__device__ __forceinline__ void lane_dots(const T *wrow, const uint4 *pre, const float *x, int n, int rows, int lane, float (*acc)[RB]) {
    constexpr int VL = Vec16<T>::N;
    uint4 cur[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) cur[f] = pre[f];
#pragma unroll 1
    for (int k0 = lane * VL; k0 < n; k0 += 32 * VL) {
        const int kn = k0 + 32 * VL;
        uint4 nxt[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) nxt[f] = kn < n ? Vec16<T>::load(wrow + (int64_t)f * n + kn) : cur[f];
        float w[NF][VL];
#pragma unroll
        for (int f = 0; f < NF; ++f) Vec16<T>::unpack(cur[f], w[f]);
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            if (r % 4 == 0 && r >= rows) break;  // rows in fours, as xs is filled
            const float4 *xr = reinterpret_cast<const float4 *>(x + r * n + k0);
#pragma unroll
            for (int i = 0; i < VL / 4; ++i) {
                const float4 xv = xr[i];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    acc[f][r] = fmaf(w[f][4 * i + 0], xv.x, acc[f][r]);
                    acc[f][r] = fmaf(w[f][4 * i + 1], xv.y, acc[f][r]);
                    acc[f][r] = fmaf(w[f][4 * i + 2], xv.z, acc[f][r]);
                    acc[f][r] = fmaf(w[f][4 * i + 3], xv.w, acc[f][r]);
                }
            }
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) cur[f] = nxt[f];
    }
}

// after the call lane r (r < RB) holds the warp-wide sum of acc[r]
__device__ __forceinline__ float reduce_rows(float *acc, int lane) {
    // fold 16 accumulators over 32 lanes: halve the accumulator count while halving the lane distance
#pragma unroll
    for (int r = 0; r < 8; ++r) {  // distance 16: lanes < 16 keep rows 0..7, lanes >= 16 keep rows 8..15
        const float keep = (lane & 16) ? acc[r + 8] : acc[r];
        const float give = (lane & 16) ? acc[r] : acc[r + 8];
        acc[r] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float keep = (lane & 8) ? acc[r + 4] : acc[r];
        const float give = (lane & 8) ? acc[r] : acc[r + 4];
        acc[r] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const float keep = (lane & 4) ? acc[r + 2] : acc[r];
        const float give = (lane & 4) ? acc[r] : acc[r + 2];
        acc[r] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
    }
    {
        const float keep = (lane & 2) ? acc[1] : acc[0];
        const float give = (lane & 2) ? acc[0] : acc[1];
        acc[0] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    // lane l now holds row ((l>>4)&1)*8 + ((l>>3)&1)*4 + ((l>>2)&1)*2 + ((l>>1)&1)
    return acc[0];
}
__device__ __forceinline__ int row_of_lane(int lane) {
    return ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
}

// raw layer: 16 bytes of input row r's stored heads, from stored channel c on, into the row's place in the cache
template <typename T>
__device__ __forceinline__ void copy_raw_vec(const EncodeArgs &a, const EncPlan &pl, const T *src, const int32_t *seq_ids, int r, int c) {
    const int seq = seq_ids[r], t = a.seq_len[seq];
    const int page = a.block_table[(int64_t)seq * a.max_pages_per_seq + t / a.page_tokens];
    const int64_t pr = (int64_t)page * a.page_tokens + t % a.page_tokens;
    *reinterpret_cast<uint4 *>(reinterpret_cast<T *>(pl.pool) + pr * pl.width + c) =
        Vec16<T>::load(src + (int64_t)r * a.kv_width + pl.heads[c / a.hd] * a.hd + c % a.hd);
}

// A raw layer's whole append of one token per sequence, K and V: the exact current rows (all heads) and the cache rows.  Thread
// `tid` of `n_threads` that share the work.
template <typename T>
__device__ __forceinline__ void append_raw_rows(const EncodeArgs &a, const int32_t *seq_ids, int n_rows, int tid, int n_threads) {
    constexpr int VL = Vec16<T>::N;
    const int wv = a.kv_width / VL;
    for (int which = 0; which < 2; ++which) {
        const EncPlan &pl = a.plan[which];
        const T *src = reinterpret_cast<const T *>(which == 0 ? a.k : a.v);
        const int nv = pl.in_dim / VL, per_row = wv + nv;
        for (int idx = tid; idx < n_rows * per_row; idx += n_threads) {
            const int r = idx / per_row, i = idx % per_row;
            if (i < wv)
                reinterpret_cast<uint4 *>(reinterpret_cast<T *>(pl.cur) + (int64_t)seq_ids[r] * a.kv_width)[i] =
                    reinterpret_cast<const uint4 *>(src + (int64_t)r * a.kv_width)[i];
            else
                copy_raw_vec<T>(a, pl, src, seq_ids, r, (i - wv) * VL);
        }
    }
}

// STAGE 1: hidden = LeakyReLU(BN(W1 x + b1)) -> scratch.  STAGE 2: latent = W2 hidden + b2 -> cache rows.
// A warp takes NF features: a row's values are read from shared memory once per NF weights, and those reads bound the block when
// many row blocks share a launch (256 rows of the GPT-2 shape: see latent_front_kernel).
// Block (bx, by, which) of ceil(features / (warps x NF)) x ceil(rows / RB) x 2 [K, V]; xs: [RB][n_in] floats of shared memory, 16-byte
// aligned.  Weights are requested before the wait for the preceding kernels of the stream.  EARLY: dependent launches may start
// before that wait.
template <typename T, int STAGE, bool EARLY, int NF>
__device__ __forceinline__ void encode_fc_block(const EncodeArgs &a, const int32_t *seq_ids, int n_seqs, float *hid, int hid_pitch,
                                                int max_batch, float *xs, int bx, int by, int which, int nbx) {
    const int NW = (blockDim.x >> 5) * NF;  // output features of a block
    const EncPlan &pl = a.plan[which];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_rows = n_seqs, r0 = by * RB;
    const int in_dim = pl.in_dim, m = pl.m, d = pl.d;
    const int n_in = STAGE == 1 ? in_dim : m, n_out = STAGE == 1 ? m : d;
    const int j = bx * NW + warp * NF;  // this warp's first output feature
    const T *src = reinterpret_cast<const T *>(which == 0 ? a.k : a.v);
    const bool compressed = pl.compressed != 0;

    // weights do not depend on anything earlier in the stream: start fetching them right away
    constexpr int VL = Vec16<T>::N;
    const T *wrow = reinterpret_cast<const T *>(STAGE == 1 ? pl.w1r : pl.w2r) + (int64_t)j * n_in;
    uint4 pre[NF];
    float p0[NF], p1[NF];  // stage 1: fused BatchNorm scale, shift; stage 2: bias
    const bool active = compressed && j < n_out;  // n_out is a multiple of NF where NF > 1
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        pre[f] = make_uint4(0, 0, 0, 0);
        p0[f] = p1[f] = 0.f;
        if (active) {
            if (lane * VL < n_in) pre[f] = Vec16<T>::load(wrow + (int64_t)f * n_in + lane * VL);
            p0[f] = STAGE == 1 ? pl.s1[j + f] : pl.b2[j + f];
            if (STAGE == 1) p1[f] = pl.t1[j + f];
        }
    }
    if (EARLY) launch_dependents();
    grid_dependency_wait();  // inputs, page table and (stage 2) the hidden scratch are final from here on

    const int rows_here = min(RB, n_rows - r0), rows4 = (rows_here + 3) & ~3;
    const int my_row = row_of_lane(lane);
    int64_t prow = -1;  // stage 2: cache row of the input row this lane will write
    if (STAGE == 2 && active && !(lane & 1) && my_row < rows_here) {
        const int seq = seq_ids[r0 + my_row], t = a.seq_len[seq];
        const int page = a.block_table[(int64_t)seq * a.max_pages_per_seq + t / a.page_tokens];
        prow = (int64_t)page * a.page_tokens + t % a.page_tokens;
    }
    if (STAGE == 1) {
        const int wv = a.kv_width / VL;  // 16-byte vectors per input row (head_dim is a multiple of the vector)
        if (bx == 0) {  // exact current-token rows (all heads)
#pragma unroll 1
            for (int idx = threadIdx.x; idx < rows_here * wv; idx += blockDim.x) {
                const int rr = idx / wv, cv = idx % wv, r = r0 + rr;
                reinterpret_cast<uint4 *>(reinterpret_cast<T *>(pl.cur) + (int64_t)seq_ids[r] * a.kv_width)[cv] =
                    reinterpret_cast<const uint4 *>(src + (int64_t)r * a.kv_width)[cv];
            }
        }
        if (!compressed) {
            const int nv = in_dim / VL;
#pragma unroll 1
            for (int idx = bx * blockDim.x + threadIdx.x; idx < rows_here * nv; idx += nbx * blockDim.x)
                copy_raw_vec<T>(a, pl, src, seq_ids, r0 + idx / nv, (idx % nv) * VL);
            return;
        }
        if (bx * NW >= n_out) return;
        // stage the stored heads' slices of this block's rows as fp32, 16 bytes per load, four loads in flight
        const int nv = in_dim / VL, total = rows_here * nv;
#pragma unroll 1
        for (int base = threadIdx.x; base < total; base += 4 * blockDim.x) {
            uint4 v[4];
            int dst[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = base + u * blockDim.x;
                dst[u] = -1;
                if (idx < total) {
                    const int rr = idx / nv, c = (idx % nv) * VL;
                    v[u] = Vec16<T>::load(src + (int64_t)(r0 + rr) * a.kv_width + pl.heads[c / a.hd] * a.hd + c % a.hd);
                    dst[u] = rr * in_dim + c;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (dst[u] >= 0) {
                    float w[VL];
                    Vec16<T>::unpack(v[u], w);
#pragma unroll
                    for (int i = 0; i < VL; i += 4)
                        *reinterpret_cast<float4 *>(xs + dst[u] + i) = make_float4(w[i], w[i + 1], w[i + 2], w[i + 3]);
                }
        }
#pragma unroll 1
        for (int idx = rows_here * in_dim + threadIdx.x; idx < rows4 * in_dim; idx += blockDim.x) xs[idx] = 0.f;
    } else {
        if (!compressed || bx * NW >= n_out) return;
        const float *h = hid + ((int64_t)which * max_batch + r0) * hid_pitch;
        const int nv = m / 4, total = rows_here * nv;
#pragma unroll 1
        for (int base = threadIdx.x; base < total; base += 4 * blockDim.x) {
            float4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = base + u * blockDim.x;
                if (idx < total) v[u] = *reinterpret_cast<const float4 *>(h + (int64_t)(idx / nv) * hid_pitch + (idx % nv) * 4);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int idx = base + u * blockDim.x;
                if (idx < total) *reinterpret_cast<float4 *>(xs + (idx / nv) * m + (idx % nv) * 4) = v[u];
            }
        }
#pragma unroll 1
        for (int idx = rows_here * m + threadIdx.x; idx < rows4 * m; idx += blockDim.x) xs[idx] = 0.f;
    }
    __syncthreads();
    if (!active) return;
    float acc[NF][RB];
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int r = 0; r < RB; ++r) acc[f][r] = 0.f;
    lane_dots<T, NF>(wrow, pre, xs, n_in, rows_here, lane, acc);
    float sum[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) sum[f] = reduce_rows(acc[f], lane);
    if ((lane & 1) || my_row >= rows_here) return;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        if (STAGE == 1) {
            float hv = fmaf(sum[f], p0[f], p1[f]);
            hv = hv > 0.f ? hv : hv * pl.slope;
            hid[((int64_t)which * max_batch + r0 + my_row) * hid_pitch + j + f] = hv;
        } else {
            if (pl.qparam)
                a.z[((int64_t)which * max_batch + r0 + my_row) * a.z_pitch + j + f] = sum[f] + p0[f];
            else
                Vec16<T>::store(reinterpret_cast<T *>(pl.pool) + prow * pl.width + j + f, sum[f] + p0[f]);
        }
    }
}

}  // namespace enc
}  // namespace kvcar
