// Decode attention over latent rows in fp32 arithmetic: fp32 storage, head widths other than 64, pages that are no multiple of 64 tokens,
// and bf16 or int8 layers beyond the limits of kvcar_latent.cu (more than 32 query heads, hidden layers above 1024 or 384 with more than
// 16 heads, more than six source layers, wide latents, widths that are no multiples of 16).
//
// The algebra of kvcar_latent.cu (the last decoder layer is linear, so it is applied to the query before and to the weighted
// sum after the cached tokens) with everything in fp32 on the CUDA cores.  decode_generic_kernel, which restores every head of
// 128 tokens in one block, left 147 of 148 SMs idle at one sequence of 128 tokens (11.6 ms for a GPT-2-shaped fp32 layer) and
// did three times the operations.  Here a block is a tile of tokens x a chunk of hidden columns x one source:
//   fma_query_kernel   W4_h^T q per (K source, listed sequence, query head)
//   fma_hidden_kernel  K: its chunk's part of the scores of every head of the source
//   fma_hidden_kernel  V: sums the parts, softmax over the tile, its chunk of U = sum p a
//   fma_merge_kernel   tiles of a sequence -> W4_h U + b4_h sum, the exact current token, the output row
// Bound: FMA.  Tiles of 64 x 64 (8 x 4 per thread: three 16-byte shared loads per 32 FMA) where they fill the machine, else of
// 32 x 32 (a sequence of 128 tokens is 72 blocks per side instead of 18).
// The first three are programmatic dependent launches, and both hidden kernels work out their activations before they wait for what the
// launch before left.  One GPT-2-shaped fp32 layer, us, with plain launches and 256-thread merges -> now: 1 x 128 tokens 95 -> 88,
// 1 x 17 86 -> 60, 8 x 500 246 -> 211, 32 x 900 890 -> 865.
#include <algorithm>
#include <cmath>

#include "kvcar_fma.h"
#include "kvcar_pdl.cuh"

namespace kvcar {

namespace {

constexpr int KC = 32;  // latent columns staged at a time
constexpr float LOG2E = 1.4426950408889634f;

__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ld1(const float *p) { return __ldg(p); }
__device__ __forceinline__ float ld1(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
__device__ __forceinline__ float4 ld4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16 *p) {
    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p));
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                       __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ void st1(float *p, float v) { *p = v; }
__device__ __forceinline__ void st1(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

// the listed sequences of a launch: those of one group
struct FmaSeqs {
    int32_t n, first_listed;               // group's sequences are listed sequences first_listed ..
    int32_t id[KVCAR_MAX_BATCH];
    int32_t len[KVCAR_MAX_BATCH];
    int32_t tile0[KVCAR_MAX_BATCH];        // first FM_TOK-token tile of the sequence inside the group
};

struct HiddenArgs {
    const int32_t *block_table;
    const float *wq;
    float *score, *upart, *ml;
    int32_t max_pages_per_seq, page_tokens;
    int32_t hq, group, batch, max_m, n_tiles, unit_cols;  // n_tiles: of the group (score pitch)
};

// grid = (tokens of the longest sequence / TT, chunks of all sources of the side, sequences); T: weights; Q8: int8 rows.
// SIDE 0: parts of the scores.  SIDE 1: probabilities of the tile from the parts, U.  Thread = TT / 8 tokens x 4 columns.
template <typename T, bool Q8, int TT, int HC, int SIDE>
__global__ void __launch_bounds__(HC * 2) fma_hidden_kernel(const __grid_constant__ FmaLayer L, const __grid_constant__ FmaSeqs sq,
                                                           const __grid_constant__ HiddenArgs a) {
    constexpr int NT = HC * 2, RT = TT / 8;  // threads, tokens per thread
    constexpr int ZP = TT + 4;               // pitch of the staged latents [k][token]
    constexpr int PARTS = FM_TOK / TT;       // launches' tiles per partial result
    extern __shared__ __align__(16) float sm[];
    float *zs = sm;                     // [2][KC][ZP]
    float *ws = zs + 2 * KC * ZP;       // [2][KC][HC]
    float *act = ws + 2 * KC * HC;      // [TT][HC + 1]
    float *aux = act + TT * (HC + 1) + 3;
    aux -= (aux - sm) & 3;              // SIDE 0: [hq][HC] W4^T q; SIDE 1: [hq][TT] probabilities
    __shared__ int64_t rows[TT];
    __shared__ float scl[TT], zp[TT];   // int8 rows: scale and zero-point
    const int tid = threadIdx.x, si = blockIdx.z, t0 = blockIdx.x * TT;
    const int len = sq.len[si], hq = a.hq, group = a.group;
    if (t0 >= len) {
        grid_dependency_wait();
        return;
    }
    const int valid = min(TT, len - t0), seq = sq.id[si];
    // which source and chunk
    int s = 0, ch = blockIdx.y;
    while (ch >= (L.src[SIDE][s].m + HC - 1) / HC) ch -= (L.src[SIDE][s++].m + HC - 1) / HC;
    const FmaSrc &sp = L.src[SIDE][s];
    const int d = sp.d, m = sp.m, c0 = ch * HC;
    if (tid < TT) {
        const int t = t0 + (tid < valid ? tid : 0);  // rows past the end repeat a valid one; they have no probability
        const int page = a.block_table[(int64_t)seq * a.max_pages_per_seq + t / a.page_tokens];
        const int64_t r = (int64_t)page * a.page_tokens + t % a.page_tokens;
        rows[tid] = r;
        if (Q8) {
            scl[tid] = sp.qparam[2 * r];
            zp[tid] = sp.qparam[2 * r + 1];
        }
    }
    const int tile = sq.tile0[si] + t0 / FM_TOK, sub = (t0 % FM_TOK) / TT;  // partial result and place inside it
    __syncthreads();
    const T *w1 = reinterpret_cast<const T *>(sp.w1t);
    constexpr int NZ = TT * KC / 4 / NT, NW = KC * HC / 4 / NT;  // 16-byte pieces per thread
    float4 zr[NZ], wr[NW];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int i = 0; i < NZ; ++i) {
            const int x = tid + i * NT, t = x / (KC / 4), k = k0 + 4 * (x % (KC / 4));
            zr[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < d) {
                if (Q8) {  // Eq. 4: x = (code - zero-point) / scale
                    const char4 c = *reinterpret_cast<const char4 *>(reinterpret_cast<const int8_t *>(sp.pool) + rows[t] * d + k);
                    zr[i] = make_float4(((float)c.x - zp[t]) / scl[t], ((float)c.y - zp[t]) / scl[t], ((float)c.z - zp[t]) / scl[t],
                                        ((float)c.w - zp[t]) / scl[t]);
                } else {
                    zr[i] = ld4(reinterpret_cast<const T *>(sp.pool) + rows[t] * d + k);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            const int x = tid + i * NT, k = k0 + x / (HC / 4), j = c0 + 4 * (x % (HC / 4));
            wr[i] = k < d && j < m ? ld4(w1 + (int64_t)k * m + j) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    auto stage = [&](int buf) {
#pragma unroll
        for (int i = 0; i < NZ; ++i) {
            const int x = tid + i * NT, t = x / (KC / 4), k = 4 * (x % (KC / 4));
            float *z = zs + buf * KC * ZP + k * ZP + t;
            z[0] = zr[i].x;
            z[ZP] = zr[i].y;
            z[2 * ZP] = zr[i].z;
            z[3 * ZP] = zr[i].w;
        }
#pragma unroll
        for (int i = 0; i < NW; ++i) {
            const int x = tid + i * NT;
            *reinterpret_cast<float4 *>(ws + buf * KC * HC + (x / (HC / 4)) * HC + 4 * (x % (HC / 4))) = wr[i];
        }
    };
    const int tx = tid % (HC / 4), ty = tid / (HC / 4);
    float acc[RT][4];
#pragma unroll
    for (int r = 0; r < RT; ++r) acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0.f;
    fetch(0);
    stage(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < d; k0 += KC, buf ^= 1) {
        if (k0 + KC < d) fetch(k0 + KC);
        const float *z = zs + buf * KC * ZP + ty * RT, *w = ws + buf * KC * HC + tx * 4;
#pragma unroll 8
        for (int k = 0; k < KC; ++k) {
            const float4 wv = *reinterpret_cast<const float4 *>(w + k * HC);
            float zv[RT];
#pragma unroll
            for (int r = 0; r < RT; r += 4) *reinterpret_cast<float4 *>(zv + r) = *reinterpret_cast<const float4 *>(z + k * ZP + r);
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                acc[r][0] = fmaf(zv[r], wv.x, acc[r][0]);
                acc[r][1] = fmaf(zv[r], wv.y, acc[r][1]);
                acc[r][2] = fmaf(zv[r], wv.z, acc[r][2]);
                acc[r][3] = fmaf(zv[r], wv.w, acc[r][3]);
            }
        }
        if (k0 + KC < d) stage(buf ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int j = c0 + tx * 4 + e;
        const float s1 = j < m ? sp.s1[j] : 0.f, t1 = j < m ? sp.t1[j] : 0.f;
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const float x = fmaf(acc[r][e], s1, t1);
            act[(ty * RT + r) * (HC + 1) + tx * 4 + e] = x > 0.f ? x : x * sp.slope;
        }
    }
    const int nc = min(HC, m - c0);
    // The launch before left what is read from here on (W4^T q, scores); it waited itself before it let this one start, so all that
    // is older - rows, tables - was there from the beginning, and the hidden layer ran beside it.
    grid_dependency_wait();
    launch_dependents();
    if (SIDE == 0) {
        const float *wq = a.wq + ((int64_t)s * a.batch + sq.first_listed + si) * hq * a.max_m + c0;
        for (int i = tid; i < hq * HC; i += NT) aux[i] = i % HC < nc ? wq[(int64_t)(i / HC) * a.max_m + i % HC] : 0.f;
        __syncthreads();
        for (int i = tid; i < hq * TT; i += NT) {
            const int h = i / TT, t = i % TT;
            if (!((sp.kv_mask >> (h / group)) & 1u)) continue;
            const float *x = act + t * (HC + 1), *y = aux + h * HC;
            float p0 = 0.f, p1 = 0.f;
#pragma unroll 8
            for (int j = 0; j < HC; j += 2) {
                p0 = fmaf(x[j], y[j], p0);
                p1 = fmaf(x[j + 1], y[j + 1], p1);
            }
            a.score[(((int64_t)ch * a.n_tiles + tile) * hq + h) * FM_TOK + sub * TT + t] = p0 + p1;
        }
    } else {
        // the partial result's tokens: this launch's tile is one of PARTS pieces of it, but maximum and sum are of all
        const int whole = min(FM_TOK, len - (t0 - sub * TT));
        const int warp = tid >> 5, lane = tid & 31;
        for (int h = warp; h < hq; h += NT / 32) {
            if (!((sp.kv_mask >> (h / group)) & 1u)) continue;
            const int n_part = (L.src[0][L.idx[0][h / group]].m + a.unit_cols - 1) / a.unit_cols;
            float v[2] = {-INFINITY, -INFINITY};
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int t = lane + 32 * u;
                if (t < whole) {
                    float x = 0.f;
#pragma unroll 9
                    for (int c = 0; c < n_part; ++c) x += a.score[(((int64_t)c * a.n_tiles + tile) * hq + h) * FM_TOK + t];
                    v[u] = x;
                }
            }
            float M = fmaxf(v[0], v[1]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
            const float e0 = ex2(v[0] - M), e1 = ex2(v[1] - M);
            float S = e0 + e1;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
            if (lane == 0 && ch == 0 && sub == 0) {
                a.ml[((int64_t)tile * hq + h) * 2] = M;
                a.ml[((int64_t)tile * hq + h) * 2 + 1] = S;
            }
            const int b = sub * TT;
            if (lane >= b && lane < b + TT) aux[h * TT + lane - b] = e0;
            if (lane + 32 >= b && lane + 32 < b + TT) aux[h * TT + lane + 32 - b] = e1;
        }
        __syncthreads();
        for (int i = tid; i < hq * HC; i += NT) {
            const int h = i / HC, j = i % HC;
            if (!((sp.kv_mask >> (h / group)) & 1u) || j >= nc) continue;
            const float *p = aux + h * TT, *x = act + j;
            float u0 = 0.f, u1 = 0.f;
#pragma unroll 8
            for (int t = 0; t < TT; t += 2) {
                u0 = fmaf(p[t], x[t * (HC + 1)], u0);
                u1 = fmaf(p[t + 1], x[(t + 1) * (HC + 1)], u1);
            }
            a.upart[(((int64_t)tile * PARTS + sub) * hq + h) * a.max_m + c0 + j] = u0 + u1;
        }
    }
}

// W4_h^T q: grid = (query heads, blocks of 64 hidden columns, blocks of 8 sequences), 8 warps; lanes over the head's channels
template <typename T>
__global__ void __launch_bounds__(256) fma_query_kernel(const __grid_constant__ FmaLayer L, const T *q, float *wq, int n_seqs, int hq,
                                                        int group, int hd, float scale, int batch, int max_m) {
    constexpr int SB = 8;
    __shared__ float qs[SB][KVCAR_MAX_HEAD_DIM];
    const int qh = blockIdx.x, si0 = blockIdx.z * SB, n_here = min(SB, n_seqs - si0), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kvh = qh / group, s = L.idx[0][kvh], slot = L.slot[0][kvh];
    const FmaSrc &sp = L.src[0][s];
    grid_dependency_wait();
    launch_dependents();
    for (int i = tid; i < SB * hd; i += 256) {
        const int k = i / hd, c = i % hd;
        qs[k][c] = k < n_here ? ld1(q + ((int64_t)(si0 + k) * hq + qh) * hd + c) * scale : 0.f;
    }
    __syncthreads();
    for (int j = blockIdx.y * 64 + warp; j < min(sp.m, (int)blockIdx.y * 64 + 64); j += 8) {
        const T *w = reinterpret_cast<const T *>(sp.w2t) + (int64_t)j * sp.in_dim + slot * hd;
        float x[SB];
#pragma unroll
        for (int k = 0; k < SB; ++k) x[k] = 0.f;
        for (int c = lane; c < hd; c += 32) {
            const float wv = ld1(w + c);
#pragma unroll
            for (int k = 0; k < SB; ++k) x[k] = fmaf(wv, qs[k][c], x[k]);
        }
        float mine = 0.f;
#pragma unroll
        for (int k = 0; k < SB; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x[k] += __shfl_xor_sync(0xffffffffu, x[k], o);
            if (lane == k) mine = x[k];
        }
        if (lane < n_here) wq[(((int64_t)s * batch + si0 + lane) * hq + qh) * max_m + j] = mine;
    }
}

// Merge of the tiles of one (query head, sequence).  A block's time is that of its chain of loads of W4 (576 rows of 64 channels at the
// GPT-2 shape), so few blocks get 1024 threads, many 256.  FINAL: apply the last decoder layer and write the output row;
// else leave one partial result for the sequence.  `parts`: pieces of U per partial result.
struct MergeArgs {
    const float *upart, *ml;
    float *useq, *mlseq;
    const void *q;
    void *out;
    int32_t hq, group, hd, kv_width, max_m, parts, with_current, tok;  // tok: tokens of a partial result
    float scale;
};
template <typename T, bool FINAL, int THREADS>
__global__ void __launch_bounds__(THREADS) fma_merge_kernel(const __grid_constant__ FmaLayer L, const __grid_constant__ FmaSeqs sq,
                                                        const __grid_constant__ MergeArgs a) {
    extern __shared__ float u[];  // [max_m], then [THREADS] partial sums
    constexpr int WARPS = THREADS / 32;
    __shared__ float red[WARPS], bred[WARPS];
    grid_dependency_wait();
    launch_dependents();
    const int qh = blockIdx.x, si = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, hd = a.hd;
    const int listed = sq.first_listed + si;
    const int kvh = qh / a.group, slot = L.slot[1][kvh];
    const FmaSrc &sp = L.src[1][L.idx[1][kvh]];
    const int n = (sq.len[si] + a.tok - 1) / a.tok;
    const int64_t t0 = sq.tile0[si];
    auto block_max = [&](float v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0) red[warp] = v;
        __syncthreads();
        v = red[0];
        for (int i = 1; i < WARPS; ++i) v = fmaxf(v, red[i]);
        return v;
    };
    auto block_sum = [&](float v, float *buf) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) buf[warp] = v;
        __syncthreads();
        v = buf[0];
        for (int i = 1; i < WARPS; ++i) v += buf[i];
        return v;
    };
    float M = -INFINITY, S = 0.f;
    for (int t = tid; t < n; t += THREADS) M = fmaxf(M, a.ml[((t0 + t) * a.hq + qh) * 2]);
    M = block_max(M);
    for (int t = tid; t < n; t += THREADS) S += ex2(a.ml[((t0 + t) * a.hq + qh) * 2] - M) * a.ml[((t0 + t) * a.hq + qh) * 2 + 1];
    __syncthreads();
    S = block_sum(S, bred);
    const int tpp = FM_TOK / a.parts;  // tokens of a piece
    for (int j = tid; j < sp.m; j += THREADS) {
        float acc = 0.f;
        for (int t = 0; t < n; ++t) {
            const float w = ex2(a.ml[((t0 + t) * a.hq + qh) * 2] - M);
            const int pieces = a.parts == 1 ? 1 : min(a.parts, (sq.len[si] - t * FM_TOK + tpp - 1) / tpp);
            for (int p = 0; p < pieces; ++p) acc = fmaf(w, a.upart[(((t0 + t) * a.parts + p) * a.hq + qh) * a.max_m + j], acc);
        }
        if (FINAL)
            u[j] = acc;
        else
            a.useq[((int64_t)listed * a.hq + qh) * a.max_m + j] = acc;
    }
    if (!FINAL) {
        if (tid == 0) {
            a.mlseq[((int64_t)listed * a.hq + qh) * 2] = M;
            a.mlseq[((int64_t)listed * a.hq + qh) * 2 + 1] = S;
        }
        return;
    }
    __syncthreads();
    // thread = (channel, share of the hidden range)
    float *sums = u + a.max_m;
    const int np = THREADS / hd, c = tid % hd, part = tid / hd;
    float o = 0.f;
    if (part < np) {
        const T *w = reinterpret_cast<const T *>(sp.w2t) + slot * hd + c;
#pragma unroll 12
        for (int j = part; j < sp.m; j += np) o = fmaf(ld1(w + (int64_t)j * sp.in_dim), u[j], o);
    }
    sums[tid] = o;
    // scores were taken without q . b4_h, the same for every token: it only matters against the current token
    float sc = 0.f, bias = 0.f;
    if (tid < hd) {
        const int kslot = L.slot[0][kvh];
        const float qv = ld1(reinterpret_cast<const T *>(a.q) + ((int64_t)listed * a.hq + qh) * hd + tid) * a.scale;
        bias = qv * L.src[0][L.idx[0][kvh]].b2[kslot * hd + tid];
        if (a.with_current) sc = qv * ld1(reinterpret_cast<const T *>(L.cur[0][kvh]) + (int64_t)sq.id[si] * a.kv_width + tid);
    }
    __syncthreads();
    bias = block_sum(bias, red);
    __syncthreads();
    sc = block_sum(sc, bred);
    if (tid >= hd) return;
    for (int p = 1; p < np; ++p) o += sums[tid + p * hd];
    o += sp.b2[slot * hd + tid] * S;
    if (a.with_current) {
        const float Mb = M == -INFINITY ? M : M + bias, Mn = fmaxf(Mb, sc);
        const float w0 = Mb == -INFINITY ? 0.f : ex2(Mb - Mn), w1 = ex2(sc - Mn);
        const float vc = ld1(reinterpret_cast<const T *>(L.cur[1][kvh]) + (int64_t)sq.id[si] * a.kv_width + tid);
        S = S * w0 + w1;
        o = o * w0 + vc * w1;
    }
    st1(reinterpret_cast<T *>(a.out) + ((int64_t)listed * a.hq + qh) * hd + tid, S > 0.f ? o / S : 0.f);
}

int padded(int m) { return (m + 63) / 64 * 64; }
int group_tiles(int max_len) { return std::max(FM_GROUP_TILES, (max_len + FM_TOK - 1) / FM_TOK); }

template <typename T, bool Q8, int TT, int HC>
cudaError_t launch_hidden(const FmaLayer &L, const FmaSeqs &sq, const HiddenArgs &h, int max_len, cudaStream_t st) {
    const size_t smem = (size_t)(2 * KC * (TT + 4) + 2 * KC * HC + TT * (HC + 1) + 4 + h.hq * std::max(TT, HC)) * sizeof(float);
    auto k = fma_hidden_kernel<T, Q8, TT, HC, 0>;
    auto v = fma_hidden_kernel<T, Q8, TT, HC, 1>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(v, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int units[2] = {0, 0};
    for (int w = 0; w < 2; ++w)
        for (int s = 0; s < L.n_src[w]; ++s) units[w] += (L.src[w][s].m + HC - 1) / HC;
    const int tiles = (max_len + TT - 1) / TT;
    cudaError_t e = launch_pdl(k, dim3(tiles, units[0], sq.n), HC * 2, smem, st, L, sq, h);
    if (e != cudaSuccess) return e;
    return launch_pdl(v, dim3(tiles, units[1], sq.n), HC * 2, smem, st, L, sq, h);
}

template <typename T, bool Q8>
cudaError_t launch_tiles(FmaState &st, const kvcar_config &cfg, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens,
                         const FmaLayer &L, cudaStream_t stream, int *n_launches) {
    int max_mk = 0;
    for (int s = 0; s < L.n_src[0]; ++s) max_mk = std::max(max_mk, L.src[0][s].m);
    cudaError_t e = launch_pdl(fma_query_kernel<T>, dim3(a.hq, (max_mk + 63) / 64, (seqs.n + 7) / 8), 256, 0, stream, L,
                               reinterpret_cast<const T *>(a.q), st.wq, seqs.n, a.hq, a.hq / a.hkv, a.hd, a.scale * LOG2E, st.batch,
                               (int)st.max_m);
    if (e != cudaSuccess) return e;
    *n_launches = 1;
    int n_all = 0;
    for (int i = 0; i < seqs.n; ++i) n_all += (lens[i] + FM_TOK - 1) / FM_TOK;
    st.per_seq = n_all > st.group_tiles;
    // tiles of 64 x 64 where they make at least two waves of blocks, else of 32 x 32 (whose parts of the scores are 32 wide)
    int cols = 0;
    for (int s = 0; s < L.n_src[0]; ++s) cols += L.src[0][s].m;
    const bool small = (int64_t)n_all * ((cols + 63) / 64) < 4 * st.n_sms;
    HiddenArgs h;
    h.block_table = a.block_table;
    h.wq = st.wq;
    h.score = st.score;
    h.upart = st.upart;
    h.ml = st.ml;
    h.max_pages_per_seq = a.max_pages_per_seq;
    h.page_tokens = a.page_tokens;
    h.hq = a.hq;
    h.group = a.hq / a.hkv;
    h.batch = st.batch;
    h.max_m = st.max_m;
    h.unit_cols = small ? 32 : 64;
    for (int i0 = 0; i0 < seqs.n;) {
        FmaSeqs g;
        g.n = 0;
        g.first_listed = i0;
        int t = 0, longest = 0;
        while (i0 < seqs.n) {
            const int n = (lens[i0] + FM_TOK - 1) / FM_TOK;
            if (g.n > 0 && t + n > st.group_tiles) break;
            g.id[g.n] = seqs.id[i0];
            g.len[g.n] = lens[i0];
            g.tile0[g.n] = t;
            t += n;
            longest = std::max(longest, lens[i0]);
            ++g.n;
            ++i0;
        }
        if (longest == 0) {
            if (!st.per_seq) continue;
        } else {
            h.n_tiles = t;
            e = small ? launch_hidden<T, Q8, 32, 32>(L, g, h, longest, stream) : launch_hidden<T, Q8, 64, 64>(L, g, h, longest, stream);
            if (e != cudaSuccess) return e;
            *n_launches += 2;
        }
        if (st.per_seq) {
            MergeArgs m{};
            m.upart = st.upart;
            m.ml = st.ml;
            m.useq = st.useq;
            m.mlseq = st.mlseq;
            m.hq = a.hq;
            m.group = a.hq / a.hkv;
            m.hd = a.hd;
            m.max_m = st.max_m;
            m.parts = small ? 2 : 1;
            m.tok = FM_TOK;
            e = launch_pdl(fma_merge_kernel<T, false, 256>, dim3(a.hq, g.n), 256, 0, stream, L, g, m);
            if (e != cudaSuccess) return e;
            ++*n_launches;
        }
    }
    st.last_parts = small ? 2 : 1;
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_merge(FmaState &st, const kvcar_config &cfg, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens,
                         const FmaLayer &L, cudaStream_t stream) {
    FmaSeqs g;
    g.n = seqs.n;
    g.first_listed = 0;
    int t = 0;
    for (int i = 0; i < seqs.n; ++i) {
        g.id[i] = seqs.id[i];
        g.len[i] = st.per_seq ? (lens[i] > 0 ? 1 : 0) : lens[i];
        g.tile0[i] = st.per_seq ? i : t;
        t += (lens[i] + FM_TOK - 1) / FM_TOK;
    }
    MergeArgs m{};
    m.upart = st.per_seq ? st.useq : st.upart;
    m.ml = st.per_seq ? st.mlseq : st.ml;
    m.q = a.q;
    m.out = a.out;
    m.hq = a.hq;
    m.group = a.hq / a.hkv;
    m.hd = a.hd;
    m.kv_width = a.hkv * a.hd;
    m.max_m = st.max_m;
    m.parts = st.per_seq ? 1 : st.last_parts;
    m.tok = FM_TOK;
    m.with_current = (a.flags & KVCAR_INCLUDE_CURRENT_EXACT) != 0;
    m.scale = a.scale * LOG2E;
    const bool few = a.hq * seqs.n <= 2 * st.n_sms && (st.max_m + 1024) * sizeof(float) <= 48 * 1024;
    const int threads = few ? 1024 : 256;
    return launch_pdl(few ? fma_merge_kernel<T, true, 1024> : fma_merge_kernel<T, true, 256>, dim3(a.hq, seqs.n), threads,
                      (size_t)(st.max_m + threads) * sizeof(float), stream, L, g, m);
}

}  // namespace

size_t fma_ws_bytes(const kvcar_config &cfg, int max_k_sources, int max_m, int batch, int max_len) {
    if (max_m <= 0) return 0;
    const size_t m = padded(max_m), hq = cfg.n_q_heads, gt = group_tiles(max_len);
    return ((size_t)std::min(max_k_sources, FM_MAX_SRC) * batch * hq * m + (m / 32) * gt * hq * FM_TOK + gt * hq * (2 * m + 2) +
            (size_t)batch * hq * (m + 2)) * sizeof(float);
}

void fma_setup(FmaState &st, const kvcar_config &cfg, const std::vector<LayerPlan> &plans, int max_k_sources, int max_m, int batch,
               int max_len, char *ws_area) {
    st.layer.clear();
    if (max_m <= 0) return;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&st.n_sms, cudaDevAttrMultiProcessorCount, dev);
    st.layer.assign(cfg.n_layers, FmaLayer{});
    st.max_m = padded(max_m);
    st.batch = batch;
    st.group_tiles = group_tiles(max_len);
    const size_t m = st.max_m, hq = cfg.n_q_heads, gt = st.group_tiles;
    float *p = reinterpret_cast<float *>(ws_area);
    st.wq = p;
    p += (size_t)std::min(max_k_sources, FM_MAX_SRC) * batch * hq * m;
    st.score = p;
    p += (m / 32) * gt * hq * FM_TOK;
    st.upart = p;
    p += gt * hq * 2 * m;  // two pieces per partial result with the small tiles
    st.ml = p;
    p += gt * hq * 2;
    st.useq = p;
    p += (size_t)batch * hq * m;
    st.mlseq = p;
    const size_t elem = cfg.storage == KVCAR_F32 ? 4 : 2;
    for (int l = 0; l < cfg.n_layers; ++l) {
        FmaLayer &L = st.layer[l];
        bool ok = true;
        int quant = 0, plain = 0;
        for (int w = 0; w < 2 && ok; ++w) {
            const WhichPlan &wp = plans[l].w[w];
            ok = wp.n_src > 0 && wp.n_src <= FM_MAX_SRC;
            L.n_src[w] = wp.n_src;
            for (int s = 0; s < wp.n_src && ok; ++s) {
                const SourcePlan &sp = wp.src[s];
                ok = sp.compressed && sp.d % 4 == 0 && sp.m % 4 == 0 && sp.width == sp.d;
                if (!ok) break;
                (sp.qparam ? quant : plain)++;
                FmaSrc &f = L.src[w][s];
                f = {sp.pool, sp.w1t, sp.w2t, sp.s1, sp.t1, sp.b2, sp.qparam, sp.d, sp.m, sp.in_dim, sp.slope, 0u};
                // matrices are read in pieces of four elements
                ok = ((uintptr_t)sp.w1t % (4 * elem)) == 0;
                for (int i = 0; i < sp.n_need; ++i) {
                    const int h = sp.kv_head[i];
                    f.kv_mask |= 1u << h;
                    L.idx[w][h] = (uint8_t)s;
                    L.slot[w][h] = (uint8_t)sp.slot[i];
                    L.cur[w][h] = reinterpret_cast<const char *>(plans[l].cur[w][h]) + (size_t)plans[l].cur_head[w][h] * cfg.head_dim * elem;
                }
            }
        }
        L.quant = quant > 0;
        L.ok = ok && !(quant && plain) && cfg.head_dim <= KVCAR_MAX_HEAD_DIM;
    }
}

cudaError_t fma_launch_tiles(FmaState &st, const kvcar_config &cfg, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens,
                             int layer, cudaStream_t stream, int *n_launches) {
    const FmaLayer &L = st.layer[layer];
    if (cfg.storage == KVCAR_F32) return launch_tiles<float, false>(st, cfg, a, seqs, lens, L, stream, n_launches);
    return L.quant ? launch_tiles<__nv_bfloat16, true>(st, cfg, a, seqs, lens, L, stream, n_launches)
                   : launch_tiles<__nv_bfloat16, false>(st, cfg, a, seqs, lens, L, stream, n_launches);
}

cudaError_t fma_launch_merge(FmaState &st, const kvcar_config &cfg, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens,
                             int layer, cudaStream_t stream) {
    return cfg.storage == KVCAR_F32 ? launch_merge<float>(st, cfg, a, seqs, lens, st.layer[layer], stream)
                                    : launch_merge<__nv_bfloat16>(st, cfg, a, seqs, lens, st.layer[layer], stream);
}

}  // namespace kvcar
