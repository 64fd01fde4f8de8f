// Decode attention over latent rows without restored K and V rows (bf16 storage, sm_100a).
//
// The decoder of a (layer, K/V) is FC -> BatchNorm -> LeakyReLU -> FC with nothing after the last FC (Sec. "Network
// Architecture").  With a the activated hidden vector of a cached token,
//     q . k'   = q . (W4_h a + b4_h)     = a . (W4_h^T q) + q . b4_h
//     sum p v' = sum p (W4_h a + b4_h)   = W4_h (sum p a) + b4_h sum p
// so the last layer is applied once per sequence and head (to the query before the tiles, to the weighted sum after
// them) instead of once per token: at the GPT-2 shape 0.91 instead of 2.66 MFLOP per cached token and layer, and the
// epilogues that consumed restored rows go away.  W4_h^T q and the probabilities enter their products as two bf16
// terms (value = high + low, 16 bits and the sign; what is left out is 2^-18 of the value, against the 2^-9 that the
// bf16 hidden vector itself carries), so nothing is rounded more coarsely than in the form that restores the rows;
// with KVCAR_ABSORBED (| KVCAR_ABSORBED_V) the caller takes one bf16 term, as that flag says.
//
// Three launches per call, four on small grids, one behind the other in the caller's stream as programmatic dependent launches
// (each starts while its predecessor ends and waits for it only where it needs its results):
//   latent_front_kernel   W4_h^T q per (K source, listed sequence, query head) -> bf16 rows, high and low part; in a step also
//                         the first layer of the new rows' encoder
//   decode_latent_kernel  tiles of 128 cached tokens -> per run of tiles: reference maximum, sum, U = sum p a.  Small grids: one
//                         launch for the scores and one for U, their clusters side by side (see lat_launch)
//   latent_back_kernel    runs of a sequence -> W4_h U + b4_h sum, the exact current token, the output row; in a step also the
//                         second layer of the encoder
//
// decode_latent_kernel.  A cluster of two CTAs walks two runs of consecutive tiles in step, one run per CTA; every
// product is one tcgen05.mma.cta_group::2 of M = 256 (both tiles), so a weight slab crosses L2 -> shared memory once
// per 256 tokens, half into each CTA.  Per step the K side of a tile, then the V side of the tile before (so that the way from S to
// the probabilities is behind the next scores' products), per source layer, per chunk of 192 hidden columns (128: below):
//   hidden   H[256 tok x 192] = Z[256 tok x d] . W1[192 x d]^T into one of two accumulators in tensor memory; the hidden
//            warps add the shift, apply LeakyReLU, round to bf16 and write 64-column slabs into a ring.  The BatchNorm
//            scale is not theirs: its sign is in W1, its size in W4^T q and in the merge (LeakyReLU is positively
//            homogeneous; a slope above 1 is turned round on the host).  The accumulator is read in matrix-fragment layout: a lane needs eight shifts instead of 32
//            (scale and shift fetched per column took 750-900 of a slab's 1 300 cycles) and stores with stmatrix.
//   K side   S[256 tok x 2R] += slab . (W4^T q rows)^T, over the columns of a source; the output warps take of it the heads that the
//            source serves (a stray NaN in one source's rows stays with its heads).  Columns R r .. belong to CTA r (its own
//            sequence's queries)
//   V side   per two slabs: U[256 x 2R] = (slab pair)^T [128 features] . P^T over the tile's 128 tokens.  Each CTA supplies
//            its own hidden slabs and its own probabilities, so in its accumulator its own R columns are its tile's
// S and the U blocks share two 64-column accumulators in turn; the output warps turn S into probabilities and keep the
// running sums of U in registers over a run, rescaled when the reference maximum moves (online softmax), so only one
// partial result per (CTA, sequence) leaves the SM.
//
// What bounds it at the GPT-2 shape (d 384, m 576, 12 heads): the tensor pipe.  A product of M 256 x N x K 16 takes
// max(53, N / 2) cycles (measured alone, whatever the operands' layout), so a pair of tiles needs 2 x 72 x 96 for the hidden
// layers, 36 x 53 for S and 40 x 53 for U: 17 900 cycles.  The latents stay in shared memory for all chunks of a side (96 KB),
// which leaves 64 KB for hidden slabs and 48 KB for weight slabs; 192 columns per chunk because 2 x 192 + 2 x 64 fill
// tensor memory.
//
// Instruction fetch is the other bound: 24 warps run five programs, and with every wait's time limit inlined, U's blocks unrolled and
// two forms of the epilogue the kernel was 88 KB of code, of whose instruction-cache requests 18 % missed (trivial stretches took 300
// cycles).  Waiting is a function now, loops are kept as loops, the epilogue has one form: 61 KB.  With the accumulator given back
// before the ring is waited for, one wait for all of a job's places, and four to twelve query slabs in flight instead of two or three
// (the shifts come through L1), 12-layer steps: GPT-2 8 x 1024 tokens 649 -> 609 us, TinyLLaMA (22 layers) 4 x 32768 1800 -> 1711,
// 32 x 2048 1264 -> 1215.
//
// Two warps issue products, one the hidden jobs, one S and U: with a single issuing thread the two took turns (6 800
// cycles per chunk, 2 700 of them pipe time), and each waited for what only the other needed.  A warp of the hidden
// epilogue takes one slab of a job (three slabs, four lane quarters: twelve warps).
//
// int8 latent rows (Eq. 4: x = (code - zero-point) / scale).  latent_widen_kernel, ahead of the front, writes code - z0 as bf16 rows
// into the workspace, z0 the zero-point kept to [-128, 128]: whole numbers of at most 256, exact in bf16 (a row whose range holds
// zero, as latents have it, has z0 = zero-point).  The hidden warps of the Q8 builds then apply 1 / scale per token, and where a row
// has some of its zero-point left over, that times the weights' row sum.  The fp32 kernels that these builds stand in for keep hidden
// vectors and probabilities in fp32, so here both are two bf16 terms (2^-17 of the value is left out; one term of the hidden vectors
// made the outputs' error 1.8 times that of fp32 at queries of 8 times the usual size, two terms leave it where it was).  A job is 128
// columns then: a pair of slabs of high terms, a pair of low ones, which S and U take into the same accumulators one after the other.
// 12-layer step of the GPT-2 shape, 8 x 1024 tokens: 1024 us (763 with one term), 6404 us in fp32 on the CUDA cores.
//
// Warp roles: 0 loads of latents and query rows, 1 hidden products (leader CTA) and tensor memory, 2 weight loads,
// 3 S and U products (leader CTA), then the hidden warps (twelve; eight where a job is 128 columns) and eight output warps.  All waits are bounded and record a code in the
// status word.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "kvcar_encode.cuh"
#include "kvcar_latent.h"
#include "kvcar_ptx.cuh"

namespace kvcar {

using namespace ptx;

namespace {

constexpr int TILE = 128;                 // tokens per CTA tile
constexpr int SLAB = 16384;               // 128 rows x 64 bf16, 128-byte swizzle
constexpr int HID_WARP = 4, N_OUT = 8;    // first hidden warp, output warps
constexpr int READY_BARS = 8;             // jobs' terms between their epilogue and their product: at most as many as slabs

// What follows from the hidden columns of a job: 192 where the hidden vector is one bf16 term, 128 where it is two (two slabs
// of each term: U's products take their 128 features from a pair of slabs, so a job is one such pair per term), and where latents of
// more than seven slabs leave no room for more (two or four hidden slabs and two weight slabs of 8 KB: latents up to 640 wide).
__host__ __device__ constexpr int wstage(int cn) { return cn / 2 * 128; }  // this CTA's half of a weight slab
__host__ __device__ constexpr int n_threads(int cn) { return 32 * (HID_WARP + 4 * (cn / 64) + N_OUT); }

// Query heads padded to NQ.  Up to 16: high and low terms of an operand are rows of one operand.  32: the terms of W4^T q
// are two operands, and so are those of the probabilities in the P2 builds.  The others take one term of the probabilities: bf16 rows
// of groups of more than two heads, whose restoring form rounds restored K, restored V and the probabilities to bf16, the same class
// (of groups of up to two it keeps the probabilities in fp32).
__host__ __device__ constexpr int op_rows(int nq) { return nq <= 16 ? 2 * nq : nq; }  // operand rows of a CTA in S and U
__host__ __device__ constexpr int wq_rows(int nq) { return 2 * nq; }                  // rows of W4^T q per sequence and source
__host__ __device__ constexpr int wq_slab(int nq) { return wq_rows(nq) * 128; }       // one 64-column slab of them

struct Params {
    CUtensorMap pool[2][LT_MAX_SRC], w1[2][LT_MAX_SRC], tm_wq;
    // MODE_BOTH: list[0] = K, list[1] = V.  MODE_K / MODE_V: list[p] = part p of that side's columns, one cluster per part
    LatList list[LT_MAX_PARTS];
    int32_t mode, n_parts, k_parts;  // k_parts: parts of the scores (MODE_V sums them)
    float *score;
    LatSeqs sq;
    const int32_t *block_table;
    int32_t *status;
    float *upart, *ml;
    int32_t max_pages_per_seq, page_tokens;
    int32_t hq, m_pad, wq_batch;
    int32_t nz, nh, nw, nqs;           // places for latent, hidden, weight and query slabs
    int32_t wide;                      // latents come from the widened rows of the launch's tiles
    int32_t two_terms_k, two_terms_v;  // low parts of the query rows / of the probabilities are used
};

constexpr int MODE_BOTH = 0, MODE_K = 1, MODE_V = 2;

// The waiting itself, out of line: some twenty waits with the time limit inlined made the tile kernel 80 KB of code, far more than
// the instruction cache holds (see decode_latent_kernel).
__device__ __noinline__ void mbar_wait_long(uint32_t bar, uint32_t parity, int32_t *status, volatile int *abort_flag, int code) {
    uint32_t n = 0;
    uint64_t t0 = 0;
    while (!mbar_try(bar, parity)) {
        if ((++n & 255u) == 0) {
            const uint64_t now = global_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > (*abort_flag ? 2000000ull : 2000000000ull)) {  // 2 ms after a failure, else 2 s
                *abort_flag = 1;
                atomicCAS(status, 0, code);
                return;
            }
        }
    }
}
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, int32_t *status, volatile int *abort_flag, int code) {
    if (!mbar_try(bar, parity)) mbar_wait_long(bar, parity, status, abort_flag, code);
}

// the tiles of one CTA, in order
struct TileWalk {
    int si, chunk, n, left;  // listed sequence, tile inside it, its tiles, tiles left of the run (this one included)
    __device__ __forceinline__ int first(const LatSeqs &sq, int i) const { return (int)(sq.first[i] & 0xffffffu); }
    __device__ __forceinline__ void idle() { si = chunk = left = 0; n = 1; }
    __device__ __forceinline__ void start(const LatSeqs &sq, int t) {
        idle();
        if (t >= sq.n_tiles) return;
        left = min(sq.per, sq.n_tiles - t);
        int lo = 0, hi = sq.n;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (first(sq, mid) <= t) lo = mid; else hi = mid;
        }
        si = lo;
        chunk = t - first(sq, lo);
        n = first(sq, lo + 1) - first(sq, lo);
    }
    __device__ __forceinline__ int valid(const LatSeqs &sq) const {
        return left == 0 ? 0 : chunk + 1 < n ? TILE : (int)(sq.first[si] >> 24) + 1;
    }
    __device__ __forceinline__ bool ends_run() const { return left == 1 || (left > 0 && chunk + 1 == n); }
    __device__ __forceinline__ void next(const LatSeqs &sq) {
        if (left == 0) return;
        if (--left == 0) {
            idle();
            return;
        }
        if (++chunk == n) {
            do {
                ++si;
                n = first(sq, si + 1) - first(sq, si);
            } while (n == 0);
            chunk = 0;
        }
    }
};

// (the tile kernel looks before it waits: see kvcar_pdl.cuh)
__device__ __noinline__ int pool_row(const int32_t *table, int page_tokens, int tok) {
    return table[tok / page_tokens] * page_tokens + tok % page_tokens;
}
__device__ __forceinline__ float redux_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
// N values per lane (N = 6, 8 or 16): afterwards lane L holds the maximum (or the sum) over the warp of value L (L < N); halves
// the values while it halves the lanes' distance, so about N shuffles instead of 5 N
template <int N, bool SUM>
__device__ __forceinline__ float over_lanes(const float *v, int lane) {
    constexpr int P = N <= 8 ? 8 : 16;
    float x[P];
    auto fold = [](float a, float b) { return SUM ? a + b : fmaxf(a, b); };
#pragma unroll
    for (int i = 0; i < P; ++i) x[i] = i < N ? v[i] : SUM ? 0.f : -INFINITY;
#pragma unroll
    for (int w = P / 2; w > 0; w >>= 1) {
        const bool up = (lane & w) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const float keep = up ? x[i + w] : x[i], give = up ? x[i] : x[i + w];
            x[i] = fold(keep, __shfl_xor_sync(0xffffffffu, give, w));
        }
    }
#pragma unroll
    for (int w = P; w < 32; w <<= 1) x[0] = fold(x[0], __shfl_xor_sync(0xffffffffu, x[0], w));
    return x[0];
}
__device__ __forceinline__ float ex2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void stmatrix_x4(uint32_t addr, const uint32_t *w) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                 : "memory");
}
__device__ __forceinline__ void st_smem_u16(uint32_t addr, uint16_t v) {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}

// *p = v if i < limit, without a branch
__device__ __forceinline__ void st_global_below(float *p, float v, int i, int limit) {
    asm volatile("{\n .reg .pred p;\n setp.lt.s32 p, %2, %3;\n @p st.global.f32 [%0], %1;\n}" ::"l"(p), "f"(v), "r"(i), "r"(limit) : "memory");
}

// what the warps share besides operands and barriers (everything is dynamic shared memory, so that the operand places
// start at an aligned address and nothing is lost to padding)
template <int NQ>
struct __align__(8) Scratch {
    uint32_t tmem_slot;
    int abort_flag;
    float mrun[2][NQ];    // by tile parity: reference maximum before the tile
    float red[2][NQ][4];  // by tile parity: maxima of the four lane quarters
    float lred[NQ][4];    // sums of the four lane quarters at the end of a run
};

// ---------------------------------------------------------------------------- optional time stamps
// Compiled with -DKVCAR_TRACE, six threads of one cluster (in both CTAs: the two loading ones, the two issuing ones of the leader,
// lane 0 of the first hidden and of the first output warp) record (clock64 << 8) | tag at the points marked TR;
// kvcar_debug_trace_select picks the cluster, kvcar_debug_trace_dump fetches the records of the last launch.  Without the macro the
// marks compile to nothing.  Tags: loads 2 = a latent or weight slab's load issued, 3 = a query slab's; issuers 0x10 | kind = the
// accumulator is free, a job begins (kind 1 = hidden chunk, 3 = S, 4 = a block of U), 0x30 = a slab's operands are in place, 0x31 = its
// products and releases are issued, 0x19 = job committed; hidden and output warps (kind << 4) | phase with kind 4 = hidden chunk,
// 7 = S and its probabilities, 8 = a block of U and phase 0 = waits for the job, 1 = job seen complete, 2 = accumulator read and given
// back, 3 = done with the job.
enum { TR_ROWS, TR_WEIGHTS, TR_HIDDEN_ISSUE, TR_HIDDEN, TR_OUT_ISSUE, TR_OUT, TR_ROLES };
#ifdef KVCAR_TRACE
constexpr int TRACE_LEN = 4096;
__device__ unsigned long long g_trace[2][TR_ROLES][TRACE_LEN];
__device__ int g_trace_n[2][TR_ROLES];
__device__ int g_trace_cluster = 0;
#define TR(role, tag)                                                                                       \
    do {                                                                                                    \
        if (tr_on) {                                                                                        \
            if (tr_cnt < TRACE_LEN) g_trace[rank][role][tr_cnt++] = ((unsigned long long)clock64() << 8) | (unsigned)(tag); \
            g_trace_n[rank][role] = tr_cnt;                                                                 \
        }                                                                                                   \
    } while (0)
#else
#define TR(role, tag) \
    do {              \
    } while (0)
#endif

// NQ: query heads padded.  NB: U blocks of 128 hidden features at most; fixes the registers of the running sums.  CN: hidden columns
// of a job.  Q8: int8 rows, whose hidden vectors are two bf16 terms.  P2: two operands for the probabilities (NQ = 32).
template <int NQ, int NB, int CN, bool Q8, bool P2>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(n_threads(CN), 1)
    decode_latent_kernel(const __grid_constant__ Params a) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    constexpr int R = op_rows(NQ), PSLAB = R * 128, QSLAB = wq_slab(NQ), WSTAGE = wstage(CN), CSLABS = CN / 64;
    constexpr int TERMS = Q8 ? 2 : 1, P_SLABS = P2 ? 4 : 2;
    constexpr int TM_OUT = 2 * CN;  // tensor-memory columns: hidden 0, CN; outputs 2 CN, 2 CN + 64
    constexpr int N_HID = 4 * CSLABS, OUT_WARP = HID_WARP + N_HID;
    static_assert(TERMS == 1 || CSLABS == 2, "a term of a job is a pair of slabs");
    static_assert(!P2 || NQ > 16, "up to 16 heads both terms of the probabilities are rows of one operand");

    const uint32_t rank = blockIdx.x & 1u;
    const bool leader = rank == 0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#ifdef KVCAR_TRACE
    // one thread of warps 0 to 3 runs their loops
    const bool tr_on = (int)(blockIdx.x >> 1) == g_trace_cluster && (warp < HID_WARP || ((warp == HID_WARP || warp == OUT_WARP) && lane == 0));
    int tr_cnt = 0;
#endif
    const uint32_t s_z = smem_u32(smem_raw), s_h = s_z + a.nz * SLAB, s_w = s_h + a.nh * SLAB, s_q = s_w + a.nw * WSTAGE;
    const uint32_t s_p = s_q + a.nqs * QSLAB, s_bar = s_p + P_SLABS * PSLAB;
    const uint32_t w_full = s_bar, w_empty = w_full + 8 * a.nw;
    const uint32_t z_full = w_empty + 8 * a.nw, z_empty = z_full + 8 * a.nz;
    const uint32_t q_full = z_empty + 8 * a.nz, q_empty = q_full + 8 * a.nqs;
    const uint32_t h_ready = q_empty + 8 * a.nqs, h_free = h_ready + 8 * READY_BARS;
    const uint32_t t_full = h_free + 8 * a.nh, t_empty = t_full + 16, o_full = t_empty + 16, o_empty = o_full + 16;
    const uint32_t p_ready = o_empty + 16;
    Scratch<NQ> &sh = *reinterpret_cast<Scratch<NQ> *>(smem_raw + (p_ready + 8 - s_z));
    volatile int &abort_flag = sh.abort_flag;
    // pair of runs, and which part of a side's hidden columns (one part unless the grid is small)
    const int pair = (int)(blockIdx.x >> 1) / a.n_parts, part = (int)(blockIdx.x >> 1) % a.n_parts;
    const int side_lo = a.mode == MODE_V ? 1 : 0, side_hi = a.mode == MODE_K ? 1 : 2;
    // (opaque to the compiler, as `lag` below: it would make two copies of every loop, one per mode)
    int list0 = a.mode == MODE_BOTH ? 0 : part, list_step = a.mode == MODE_BOTH ? 1 : 0;
    asm volatile("" : "+r"(list0), "+r"(list_step));
    auto list_of = [&](int side) -> const LatList & { return a.list[list0 + side * list_step]; };
    // tiles of the cluster's longer run (the leader's); the other CTA idles through the last ones it does not have
    const int my_run = 2 * pair + (int)rank;
    const int n_it = max(0, min(a.sq.per, a.sq.n_tiles - 2 * pair * a.sq.per));
    const int my_first = my_run * a.sq.per;
    // MODE_BOTH: in step `it` the K side of tile `it`, then the V side of the tile before
    const int lag = list_step, n_steps = n_it > 0 ? n_it + lag : 0;
    auto tile_of = [&](int it, int side) { return it - (side == 1 ? lag : 0); };
    auto on = [&](int it, int side) { return tile_of(it, side) >= 0 && tile_of(it, side) < n_it; };
    launch_dependents();

    if (threadIdx.x == 0) {
        sh.abort_flag = 0;
#pragma unroll 1
        for (int i = 0; i < a.nw; ++i) {
            mbar_init(w_full + 8 * i, 1);
            mbar_init(w_empty + 8 * i, 1);
        }
#pragma unroll 1
        for (int i = 0; i < a.nz; ++i) {
            mbar_init(z_full + 8 * i, 1);
            mbar_init(z_empty + 8 * i, 1);
        }
#pragma unroll 1
        for (int i = 0; i < a.nqs; ++i) {
            mbar_init(q_full + 8 * i, 1);
            mbar_init(q_empty + 8 * i, 1);
        }
#pragma unroll 1
        for (int i = 0; i < a.nh; ++i) mbar_init(h_free + 8 * i, 1);
#pragma unroll 1
        for (int i = 0; i < READY_BARS; ++i) mbar_init(h_ready + 8 * i, 2 * N_HID);
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
            mbar_init(t_full + 8 * i, 1);
            mbar_init(t_empty + 8 * i, 2 * N_HID);
            mbar_init(o_full + 8 * i, 1);
            mbar_init(o_empty + 8 * i, 2 * N_OUT);
        }
        mbar_init(p_ready, 2 * N_OUT);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (threadIdx.x < 2 * NQ) sh.mrun[threadIdx.x / NQ][threadIdx.x % NQ] = -INFINITY;
    if (warp == 1) {  // all of tensor memory in both CTAs (one CTA per SM by shared memory)
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem_slot)), "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers exist before either signals the other's
    tc_fence_after();
    const uint32_t tmem = sh.tmem_slot;

    if (warp == 0) {
        // ============================== latents, query rows ==============================
        // Two independent streams of loads, each into its own ring; one thread looks at the rings in turn and fills the
        // one that has a place.
        if (elect_one()) {
            auto rows_of = [&](const TileWalk &t, int *r) {  // pool rows of the tile's two 64-token halves
                r[0] = r[1] = 0;
                const int v = t.valid(a.sq);
                if (v == 0) return;
                const int tok = t.chunk * TILE;
                if (Q8) {  // widened rows lie in the order of the launch's tiles
                    r[0] = (t.first(a.sq, t.si) + t.chunk) * TILE;
                    r[1] = r[0] + (v > 64 ? 64 : 0);
                    return;
                }
                const int32_t *table = a.block_table + (int64_t)a.sq.id[t.si] * a.max_pages_per_seq;
                r[0] = pool_row(table, a.page_tokens, tok);
                r[1] = v > 64 ? pool_row(table, a.page_tokens, tok + 64) : r[0];  // no valid token there: re-read the first half
            };
            struct Pos {
                int it, side, s, k;
            };
            Pos z{0, side_lo, 0, 0}, q{a.mode == MODE_V ? n_it : 0, 0, 0, 0};
            bool waited = false;  // for the launch before, which writes the query rows
            uint32_t zslot = 0, zphase = 0, qslot = 0, qphase = 0;
            TileWalk zw, qw;
            zw.start(a.sq, my_first);
            qw = zw;
            int prow[2] = {0, 0}, row[2], nrow[2] = {0, 0};  // of the tile before, of tile z.it, of the next
            bool live = zw.left > 0, nlive = false;          // row, nrow are of a tile of this CTA
            rows_of(zw, row);
            const bool low_k = NQ <= 16 || a.two_terms_k;
            uint32_t idle = 0;
            uint64_t t0 = 0;
            while (z.it < n_steps || q.it < n_it) {
                bool moved = false;
                if (z.it < n_steps && mbar_test(z_empty + 8 * zslot, zphase ^ 1u)) {
                    moved = true;
                    if (leader) mbar_expect_tx(z_full + 8 * zslot, 2 * SLAB);
                    const LatSrc &zp_ = list_of(z.side).src[z.s];
                    const CUtensorMap *map = &a.pool[z.side][zp_.map];
                    const uint32_t fb = map_to_cta(z_full + 8 * zslot, 0), dst = s_z + zslot * SLAB;
                    const bool behind = tile_of(z.it, z.side) < z.it;  // the tile before
                    tma_load_2d_pair(dst, map, z.k * 64, behind ? prow[0] : row[0], fb);
                    tma_load_2d_pair(dst + SLAB / 2, map, z.k * 64, behind ? prow[1] : row[1], fb);
                    TR(TR_ROWS, 2);
                    if (++zslot == (uint32_t)a.nz) { zslot = 0; zphase ^= 1u; }
                    const int ks1 = (zp_.d + 63) >> 6;
                    if (++z.k == ks1) {
                        // the same rows of the tile after: from HBM into L2 while this one is worked on
                        if (z.side == side_lo && z.s == 0) {
                            zw.next(a.sq);
                            rows_of(zw, nrow);
                            nlive = zw.left > 0;
                        }
                        if (behind ? live : nlive) {
                            const int r0 = behind ? row[0] : nrow[0], r1 = behind ? row[1] : nrow[1];
#pragma unroll 1
                            for (int ks = 0; ks < ks1; ++ks) {
                                tma_prefetch_2d(map, ks * 64, r0);
                                if (r1 != r0) tma_prefetch_2d(map, ks * 64, r1);
                            }
                        }
                        z.k = 0;
                        if (++z.s == list_of(z.side).n) {
                            z.s = 0;
                            do {
                                if (++z.side == side_hi) {
                                    z.side = side_lo;
                                    ++z.it;
#pragma unroll
                                    for (int h = 0; h < 2; ++h) {
                                        prow[h] = row[h];
                                        row[h] = nrow[h];
                                    }
                                    live = nlive;
                                    nlive = false;
                                }
                            } while (z.it < n_steps && !on(z.it, z.side));
                        }
                    }
                }
                if (!waited && a.mode != MODE_V && (!moved || z.it > 0 || z.side > side_lo)) {
                    grid_dependency_wait();
                    waited = moved = true;
                }
                if (waited && q.it < n_it && mbar_test(q_empty + 8 * qslot, qphase ^ 1u)) {
                    moved = true;
                    const LatSrc &sp = list_of(0).src[q.s];
                    const int y = (sp.map * a.wq_batch + qw.si) * wq_rows(NQ), x = sp.c0 + q.k * 64;
                    if (leader) mbar_expect_tx(q_full + 8 * qslot, low_k ? 2 * QSLAB : QSLAB);
                    const uint32_t fb = map_to_cta(q_full + 8 * qslot, 0), dst = s_q + qslot * QSLAB;
                    tma_load_2d_pair(dst, &a.tm_wq, x, y, fb);
                    if (NQ > 16 && low_k) tma_load_2d_pair(dst + QSLAB / 2, &a.tm_wq, x, y + R, fb);
                    TR(TR_ROWS, 3);
                    if (++qslot == (uint32_t)a.nqs) { qslot = 0; qphase ^= 1u; }
                    if (++q.k == (sp.m + 63) >> 6) {
                        q.k = 0;
                        if (++q.s == list_of(0).n) {
                            q.s = 0;
                            ++q.it;
                            qw.next(a.sq);
                        }
                    }
                }
                if (moved) {
                    t0 = 0;
                    idle = 0;
                } else {
                    __nanosleep(20);
                    if ((++idle & 255u) == 0) {
                        const uint64_t now = global_ns();
                        if (t0 == 0) t0 = now;
                        if (now - t0 > (abort_flag ? 2000000ull : 2000000000ull)) {
                            abort_flag = 1;
                            atomicCAS(a.status, 0, 0x601);
                            break;
                        }
                    }
                }
            }
            if (!waited) grid_dependency_wait();  // every block sees the launches before complete: those after rely on it
        }
    } else if (warp == 2) {
        // ============================== weight loads ==============================
        if (elect_one()) {
            uint32_t slot = 0, phase = 0;
#pragma unroll 1
            for (int it = 0; it < n_steps; ++it)
#pragma unroll 1
                for (int side = side_lo; side < side_hi; ++side)
#pragma unroll 1
                    for (int s = 0; s < (on(it, side) ? list_of(side).n : 0); ++s) {
                        const LatSrc &sp = list_of(side).src[s];
                        const int ks1 = (sp.d + 63) >> 6, m = sp.m;
                        const CUtensorMap *map = &a.w1[side][sp.map];
#pragma unroll 1
                        for (int c0 = 0; c0 < m; c0 += CN) {
                            const int y = sp.c0 + c0 + (int)rank * (min(CN, m - c0) >> 1);
#pragma unroll 1
                            for (int ks = 0; ks < ks1; ++ks) {
                                mbar_wait(w_empty + 8 * slot, phase ^ 1u, a.status, &abort_flag, 0x602);
                                if (leader) mbar_expect_tx(w_full + 8 * slot, 2 * WSTAGE);
                                tma_load_2d_pair(s_w + slot * WSTAGE, map, ks * 64, y, map_to_cta(w_full + 8 * slot, 0));
                                TR(TR_WEIGHTS, 2);
                                if (++slot == (uint32_t)a.nw) { slot = 0; phase ^= 1u; }
                            }
                        }
                    }
        }
    } else if (warp == 1) {
        // ============================== hidden products (leader CTA) ==============================
        if (leader && elect_one()) {
            uint32_t wslot = 0, wphase = 0, zslot = 0, zphase = 0, h = 0;
            const uint64_t z_desc = make_desc(s_z), w_desc = make_desc(s_w);
#pragma unroll 1
            for (int it = 0; it < n_steps; ++it)
#pragma unroll 1
                for (int side = side_lo; side < side_hi; ++side)
#pragma unroll 1
                    for (int s = 0; s < (on(it, side) ? list_of(side).n : 0); ++s) {
                        const int d = list_of(side).src[s].d, m = list_of(side).src[s].m;
                        const int ks1 = (d + 63) >> 6, nk_last = ((d - 1) & 63) / 16 + 1;
                        uint32_t zs = 0, zp = 0;
#pragma unroll 1
                        for (int c0 = 0; c0 < m; c0 += CN, ++h) {
                            const bool first = c0 == 0, last = c0 + CN >= m;
                            const uint32_t buf = h & 1u, acc = tmem + CN * buf, idesc = make_idesc(256, min(CN, m - c0));
                            mbar_wait(t_empty + 8 * buf, ((h >> 1) & 1u) ^ 1u, a.status, &abort_flag, 0x607);
                            tc_fence_after();
                            TR(TR_HIDDEN_ISSUE, 0x11);
                            zs = zslot;  // the source's latent slabs: places zslot ..
                            zp = zphase;
#pragma unroll 1
                            for (int ks = 0; ks < ks1; ++ks) {
                                if (first) mbar_wait(z_full + 8 * zs, zp, a.status, &abort_flag, 0x608);
                                mbar_wait(w_full + 8 * wslot, wphase, a.status, &abort_flag, 0x603);
                                TR(TR_HIDDEN_ISSUE, 0x30);
                                const uint64_t da = z_desc + zs * (SLAB >> 4), db = w_desc + wslot * (WSTAGE >> 4);
                                if (ks == 0)
                                    umma_pair<0>(acc, da, db, idesc);
                                else
                                    umma_pair<1>(acc, da, db, idesc);
                                if (ks + 1 < ks1 || nk_last == 4) {
                                    umma_pair<1>(acc, da + 2u, db + 2u, idesc);
                                    umma_pair<1>(acc, da + 4u, db + 4u, idesc);
                                    umma_pair<1>(acc, da + 6u, db + 6u, idesc);
                                } else {
#pragma unroll 1
                                    for (int t = 1; t < nk_last; ++t) umma_pair<1>(acc, da + 2u * t, db + 2u * t, idesc);
                                }
                                umma_commit_pair(w_empty + 8 * wslot);
                                if (last) umma_commit_pair(z_empty + 8 * zs);
                                TR(TR_HIDDEN_ISSUE, 0x31);
                                if (++wslot == (uint32_t)a.nw) { wslot = 0; wphase ^= 1u; }
                                if (++zs == (uint32_t)a.nz) { zs = 0; zp ^= 1u; }
                            }
                            umma_commit_pair(t_full + 8 * buf);
                            TR(TR_HIDDEN_ISSUE, 0x19);
                        }
                        zslot = zs;
                        zphase = zp;
                    }
        }
    } else if (warp == 3) {
        // ============================== S and U products (leader CTA) ==============================
        if (leader && elect_one()) {
            uint32_t qslot = 0, qphase = 0, hslot = 0, h = 0, o = 0;
            constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(2 * R >> 3) << 17) | (16u << 24);
            constexpr uint32_t idesc_u = idesc | (1u << 15);  // row operand MN-major
            const uint64_t h_desc = make_desc(s_h), q_desc = make_desc(s_q), p_desc = make_desc(s_p);
            const bool two = NQ > 16 && a.two_terms_k;
#pragma unroll 1
            for (int it = 0; it < n_steps; ++it) {
#pragma unroll 1
                for (int s = 0; s < (side_lo == 0 && on(it, 0) ? list_of(0).n : 0); ++s) {  // S
                    const uint32_t ob = o & 1u, acc = tmem + TM_OUT + 64u * ob;
                    mbar_wait(o_empty + 8 * ob, ((o >> 1) & 1u) ^ 1u, a.status, &abort_flag, 0x605);
                    TR(TR_OUT_ISSUE, 0x13);
                    bool begin = true;
                    const int m = list_of(0).src[s].m, ksm = (m + 63) >> 6, nk_last = ((m - 1) & 63) / 16 + 1;
                    if constexpr (TERMS == 2) {
#pragma unroll 1
                        for (int sl0 = 0; sl0 < ksm; sl0 += CSLABS) {
                            const int n_sl = min(CSLABS, ksm - sl0);
                            uint32_t qs = qslot, qp = qphase;
#pragma unroll 1
                            for (int term = 0; term < TERMS; ++term) {  // both terms meet the same query slabs
                                hslot += hslot & 1u;
                                if (hslot == (uint32_t)a.nh) hslot = 0;
                                mbar_wait(h_ready + 8 * (h & 7u), (h >> 3) & 1u, a.status, &abort_flag, 0x604);
                                tc_fence_after();
                                ++h;
                                qs = qslot;
                                qp = qphase;
#pragma unroll 1
                                for (int i = 0; i < n_sl; ++i) {
                                    mbar_wait(q_full + 8 * qs, qp, a.status, &abort_flag, 0x60e);
                                    TR(TR_OUT_ISSUE, 0x30);
                                    const uint64_t da = h_desc + hslot * (SLAB >> 4), db = q_desc + qs * (QSLAB >> 4);
                                    const int nk = sl0 + i + 1 < ksm ? 4 : nk_last;
                                    if (begin)
                                        umma_pair<0>(acc, da, db, idesc);
                                    else
                                        umma_pair<1>(acc, da, db, idesc);
                                    begin = false;
#pragma unroll 1
                                    for (int t = 1; t < nk; ++t) umma_pair<1>(acc, da + 2u * t, db + 2u * t, idesc);
                                    if (two && term == 0) {
#pragma unroll 1
                                        for (int t = 0; t < nk; ++t) umma_pair<1>(acc, da + 2u * t, db + (QSLAB / 2 >> 4) + 2u * t, idesc);
                                    }
                                    umma_commit_pair(h_free + 8 * hslot);
                                    if (term + 1 == TERMS) umma_commit_pair(q_empty + 8 * qs);
                                    TR(TR_OUT_ISSUE, 0x31);
                                    if (++hslot == (uint32_t)a.nh) hslot = 0;
                                    if (++qs == (uint32_t)a.nqs) { qs = 0; qp ^= 1u; }
                                }
                            }
                            qslot = qs;
                            qphase = qp;
                        }
                    } else {
#pragma unroll 1
                        for (int sl = 0, in_job = 0; sl < ksm; ++sl) {
                            if (in_job == 0) {  // the job's slabs, written by both CTAs
                                mbar_wait(h_ready + 8 * (h & 7u), (h >> 3) & 1u, a.status, &abort_flag, 0x604);
                                tc_fence_after();
                                ++h;
                            }
                            if (++in_job == CSLABS) in_job = 0;
                            mbar_wait(q_full + 8 * qslot, qphase, a.status, &abort_flag, 0x60e);
                            TR(TR_OUT_ISSUE, 0x30);
                            const uint64_t da = h_desc + hslot * (SLAB >> 4), db = q_desc + qslot * (QSLAB >> 4);
                            if (begin)
                                umma_pair<0>(acc, da, db, idesc);
                            else
                                umma_pair<1>(acc, da, db, idesc);
                            begin = false;
                            const int nk = sl + 1 < ksm ? 4 : nk_last;
                            if (nk > 1) umma_pair<1>(acc, da + 2u, db + 2u, idesc);
                            if (nk > 2) umma_pair<1>(acc, da + 4u, db + 4u, idesc);
                            if (nk > 3) umma_pair<1>(acc, da + 6u, db + 6u, idesc);
                            if (two) {
                                const uint64_t dl = db + (QSLAB / 2 >> 4);
                                umma_pair<1>(acc, da, dl, idesc);
                                if (nk > 1) umma_pair<1>(acc, da + 2u, dl + 2u, idesc);
                                if (nk > 2) umma_pair<1>(acc, da + 4u, dl + 4u, idesc);
                                if (nk > 3) umma_pair<1>(acc, da + 6u, dl + 6u, idesc);
                            }
                            umma_commit_pair(h_free + 8 * hslot);
                            umma_commit_pair(q_empty + 8 * qslot);
                            TR(TR_OUT_ISSUE, 0x31);
                            if (++hslot == (uint32_t)a.nh) hslot = 0;
                            if (++qslot == (uint32_t)a.nqs) { qslot = 0; qphase ^= 1u; }
                        }
                    }
                    umma_commit_pair(o_full + 8 * ob);
                    TR(TR_OUT_ISSUE, 0x19);
                    ++o;
                }
                bool p_seen = false;
#pragma unroll 1
                for (int s = 0; s < (side_hi == 2 && on(it, 1) ? list_of(1).n : 0); ++s) {  // U
                    const int ksm = (list_of(1).src[s].m + 63) >> 6;
                    if constexpr (TERMS == 2) {
#pragma unroll 1
                        for (int sl0 = 0; sl0 < ksm; sl0 += CSLABS) {
                            const uint32_t ob = o & 1u, accu = tmem + TM_OUT + 64u * ob;
#pragma unroll 1
                            for (int term = 0; term < TERMS; ++term) {
                                hslot += hslot & 1u;
                                if (hslot == (uint32_t)a.nh) hslot = 0;
                                mbar_wait(h_ready + 8 * (h & 7u), (h >> 3) & 1u, a.status, &abort_flag, 0x604);
                                ++h;
                                if (!p_seen) {
                                    mbar_wait(p_ready, (uint32_t)tile_of(it, 1) & 1u, a.status, &abort_flag, 0x606);
                                    p_seen = true;
                                }
                                if (term == 0) {
                                    mbar_wait(o_empty + 8 * ob, ((o >> 1) & 1u) ^ 1u, a.status, &abort_flag, 0x605);
                                    TR(TR_OUT_ISSUE, 0x14);
                                }
                                tc_fence_after();
                                TR(TR_OUT_ISSUE, 0x30);
                                uint64_t da = h_desc + hslot * (SLAB >> 4);  // as below
                                da = (da & ~((uint64_t)0x3FFF << 16)) | ((uint64_t)(SLAB >> 4) << 16);
                                if (term == 0)
                                    umma_pair<0>(accu, da, p_desc, idesc_u);
                                else
                                    umma_pair<1>(accu, da, p_desc, idesc_u);
#pragma unroll
                                for (int t = 1; t < TILE / 16; ++t)
                                    umma_pair<1>(accu, da + (uint64_t)(t * (16 * 128 >> 4)),
                                                 p_desc + (uint64_t)((t >> 2) * (PSLAB >> 4) + (t & 3) * 2), idesc_u);
                                if (P2 && term == 0 && a.two_terms_v) {
#pragma unroll
                                    for (int t = 0; t < TILE / 16; ++t)
                                        umma_pair<1>(accu, da + (uint64_t)(t * (16 * 128 >> 4)),
                                                     p_desc + (uint64_t)((2 + (t >> 2)) * (PSLAB >> 4) + (t & 3) * 2), idesc_u);
                                }
                                umma_commit_pair(h_free + 8 * hslot);
                                if (sl0 + 1 < ksm) umma_commit_pair(h_free + 8 * (hslot + 1));
                                TR(TR_OUT_ISSUE, 0x31);
                                hslot += min(CSLABS, ksm - sl0);
                                if (hslot == (uint32_t)a.nh) hslot = 0;
                            }
                            umma_commit_pair(o_full + 8 * ob);
                            TR(TR_OUT_ISSUE, 0x19);
                            ++o;
                        }
                        continue;
                    }
                    hslot += hslot & 1u;  // slabs go in pairs: a source starts at an even place
                    if (hslot == (uint32_t)a.nh) hslot = 0;
#pragma unroll 1
                    for (int sl = 0, in_job = 0; sl < ksm; ++sl) {
                        if (in_job == 0) {
                            mbar_wait(h_ready + 8 * (h & 7u), (h >> 3) & 1u, a.status, &abort_flag, 0x604);
                            tc_fence_after();
                            ++h;
                        }
                        if (++in_job == CSLABS) in_job = 0;
                        const uint32_t hs = hslot;
                        if (++hslot == (uint32_t)a.nh) hslot = 0;
                        if (!(sl & 1) && sl + 1 < ksm) continue;
                        if (!p_seen) {
                            mbar_wait(p_ready, (uint32_t)tile_of(it, 1) & 1u, a.status, &abort_flag, 0x606);
                            p_seen = true;
                        }
                        const uint32_t ob = o & 1u, accu = tmem + TM_OUT + 64u * ob, h0 = hs & ~1u;
                        mbar_wait(o_empty + 8 * ob, ((o >> 1) & 1u) ^ 1u, a.status, &abort_flag, 0x605);
                        tc_fence_after();
                        TR(TR_OUT_ISSUE, 0x14);
                        TR(TR_OUT_ISSUE, 0x30);
                        // rows = features: two 64-feature atoms a slab apart, 8-token groups 1 KB apart (MN-major)
                        uint64_t da = h_desc + h0 * (SLAB >> 4);
                        da = (da & ~((uint64_t)0x3FFF << 16)) | ((uint64_t)(SLAB >> 4) << 16);
                        umma_pair<0>(accu, da, p_desc, idesc_u);
#pragma unroll
                        for (int t = 1; t < TILE / 16; ++t)
                            umma_pair<1>(accu, da + (uint64_t)(t * (16 * 128 >> 4)),
                                         p_desc + (uint64_t)((t >> 2) * (PSLAB >> 4) + (t & 3) * 2), idesc_u);
                        if (P2 && a.two_terms_v) {
#pragma unroll
                            for (int t = 0; t < TILE / 16; ++t)
                                umma_pair<1>(accu, da + (uint64_t)(t * (16 * 128 >> 4)),
                                             p_desc + (uint64_t)((2 + (t >> 2)) * (PSLAB >> 4) + (t & 3) * 2), idesc_u);
                        }
                        umma_commit_pair(h_free + 8 * h0);
                        if (hs != h0) umma_commit_pair(h_free + 8 * hs);
                        umma_commit_pair(o_full + 8 * ob);
                        TR(TR_OUT_ISSUE, 0x31);
                        TR(TR_OUT_ISSUE, 0x19);
                        ++o;
                    }
                }
            }
        }
    } else if (warp < OUT_WARP) {
        // ============================== hidden warps (both CTAs) ==============================
        const int my_slab = (warp - HID_WARP) >> 2;   // this warp's slab of a job
        const uint32_t lane_base = 32u * (warp & 3);  // tensor-memory lane quarter of this warp
        // where this lane's row of the 8 x 8 blocks goes (row lane % 8 of 8, block lane / 8 of 4; 128-byte swizzle)
        const uint32_t st_row = (lane_base + (lane & 7)) * 128u;
        const uint32_t ready_leader = map_to_cta(h_ready, 0), empty_leader = map_to_cta(t_empty, 0);
        uint32_t hslot = 0, hphase = 0, h = 0, r_job = 0;  // h: accumulators read, r_job: terms written
        TileWalk tw;
        tw.start(a.sq, my_first);
        auto wide_row = [&]() { return !Q8 || tw.left == 0 ? 0 : (tw.first(a.sq, tw.si) + tw.chunk) * TILE; };
        int k_valid = tw.valid(a.sq), k_row = wide_row(), v_valid = k_valid, v_row = k_row;  // of the K and of the V side's tile
#pragma unroll 1
        for (int it = 0; it < n_steps; ++it) {
#pragma unroll 1
            for (int side = side_lo; side < side_hi; ++side) {
                if (!on(it, side)) continue;
                const int valid = side == 0 ? k_valid : v_valid;
                const int n_src = list_of(side).n;
#pragma unroll 1
                for (int s = 0; s < n_src; ++s) {
                    const int m = list_of(side).src[s].m;
                    const float slope = list_of(side).src[s].slope;
                    const float2 slope2 = make_float2(slope, slope);
                    // V side: rows past the tile's end may hold anything, and zero times a stray NaN is not zero
                    const bool clear = side == 1 && valid < TILE;
                    if (side == 1) {
                        hslot += hslot & 1u;
                        if (hslot == (uint32_t)a.nh) hslot = 0;
                    }
                    float inv[4] = {1.f, 1.f, 1.f, 1.f}, left[4] = {0.f, 0.f, 0.f, 0.f};  // int8 rows: this lane's four tokens
                    bool any_left = false;
                    if (Q8) {
                        const int r0 = side == 0 ? k_row : v_row;
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int r = (int)lane_base + 8 * i + (lane >> 2);
                            if (r < valid) {
                                const float2 p = __ldcg(list_of(side).src[s].rowp + r0 + r);  // past the first-level cache: see kvcar_pdl.cuh
                                inv[i] = p.x;
                                left[i] = p.y;
                            }
                            any_left |= left[i] != 0.f;
                        }
                        any_left = __any_sync(0xffffffffu, any_left);
                    }
                    const float *shift = list_of(side).src[s].shift;
#pragma unroll 1
                    for (int c0 = 0; c0 < m; c0 += CN, ++h) {
                        const int nc = min(CN, m - c0);
                        const uint32_t buf = h & 1u, acc = tmem + CN * buf + (lane_base << 16);
                        const int col0 = 64 * my_slab, halves = col0 >= nc ? 0 : col0 + 32 >= nc ? 1 : 2;
                        const float4 *t4 = reinterpret_cast<const float4 *>(shift + c0 + col0) + 2 * (lane & 3);
                        float4 ta = make_float4(0.f, 0.f, 0.f, 0.f), tb = ta;
                        if (halves > 0) {
                            ta = __ldg(t4);
                            tb = __ldg(t4 + 1);
                        }
                        TR(TR_HIDDEN, 0x40);
                        mbar_wait(t_full + 8 * buf, (h >> 1) & 1u, a.status, &abort_flag, 0x609);
                        __syncwarp();
                        tc_fence_after();
                        TR(TR_HIDDEN, 0x41);
                        // The accumulator is read, and given back, before the job's places in the ring are free: the next
                        // hidden products do not wait for the products that still read those places.
                        uint32_t w[TERMS][2][16];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {  // 32 columns (u / 2) x 16 of the warp's 32 rows (u % 2)
                            const int half = u >> 1, f = u & 1;
                            if (half < halves) {
                                if (u == 2) {
                                    ta = __ldg(t4 + 8);
                                    tb = __ldg(t4 + 9);
                                }
                                const float2 t[4] = {make_float2(ta.x, ta.y), make_float2(ta.z, ta.w), make_float2(tb.x, tb.y),
                                                     make_float2(tb.z, tb.w)};
                                uint32_t r[16];
                                tmem_ld_frag_x4(acc + (uint32_t)f * (16u << 16) + (uint32_t)(col0 + 32 * half), r);
                                tmem_ld_wait(r);
                                if (f == 1 && half + 1 == halves) {
                                    tc_fence_before();
                                    __syncwarp();
                                    if (elect_one()) mbar_arrive_remote(empty_leader + 8 * buf);
                                }
                                if (Q8 && any_left) {
#pragma unroll
                                    for (int e = 0; e < 8; ++e) {
                                        const int i = e >> 2, j = e & 3;
                                        const float2 rs = __ldg(reinterpret_cast<const float2 *>(list_of(side).src[s].rowsum + c0 + col0 + 32 * half) +
                                                                4 * (lane & 3) + j);
                                        r[4 * j + 2 * i] = __float_as_uint(fmaf(-left[2 * f + i], rs.x, __uint_as_float(r[4 * j + 2 * i])));
                                        r[4 * j + 2 * i + 1] = __float_as_uint(fmaf(-left[2 * f + i], rs.y, __uint_as_float(r[4 * j + 2 * i + 1])));
                                    }
                                }
#pragma unroll
                                for (int e = 0; e < 8; ++e) {  // rows 8 (e / 4) .. of the 16
                                    const int i = e >> 2, j = e & 3;
                                    const float2 h2 = make_float2(__uint_as_float(r[4 * j + 2 * i]), __uint_as_float(r[4 * j + 2 * i + 1]));
                                    const float iv = inv[2 * f + i];
                                    const float2 x = Q8 ? __ffma2_rn(h2, make_float2(iv, iv), t[j]) : __fadd2_rn(h2, t[j]);
                                    const float2 y = __fmul2_rn(x, slope2);
                                    const float2 v = make_float2(fmaxf(x.x, y.x), fmaxf(x.y, y.y));  // slope <= 1
                                    const uint32_t hi = pack_bf16(v.x, v.y);
                                    w[0][half][8 * f + e] = hi;
                                    if (TERMS == 2)
                                        w[TERMS - 1][half][8 * f + e] = pack_bf16(v.x - __uint_as_float(hi << 16), v.y - __uint_as_float(hi & 0xffff0000u));
                                }
                            }
                        }
                        if (clear) {
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                if ((int)lane_base + 8 * ((e & 15) >> 2) + (lane >> 2) >= valid) {
                                    w[0][e >> 4][e & 15] = 0u;
                                    w[TERMS - 1][e >> 4][e & 15] = 0u;
                                }
                        }
                        if (halves == 0) {
                            tc_fence_before();
                            __syncwarp();
                            if (elect_one()) mbar_arrive_remote(empty_leader + 8 * buf);
                        }
                        TR(TR_HIDDEN, 0x42);
                        // The job's places in the ring.  A warp writes one of them but sees every one free: a phase that it
                        // skipped would let a later wait on the same place pass one phase early.
                        // One lane per place.
                        const int n_sl = (nc + 63) >> 6;
                        const uint32_t nh = (uint32_t)a.nh;
#pragma unroll
                        for (int term = 0; term < TERMS; ++term) {
                            if (TERMS == 2) {
                                hslot += hslot & 1u;
                                if (hslot == nh) hslot = 0;
                            }
                            const uint32_t place = hslot + lane < nh ? hslot + lane : hslot + lane - nh;
                            if (lane < n_sl) mbar_wait(h_free + 8 * place, ((hphase >> place) & 1u) ^ 1u, a.status, &abort_flag, 0x60a);
                            const uint32_t slot = hslot + my_slab < nh ? hslot + my_slab : hslot + my_slab - nh;
                            const uint32_t passed = ((1u << n_sl) - 1u) << hslot;
                            hphase ^= (passed | passed >> nh) & ((1u << nh) - 1u);
                            hslot = hslot + n_sl < nh ? hslot + n_sl : hslot + n_sl - nh;
                            __syncwarp();
                            const uint32_t dst = s_h + slot * SLAB + st_row;
#pragma unroll
                            for (int half = 0; half < 2; ++half)
                                if (half < halves) {
#pragma unroll
                                    for (int i = 0; i < 4; ++i)
                                        stmatrix_x4(dst + (uint32_t)(((4 * half + (lane >> 3)) ^ (lane & 7)) << 4) + 1024u * i, w[term][half] + 4 * i);
                                }
                            fence_async_smem();
                            __syncwarp();
                            if (elect_one()) mbar_arrive_remote(ready_leader + 8 * (r_job & 7u));
                            ++r_job;
                        }
                        TR(TR_HIDDEN, 0x43);
                    }
                }
            }
            if (lag) {
                v_valid = k_valid;
                v_row = k_row;
            }
            tw.next(a.sq);
            k_valid = tw.valid(a.sq);
            k_row = wide_row();
            if (!lag) {
                v_valid = k_valid;
                v_row = k_row;
            }
        }
    } else {
        // ============================== output warps (both CTAs) ==============================
        // S: thread = token; U: thread = hidden feature of a block.  The two warps of a lane quarter take half of the
        // query heads each.
        constexpr int NT = NQ / 2;
        const int half = (warp - OUT_WARP) >> 2, quarter = warp & 3;
        const int row = 32 * quarter + lane;
        const uint32_t lane_sel = (uint32_t)(32 * quarter) << 16;
        const uint32_t empty_leader = map_to_cta(o_empty, 0), pready_leader = map_to_cta(p_ready, 0);
        const uint32_t col = TM_OUT + R * rank + NT * half;
        const int q0 = NT * half;
        const bool low_v = a.two_terms_v != 0;
        float acc[NB][NT], l = 0.f;  // l: lane q, this warp's part of head q0 + q's sum
#pragma unroll
        for (int q = 0; q < NT; ++q)
#pragma unroll
            for (int b = 0; b < NB; ++b) acc[b][q] = 0.f;
        uint32_t o = 0;
        auto half_sync = [&]() {  // the four warps of this half
            if (half == 0)
                asm volatile("bar.sync 1, 128;" ::: "memory");
            else
                asm volatile("bar.sync 2, 128;" ::: "memory");
        };
        // this warp's columns of the next output accumulator: one value per query head of its half
        auto fetch = [&](float *v, int kind) {
            const uint32_t ob = o & 1u, addr = tmem + lane_sel + col + 64u * ob;
            TR(TR_OUT, kind << 4);
            mbar_wait(o_full + 8 * ob, (o >> 1) & 1u, a.status, &abort_flag, 0x60b);
            __syncwarp();
            tc_fence_after();
            TR(TR_OUT, kind << 4 | 1);
            float r[16];
            tmem_ld8(addr, r);
            tmem_ld8(NQ <= 16 ? addr + NQ : addr + 8u, r + 8);
            tmem_ld_wait(r);
            tc_fence_before();
            __syncwarp();
            if (elect_one()) mbar_arrive_remote(empty_leader + 8 * ob);
            TR(TR_OUT, kind << 4 | 2);
            ++o;
#pragma unroll
            for (int q = 0; q < NT; ++q) v[q] = NQ <= 16 ? r[q] + r[8 + q] : r[q];  // the low terms have columns of their own
        };
        // probabilities of the tile whose scores are s
        auto probabilities = [&](float *s, int valid, int par) {
#pragma unroll
            for (int q = 0; q < NT; ++q)
                if (row >= valid) s[q] = -INFINITY;
            const float keep = over_lanes<NT, false>(s, lane);
            if (lane < NT) sh.red[par][q0 + lane][quarter] = keep;
            half_sync();
            // reference maxima: one head per lane, then broadcast by shuffles of the few values that follow from them
            float m_new = 0.f, f = 1.f;
            if (lane < NT) {
                const float *r = sh.red[par][q0 + lane];
                const float m_old = sh.mrun[par][q0 + lane];
                m_new = fmaxf(m_old, fmaxf(fmaxf(r[0], r[1]), fmaxf(r[2], r[3])));
                if (m_new != m_old) f = ex2(m_old - m_new);
                if (quarter == 0) sh.mrun[par ^ 1][q0 + lane] = m_new;
            }
            const uint32_t t6 = row & 63;
            const uint32_t pbase = s_p + (uint32_t)(row >> 6) * PSLAB + (t6 & 7u) * 2u;
#pragma unroll
            for (int q = 0; q < NT; ++q) {
                const float mq = __shfl_sync(0xffffffffu, m_new, q);
                const float p = valid > 0 ? ex2(s[q] - mq) : 0.f;
                s[q] = p;
                // operand row q0 + q, token t6 of atom row >> 6 (K-major, 128-byte swizzle)
                const uint32_t qr = q0 + q;
                const __nv_bfloat16 hi = __float2bfloat16_rn(p);
                st_smem_u16(pbase + qr * 128u + (((t6 >> 3) ^ (qr & 7u)) << 4), __bfloat16_as_ushort(hi));
                if (NQ <= 16) {
                    const uint32_t ql = qr + NQ;
                    const __nv_bfloat16 lo = __float2bfloat16_rn(low_v ? p - __bfloat162float(hi) : 0.f);
                    st_smem_u16(pbase + ql * 128u + (((t6 >> 3) ^ (ql & 7u)) << 4), __bfloat16_as_ushort(lo));
                } else if (P2) {  // an operand of its own, behind the high terms
                    const __nv_bfloat16 lo = __float2bfloat16_rn(p - __bfloat162float(hi));
                    st_smem_u16(pbase + 2 * PSLAB + qr * 128u + (((t6 >> 3) ^ (qr & 7u)) << 4), __bfloat16_as_ushort(lo));
                }
            }
            fence_async_smem();
            __syncwarp();
            if (elect_one()) mbar_arrive_remote(pready_leader);
            // the running sums, while the products run
            l = l * f + over_lanes<NT, true>(s, lane);
            if (__any_sync(0xffffffffu, f != 1.f)) {
#pragma unroll
                for (int q = 0; q < NT; ++q) {
                    const float fq = __shfl_sync(0xffffffffu, f, q);
#pragma unroll
                    for (int b = 0; b < NB; ++b) acc[b][q] *= fq;
                }
            }
        };
        TileWalk tw;
        tw.start(a.sq, my_first);
        int u_si = 0;          // the tile whose U comes next: its sequence, and whether it ends the run
        bool u_ends = false;
        // in step `it` the scores of tile `it`, U of the tile before, then the probabilities of tile `it`
#pragma unroll 1
        for (int it = 0; it <= n_it; ++it) {
            float s[NT];
            if (it < n_it && a.mode != MODE_V) {
                // a source's columns count for the heads that it serves only
#pragma unroll
                for (int q = 0; q < NT; ++q) s[q] = 0.f;
#pragma unroll 1
                for (int si = 0; si < list_of(0).n; ++si) {
                    const uint32_t mask = list_of(0).src[si].mask >> q0;
                    float v[NT];
                    fetch(v, 7);
#pragma unroll
                    for (int q = 0; q < NT; ++q)
                        if ((mask >> q) & 1u) s[q] += v[q];
                    if (si + 1 < list_of(0).n) TR(TR_OUT, 0x73);
                }
            } else if (it < n_it) {
                if (it == 0) grid_dependency_wait();  // the launch before holds the scores
#pragma unroll
                for (int q = 0; q < NT; ++q) s[q] = 0.f;
                const float *sp = a.score + ((int64_t)(pair * a.k_parts * 2 + (int)rank) * NQ + q0) * TILE + row;
#pragma unroll 4
                for (int p = 0; p < a.k_parts; ++p, sp += 2 * NQ * TILE) {
#pragma unroll
                    for (int q = 0; q < NT; ++q) s[q] += sp[q * TILE];
                }
            }
            if (a.mode == MODE_K) {  // one cluster's part of the sums over the hidden columns
                if (it == n_it) break;
                float *sp = a.score + ((int64_t)blockIdx.x * NQ + q0) * TILE + row;
#pragma unroll
                for (int q = 0; q < NT; ++q) sp[q * TILE] = s[q];
                continue;
            }
#pragma unroll 1
            for (int si = 0; si < (it > 0 ? list_of(1).n : 0); ++si) {
                const int n_blk = (((list_of(1).src[si].m + 63) >> 6) + 1) >> 1;
                const uint32_t mask = list_of(1).src[si].mask >> q0;
#pragma unroll 1
                for (int blk = 0; blk < n_blk; ++blk) {
                    float u[NT];
                    fetch(u, 8);
#pragma unroll
                    for (int q = 0; q < NT; ++q)
                        if (!((mask >> q) & 1u)) u[q] = 0.f;
#pragma unroll
                    for (int b = 0; b < NB; ++b)
                        if (b == blk) {
#pragma unroll
                            for (int q = 0; q < NT; ++q) acc[b][q] += u[q];
                        }
                    TR(TR_OUT, 0x83);
                }
            }
            if (u_ends) {
                const int64_t run = (int64_t)my_run + u_si;  // run and sequence only ever grow along the runs: unique
#pragma unroll 1
                for (int si = 0; si < list_of(1).n; ++si) {
                    const int m_left = list_of(1).src[si].m - row;
                    const uint32_t mask = list_of(1).src[si].mask >> q0;
                    float *u = a.upart + (run * a.hq + q0) * a.m_pad + list_of(1).src[si].c0 + row;
#pragma unroll
                    for (int q = 0; q < NT; ++q, u += a.m_pad) {
                        const int limit = (mask >> q) & 1u ? m_left : 0;
#pragma unroll
                        for (int b = 0; b < NB; ++b) st_global_below(u + 128 * b, acc[b][q], 128 * b, limit);
                    }
                }
#pragma unroll
                for (int q = 0; q < NT; ++q)
#pragma unroll
                    for (int b = 0; b < NB; ++b) acc[b][q] = 0.f;
                if (lane < NT) sh.lred[q0 + lane][quarter] = l;
                l = 0.f;
                half_sync();
                if (quarter == 0 && lane < NT) {
                    float *m_run = &sh.mrun[it & 1][q0 + lane];
                    if (q0 + lane < a.hq && part == 0) {
                        const float *r = sh.lred[q0 + lane];
                        float *ml = a.ml + (run * a.hq + q0 + lane) * 2;
                        ml[0] = *m_run;
                        ml[1] = (r[0] + r[1]) + (r[2] + r[3]);
                    }
                    *m_run = -INFINITY;
                }
                u_ends = false;
            }
            if (it < n_it) {
                probabilities(s, tw.valid(a.sq), it & 1);
                TR(TR_OUT, 0x73);
                u_si = tw.si;
                u_ends = tw.ends_run();
                tw.next(a.sq);
            }
        }
    }
    // ---- teardown: nobody leaves while the peer may still signal this CTA ----
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

// ---------------------------------------------------------------------------- front
// Encoder blocks first (where the call carries the encoder), then the query blocks: (query head, 256 hidden columns, 8 sequences),
// thread = two hidden columns and four of the sequences, all 64 rows of the head.  The query is scaled by 1/sqrt(head_dim) and by
// log2(e): the tile kernel's exponentials are powers of two.  Bound by the latency of the weight loads at few sequences, so all
// of them are in flight before the wait for the preceding kernels; everything else comes from the parameters.  Operand rows of
// sources that do not serve the head are left as they are: nobody reads their scores.
// Every block runs its code once, so instruction fetch counts like the loads: with loops unrolled only where that keeps loads in flight,
// addresses stepped instead of computed per load and the encoder's rows bounded, this kernel went from 63 to 39 KB of code and
// latent_back_kernel from 41-47 to 33-37; 12 layers of GPT-2's shape, 1 x 200 tokens an eighth less, 8 x 1024 609 -> 580 us; 22 of
// TinyLLaMA's, 32 x 2048 1213 -> 1174.
constexpr int LQ_SB = 8, LQ_COLS = 256, LF_THREADS = 256;
struct QueryArgs {
    const __nv_bfloat16 *q;
    __nv_bfloat16 *wq;
    float *qbias;
    int32_t n_seqs, hq, group, nq, m_pad, batch, two_terms;
    int32_t col_blocks;
    float scale;
};
__device__ __forceinline__ void query_block(const LatHeads &hp, const QueryArgs &a, int b) {
    __shared__ __align__(16) float qs[64][LQ_SB];
    const int qh = b % a.hq, cb = b / a.hq % a.col_blocks, si0 = b / a.hq / a.col_blocks * LQ_SB, tid = threadIdx.x;
    const int n_here = min(LQ_SB, a.n_seqs - si0), i0 = 4 * (tid >> 7);
    const int kvh = qh / a.group, s = hp.idx[0][kvh], slot = hp.slot[0][kvh];
    const LatHeads::Src &sp = hp.src[0][s];
    const int m2 = sp.m >> 1, j = cb * (LQ_COLS / 2) + (tid & 127);
    // threads past the last feature pair take the last one's weights and store nothing
    const int jj = min(j, m2 - 1);
    const uint32_t *w = reinterpret_cast<const uint32_t *>(sp.w2k) + (int64_t)slot * 64 * m2 + jj;
    uint32_t u[64];
#pragma unroll
    for (int c = 0; c < 64; ++c, w += m2) u[c] = __ldg(w);
    const float2 sab = __ldg(reinterpret_cast<const float2 *>(sp.sabs) + jj);  // the hidden vector is short of these
    grid_dependency_wait();
    launch_dependents();
    for (int i = tid; i < 64 * LQ_SB; i += LF_THREADS) {
        const int k = i >> 6, c = i & 63;
        qs[c][k] = k < n_here ? __bfloat162float(a.q[((int64_t)(si0 + k) * a.hq + qh) * 64 + c]) * a.scale : 0.f;
    }
    __syncthreads();
    float x[4] = {0.f, 0.f, 0.f, 0.f}, y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 64; ++c) {
        const float w0 = __uint_as_float(u[c] << 16), w1 = __uint_as_float(u[c] & 0xffff0000u);
        const float4 q4 = *reinterpret_cast<const float4 *>(&qs[c][i0]);
        x[0] = fmaf(w0, q4.x, x[0]);
        x[1] = fmaf(w0, q4.y, x[1]);
        x[2] = fmaf(w0, q4.z, x[2]);
        x[3] = fmaf(w0, q4.w, x[3]);
        y[0] = fmaf(w1, q4.x, y[0]);
        y[1] = fmaf(w1, q4.y, y[1]);
        y[2] = fmaf(w1, q4.z, y[2]);
        y[3] = fmaf(w1, q4.w, y[3]);
    }
    const int rows = wq_rows(a.nq);  // operand rows per (source, sequence): high terms, then low terms
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        x[i] *= sab.x;
        y[i] *= sab.y;
        hi[i] = pack_bf16(x[i], y[i]);
        lo[i] = a.two_terms ? pack_bf16(x[i] - __uint_as_float(hi[i] << 16), y[i] - __uint_as_float(hi[i] & 0xffff0000u)) : 0u;
    }
    const int64_t seq_step = (int64_t)rows * (a.m_pad >> 1), low = (int64_t)a.nq * (a.m_pad >> 1);
    uint32_t *r = reinterpret_cast<uint32_t *>(a.wq) + ((int64_t)s * a.batch + si0 + i0) * seq_step + (int64_t)qh * (a.m_pad >> 1) + j;
    if (j < m2) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i0 + i < n_here) {
                r[i * seq_step] = hi[i];
                r[i * seq_step + low] = lo[i];
            }
    }
    if (cb != 0) return;
    const int warp = tid >> 5, lane = tid & 31;
    if (warp < n_here) {
        float bias = qs[lane][warp] * sp.b2[slot * 64 + lane] + qs[lane + 32][warp] * sp.b2[slot * 64 + lane + 32];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) bias += __shfl_xor_sync(0xffffffffu, bias, d);
        if (lane == 0) a.qbias[(int64_t)(si0 + warp) * a.hq + qh] = bias;
    }
}

// n_enc = encoder blocks (0: none): nbx x nby x 2
struct EncodeGrid {
    int32_t n_enc, nbx, nby;
};
template <int NF>
__global__ void __launch_bounds__(LF_THREADS) latent_front_kernel(const __grid_constant__ LatHeads hp, const __grid_constant__ QueryArgs a,
                                                                  const __grid_constant__ LatEncode e, const __grid_constant__ SeqList seqs,
                                                                  const __grid_constant__ EncodeGrid g) {
    extern __shared__ __align__(16) float xs[];
    const int b = blockIdx.x;
    if (b < g.n_enc)
        enc::encode_fc_block<__nv_bfloat16, 1, false, NF>(e.a, seqs.id, seqs.n, e.hid, e.pitch, e.max_batch, xs, b % g.nbx, b / g.nbx % g.nby,
                                                      b / g.nbx / g.nby, g.nbx);
    else
        query_block(hp, a, b - g.n_enc);
}

// ---------------------------------------------------------------------------- back
// Encoder blocks first, then the merge: (query head, SB sequences).  The last decoder layer's 64 rows of the head (73 KB at m = 576) are read once
// per SB sequences: SB = 4 where that still fills the machine, else 1 (at 8 sequences x 12 heads, 4 sequences per block left 24
// blocks and took 57 us; SB = 1 with 288 threads 15 us, a chain of dependent loads; 8 us with threads whose registers take the
// weights before anything else is known).
constexpr int LM_PRE = 36;  // weight words a lane holds ahead: all of them up to m = 576 at 16 warps
struct MergeArgs {
    const float *upart, *ml, *qbias;
    const __nv_bfloat16 *q;
    __nv_bfloat16 *out;
    int32_t hq, group, kv_width, m_pad;
    float scale;
    int32_t with_current;
};
template <int SB, int LM_THREADS>
__device__ __forceinline__ void merge_block(const LatHeads &hp, const LatSeqs &sq, const MergeArgs &a, float *u, int b) {
    // u: [SB][m_pad], with SB = 1 then the groups' partial sums [LM_THREADS][4]
    constexpr int LM_WARPS = LM_THREADS / 32;
    __shared__ float wts[SB][LT_MAX_CTAS];
    __shared__ float fin[SB][2];  // (sum of the runs, exponent reference) per sequence
    __shared__ float osum[LM_WARPS][SB][64];
    const int qh = b % a.hq, si0 = b / a.hq * SB, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_here = min(SB, sq.n - si0);
    const int kvh = qh / a.group, slot = hp.slot[1][kvh];
    const LatHeads::Src &sp = hp.src[1][hp.idx[1][kvh]];
    const int m = sp.m, m_pad = a.m_pad;
    // lane = two channels of the head, warp = every LM_WARPS-th hidden feature
    const uint32_t *w = reinterpret_cast<const uint32_t *>(sp.w2t) + slot * 32 + lane;
    const int64_t pitch = sp.in_dim >> 1;
    uint32_t pre[SB == 1 ? LM_PRE : 1];
    if (SB == 1) {
#pragma unroll
        for (int k = 0; k < LM_PRE; ++k) {
            const int j = warp + k * LM_WARPS;
            pre[k] = j < m ? __ldg(w + j * pitch) : 0u;
        }
    }
    grid_dependency_wait();
    launch_dependents();
    auto first = [&](int i) { return (int)(sq.first[i] & 0xffffffu); };
    auto runs = [&](int si, int &k0) {  // runs of a sequence: k0 .. k0 + n - 1
        const int f0 = first(si), f1 = first(si + 1);
        k0 = f0 / sq.per;
        return f1 > f0 ? (f1 - 1) / sq.per - k0 + 1 : 0;
    };
    if (warp < n_here) {  // one warp per sequence: reference maximum over its runs, their weights, the sum
        const int si = si0 + warp;
        int k0;
        const int n_run = runs(si, k0);
        const float2 *p = reinterpret_cast<const float2 *>(a.ml) + (int64_t)(k0 + si) * a.hq + qh;
        float M = -INFINITY, S = 0.f;
#pragma unroll 1
        for (int r = lane; r < n_run; r += 32) M = fmaxf(M, p[(int64_t)r * a.hq].x);
        M = redux_max(M);
#pragma unroll 1
        for (int r = lane; r < n_run; r += 32) {
            const float2 v = p[(int64_t)r * a.hq];
            const float wr = ex2(v.x - M);
            wts[warp][r] = wr;
            S += wr * v.y;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) S += __shfl_xor_sync(0xffffffffu, S, d);
        if (lane == 0) {
            fin[warp][0] = S;
            fin[warp][1] = n_run > 0 ? M + a.qbias[(int64_t)si * a.hq + qh] : -INFINITY;
        }
    }
    __syncthreads();
    // thread = (sequence, four hidden features); with one sequence the threads that are left share its runs
    const int nf = m >> 2;
    auto add_runs = [&](int i, int f, int r0, int step) {
        int k0;
        const int n_run = runs(si0 + i, k0);
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        const float *p = a.upart + ((int64_t)(k0 + si0 + i) * a.hq + qh) * m_pad + f;
#pragma unroll 4
        for (int r = r0; r < n_run; r += step) {
            const float4 v = *reinterpret_cast<const float4 *>(p + (int64_t)r * a.hq * m_pad);
            const float wr = wts[i][r];
            acc.x = fmaf(wr, v.x, acc.x);
            acc.y = fmaf(wr, v.y, acc.y);
            acc.z = fmaf(wr, v.z, acc.z);
            acc.w = fmaf(wr, v.w, acc.w);
        }
        return acc;
    };
    auto put = [&](int i, int f, float4 acc) {
        const float4 sc = *reinterpret_cast<const float4 *>(sp.sabs + f);  // the hidden vector is short of this factor
        *reinterpret_cast<float4 *>(u + i * m_pad + f) = make_float4(acc.x * sc.x, acc.y * sc.y, acc.z * sc.z, acc.w * sc.w);
    };
    if (SB == 1) {
        float4 *part = reinterpret_cast<float4 *>(u + m_pad);
        const int n_grp = max(1, LM_THREADS / nf), grp = tid / nf;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (grp < n_grp) acc = add_runs(0, 4 * (tid % nf), grp, n_grp);
        part[tid] = acc;
        __syncthreads();
        if (tid < nf) {
#pragma unroll 2
            for (int g = 1; g < n_grp; ++g) {
                const float4 v = part[tid + g * nf];
                acc.x += v.x;
                acc.y += v.y;
                acc.z += v.z;
                acc.w += v.w;
            }
            put(0, 4 * tid, acc);
        }
    } else {
#pragma unroll 1
        for (int t = tid; t < SB * nf; t += LM_THREADS) {
            const int i = t / nf, f = 4 * (t % nf);
            put(i, f, i < n_here ? add_runs(i, f, 0, 1) : make_float4(0.f, 0.f, 0.f, 0.f));
        }
    }
    __syncthreads();
    {
        float x[SB], y[SB];
#pragma unroll
        for (int i = 0; i < SB; ++i) x[i] = y[i] = 0.f;
        auto add = [&](uint32_t v, int j) {
            const float w0 = __uint_as_float(v << 16), w1 = __uint_as_float(v & 0xffff0000u);
#pragma unroll
            for (int i = 0; i < SB; ++i) {
                const float ui = u[i * m_pad + j];
                x[i] = fmaf(w0, ui, x[i]);
                y[i] = fmaf(w1, ui, y[i]);
            }
        };
        if (SB == 1) {
#pragma unroll
            for (int k = 0; k < LM_PRE; ++k) {
                const int j = warp + k * LM_WARPS;
                if (j < m) add(pre[k], j);
            }
        }
#pragma unroll(SB == 1 ? 2 : 16)
        for (int j = warp + (SB == 1 ? LM_PRE * LM_WARPS : 0); j < m; j += LM_WARPS) add(__ldg(w + j * pitch), j);
#pragma unroll
        for (int i = 0; i < SB; ++i) *reinterpret_cast<float2 *>(&osum[warp][i][2 * lane]) = make_float2(x[i], y[i]);
    }
    __syncthreads();
    if (warp >= n_here) return;
    // one warp per sequence: add up, the head's bias, the exact current token
    const int si = si0 + warp;
    float o[2] = {0.f, 0.f};
#pragma unroll 4
    for (int k = 0; k < LM_WARPS; ++k) {
        o[0] += osum[k][warp][lane];
        o[1] += osum[k][warp][lane + 32];
    }
    float S = fin[warp][0];
    const float M = fin[warp][1];
    o[0] += sp.b2[slot * 64 + lane] * S;
    o[1] += sp.b2[slot * 64 + lane + 32] * S;
    if (a.with_current) {
        const int64_t seq = sq.id[si];
        const __nv_bfloat16 *kc = reinterpret_cast<const __nv_bfloat16 *>(hp.cur[0][kvh]) + seq * a.kv_width;
        const __nv_bfloat16 *vc = reinterpret_cast<const __nv_bfloat16 *>(hp.cur[1][kvh]) + seq * a.kv_width;
        const __nv_bfloat16 *qg = a.q + ((int64_t)si * a.hq + qh) * 64;
        float sc = __bfloat162float(qg[lane]) * __bfloat162float(kc[lane]) + __bfloat162float(qg[lane + 32]) * __bfloat162float(kc[lane + 32]);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) sc += __shfl_xor_sync(0xffffffffu, sc, d);
        sc *= a.scale;
        const float Mn = fmaxf(M, sc);
        const float c0 = M == -INFINITY ? 0.f : ex2(M - Mn), c1 = ex2(sc - Mn);
        S = S * c0 + c1;
        o[0] = o[0] * c0 + __bfloat162float(vc[lane]) * c1;
        o[1] = o[1] * c0 + __bfloat162float(vc[lane + 32]) * c1;
    }
    __nv_bfloat16 *out = a.out + ((int64_t)si * a.hq + qh) * 64;
    out[lane] = __float2bfloat16_rn(S > 0.f ? o[0] / S : 0.f);
    out[lane + 32] = __float2bfloat16_rn(S > 0.f ? o[1] / S : 0.f);
}

template <int SB, int THREADS, int NF>
__global__ void __launch_bounds__(THREADS) latent_back_kernel(const __grid_constant__ LatHeads hp, const __grid_constant__ LatSeqs sq,
                                                              const __grid_constant__ MergeArgs a, const __grid_constant__ LatEncode e,
                                                              const __grid_constant__ SeqList all, const __grid_constant__ EncodeGrid g) {
    extern __shared__ __align__(16) float sm[];
    const int b = blockIdx.x;
    if (b < g.n_enc)
        enc::encode_fc_block<__nv_bfloat16, 2, false, NF>(e.a, all.id, all.n, e.hid, e.pitch, e.max_batch, sm, b % g.nbx, b / g.nbx % g.nby,
                                                      b / g.nbx / g.nby, g.nbx);
    else
        merge_block<SB, THREADS>(hp, sq, a, sm, b - g.n_enc);
}

// int8 rows to bf16: grid = (tiles, sources of K and V, 2 pieces of a tile's rows).  Bound by memory: a byte in, two out.
__global__ void __launch_bounds__(256) latent_widen_kernel(const __grid_constant__ LatCodes c, const __grid_constant__ LatSeqs sq,
                                                           const int32_t *block_table, int max_pages_per_seq, int page_tokens,
                                                           __nv_bfloat16 *wide, float2 *rowp, int wide_rows, int pitch) {
    __shared__ int64_t rows[64];
    __shared__ int z0[64];
    const int side = (int)blockIdx.y >= c.n_src[0], s = blockIdx.y - (side ? c.n_src[0] : 0), t = blockIdx.x, tid = threadIdx.x;
    TileWalk tw;
    tw.start(sq, t);
    tw.left = 1;
    const int valid = min(64, (tw.chunk + 1 < tw.n ? TILE : (int)(sq.first[tw.si] >> 24) + 1) - 64 * (int)blockIdx.z);
    if (valid <= 0) return;
    const int64_t out0 = (int64_t)(side * LT_MAX_SRC + s) * wide_rows + t * TILE + 64 * blockIdx.z;
    grid_dependency_wait();
    launch_dependents();
    if (tid < valid) {
        const int tok = tw.chunk * TILE + 64 * blockIdx.z + tid;
        const int page = block_table[(int64_t)sq.id[tw.si] * max_pages_per_seq + tok / page_tokens];
        const int64_t r = (int64_t)page * page_tokens + tok % page_tokens;
        const float scale = c.qparam[side][s][2 * r], zp = c.qparam[side][s][2 * r + 1];
        // a row of equal values has any zero-point: its whole part within reach goes into the codes, the rest is left over
        const float z = rintf(fminf(fmaxf(zp, -128.f), 128.f));
        rows[tid] = r;
        z0[tid] = (int)z;
        rowp[out0 + tid] = make_float2(1.f / scale, zp - z);
    }
    __syncthreads();
    const int d = c.d[side][s], nv = d >> 4;
    for (int i = tid; i < valid * nv; i += 256) {
        const int r = i / nv, k = 16 * (i % nv);
        const int4 v = *reinterpret_cast<const int4 *>(c.codes[side][s] + rows[r] * d + k);
        const int words[4] = {v.x, v.y, v.z, v.w};
        uint32_t o[8];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            const int b0 = (int8_t)words[w], b1 = (int8_t)(words[w] >> 8), b2 = (int8_t)(words[w] >> 16), b3 = words[w] >> 24;
            o[2 * w] = pack_bf16((float)(b0 - z0[r]), (float)(b1 - z0[r]));
            o[2 * w + 1] = pack_bf16((float)(b2 - z0[r]), (float)(b3 - z0[r]));
        }
        uint4 *dst = reinterpret_cast<uint4 *>(wide + (out0 + r) * pitch + k);
        dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
        dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
}

using Kernel = void (*)(const Params);
// Builds, the narrowest first of each kind, jobs of 192 columns before those of 128.
struct Build {
    int nq, nb, cn;
    bool quant, p2;
    Kernel kernel;
};
template <int NQ, int NB, int CN, bool Q8, bool P2>
constexpr Build build() {
    return {NQ, NB, CN, Q8, P2, decode_latent_kernel<NQ, NB, CN, Q8, P2>};
}
const Build builds[] = {build<12, 2, 192, false, false>(), build<12, 5, 192, false, false>(), build<16, 5, 192, false, false>(),
                        build<16, 8, 192, false, false>(), build<32, 2, 192, false, false>(), build<32, 3, 192, false, false>(),
                        build<32, 3, 192, false, true>(),  build<12, 5, 128, false, false>(), build<16, 8, 128, false, false>(),
                        build<12, 2, 128, true, false>(),  build<12, 5, 128, true, false>(),  build<16, 5, 128, true, false>(),
                        build<16, 8, 128, true, false>(),  build<32, 2, 128, true, true>(),   build<32, 3, 128, true, true>()};
constexpr int N_BUILDS = sizeof(builds) / sizeof(builds[0]);

int smem_bytes(const Build &b, int nz, int nh, int nw, int nqs) {
    const int scratch = b.nq == 12 ? sizeof(Scratch<12>) : b.nq == 16 ? sizeof(Scratch<16>) : sizeof(Scratch<32>);
    return (nz + nh) * SLAB + nw * wstage(b.cn) + nqs * wq_slab(b.nq) + (b.p2 ? 4 : 2) * op_rows(b.nq) * 128 +
           8 * (2 * (nz + nw + nqs) + nh + READY_BARS + 9) + scratch;
}
constexpr int SMEM_MAX = 227 * 1024;

// one padding for all layers of a context, whose W4^T q rows share their place (12 heads: up to 640 hidden features in registers)
int padded_heads(int hq, int max_m) { return hq <= 12 && max_m <= 640 ? 12 : hq <= 16 ? 16 : 32; }

void fill_seqs(LatSeqs &q, const SeqList &seqs, const int32_t *lens, int n_sms) {
    uint32_t t = 0;
    q.n = seqs.n;
    for (int i = 0; i < seqs.n; ++i) {
        q.id[i] = seqs.id[i];
        q.first[i] = t | (uint32_t)(lens[i] > 0 ? (lens[i] - 1) % TILE : 0) << 24;
        t += (uint32_t)((lens[i] + TILE - 1) / TILE);
    }
    q.first[seqs.n] = t;
    q.n_tiles = (int32_t)t;
    const int ctas = std::min(n_sms, LT_MAX_CTAS) & ~1;
    q.per = std::max(1, ((int)t + ctas - 1) / ctas);
}

constexpr float LOG2E = 1.4426950408889634f;

}  // namespace

static int lat_wide_tiles(int batch, int max_len) {
    const int per_seq = (max_len + TILE - 1) / TILE;
    return (int)std::min<int64_t>((int64_t)batch * per_seq, std::max(LT_WIDE_TILES, per_seq));
}

static bool shape_ok(const kvcar_config &cfg) {
    return cfg.storage == KVCAR_BF16 && cfg.head_dim == 64 && cfg.n_q_heads <= LT_MAX_Q && cfg.page_tokens % 64 == 0;
}

size_t lat_ws_bytes(const kvcar_config &cfg, int max_sources, int max_m, int max_d, int batch, int max_len) {
    if (!shape_ok(cfg) || max_sources <= 0 || max_m <= 0) return 0;
    const size_t nq = padded_heads(cfg.n_q_heads, max_m), m_pad = ((size_t)max_m + 63) / 64 * 64;
    const size_t wq = (size_t)std::min(max_sources, LT_MAX_SRC) * batch * wq_rows((int)nq) * m_pad * 2;
    const size_t bias = ((size_t)batch * cfg.n_q_heads * 4 + 255) / 256 * 256;
    const size_t runs = (size_t)LT_MAX_CTAS + batch;
    size_t n = wq + bias + runs * cfg.n_q_heads * (m_pad + 2) * sizeof(float) + (size_t)LT_MAX_CTAS * nq * TILE * sizeof(float);
    if (cfg.latent_quant)  // the widened rows start at a multiple of 256 bytes
        n = (n + 255) / 256 * 256 + (size_t)(LT_MAX_SRC + std::min(max_sources, LT_MAX_SRC)) * lat_wide_tiles(batch, max_len) * TILE * (2 * (size_t)max_d + sizeof(float2));
    return n;
}

// Staging places of a layer under a build.  A side's latents stay for all its chunks (nz >= their slabs).  One-chunk layers get
// places for the other side's latents and six hidden slabs, because their jobs are shorter than the way from S to P; the others four
// hidden slabs: a chunk's three and the one its predecessor may leave unpaired, or two chunks' two, or a chunk's two terms of two.
static bool pick_places(const Build &b, const LatShape &sh, LatLayerCfg &lc) {
    const int ks = (sh.d + 63) / 64, chunks = (sh.m + b.cn - 1) / b.cn;
    int nh = chunks == 1 ? 6 : 4, nz = chunks == 1 ? std::max(4, 2 * ks) : ks, nw = 4, nqs = 4;
    auto fits = [&]() { return smem_bytes(b, nz, nh, nw, nqs) <= SMEM_MAX; };
    while (nw > 3 && !fits()) --nw;
    while (nqs > 2 && !fits()) --nqs;
    while (nz > ks && !fits()) --nz;
    while (nw > 2 && !fits()) --nw;
    if (!fits() && b.cn == 128) nh = 2;  // one chunk, or one term of it, at a time
    if (!fits()) return false;
    while (nqs < 12 && (++nqs, fits())) {}
    if (!fits()) --nqs;
    lc.nz = (uint8_t)nz;
    lc.nh = (uint8_t)nh;
    lc.nw = (uint8_t)nw;
    lc.nqs = (uint8_t)nqs;
    lc.smem = std::max(smem_bytes(b, nz, nh, nw, nqs), 120 * 1024);  // one CTA per SM: each takes all of tensor memory
    return true;
}

// the build and the staging places of a layer, false where none fits
static bool pick_build(const kvcar_config &cfg, int max_m, const LatShape &sh, LatLayerCfg &lc) {
    if (!sh.widths_ok || sh.n_src[0] < 1 || sh.n_src[0] > LT_MAX_SRC || sh.n_src[1] < 1 || sh.n_src[1] > LT_MAX_SRC) return false;
    const int nq = padded_heads(cfg.n_q_heads, max_m);
    const bool quant = cfg.latent_quant != 0, p2 = nq > 16 && (quant || cfg.n_q_heads / cfg.n_kv_heads <= 2);
    for (int v = 0; v < N_BUILDS; ++v) {
        const Build &b = builds[v];
        if (b.nq != nq || b.quant != quant || b.p2 != p2 || b.nb * 128 < sh.m || !pick_places(b, sh, lc)) continue;
        lc.variant = (uint8_t)v;
        lc.max_m = sh.m;
        lc.max_mk = sh.mk;
        return true;
    }
    return false;
}

bool lat_covers(const kvcar_config &cfg, int max_m, const LatShape &sh) {
    LatLayerCfg lc;
    return shape_ok(cfg) && pick_build(cfg, max_m, sh, lc);
}

void lat_setup(LatState &st, const kvcar_config &cfg, const std::vector<LayerPlan> &plans, size_t pool_rows,
               int max_sources, int max_m, int max_d, int batch, int max_len, char *ws_area) {
    st.available = false;
    const int nl = cfg.n_layers;
    st.layer.assign(nl, LatLayer{});
    st.heads.assign(nl, LatHeads{});
    st.cfg.assign(nl, LatLayerCfg{});
    if (lat_ws_bytes(cfg, max_sources, max_m, max_d, batch, max_len) == 0) return;
    EncodeTiledFn fn = tensor_map_encoder();
    if (!fn) return;
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int group = cfg.n_q_heads / cfg.n_kv_heads;
    st.n_sms = sms;
    for (auto k : {latent_back_kernel<4, 256, 1>, latent_back_kernel<4, 256, 2>, latent_back_kernel<1, 512, 1>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, LT_ENC_SMEM) != cudaSuccess) return;
    for (auto k : {latent_front_kernel<1>, latent_front_kernel<2>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, LT_ENC_SMEM) != cudaSuccess) return;
    st.nq = padded_heads(cfg.n_q_heads, max_m);
    st.group = group;
    st.m_pad = (max_m + 63) / 64 * 64;
    st.batch = batch;
    const size_t n_src = std::min(max_sources, LT_MAX_SRC), n_rows = n_src * batch * wq_rows(st.nq);
    if (!encode_bf16_map(fn, &st.tm_wq, ws_area, n_rows, st.m_pad, st.m_pad, op_rows(st.nq))) return;
    char *p = ws_area;
    st.wq = p;
    p += n_rows * st.m_pad * 2;
    st.qbias = reinterpret_cast<float *>(p);
    p += ((size_t)batch * cfg.n_q_heads * 4 + 255) / 256 * 256;
    st.upart = reinterpret_cast<float *>(p);
    p += (size_t)(LT_MAX_CTAS + batch) * cfg.n_q_heads * st.m_pad * sizeof(float);
    st.ml = reinterpret_cast<float *>(p);
    p += (size_t)(LT_MAX_CTAS + batch) * cfg.n_q_heads * 2 * sizeof(float);
    st.score = reinterpret_cast<float *>(p);
    p += (size_t)LT_MAX_CTAS * st.nq * TILE * sizeof(float);
    p = ws_area + ((size_t)(p - ws_area) + 255) / 256 * 256;
    st.quant = cfg.latent_quant != 0;
    st.wide_tiles = lat_wide_tiles(batch, max_len);
    const size_t wide_rows = (size_t)st.wide_tiles * TILE, regions = LT_MAX_SRC + n_src;
    st.wide = p;
    st.rowp = reinterpret_cast<float2 *>(p + regions * wide_rows * 2 * max_d);
    st.max_d = max_d;
    st.codes.assign(st.quant ? nl : 0, LatCodes{});
    for (int l = 0; l < nl; ++l) {
        LatLayer &ly = st.layer[l];
        LatHeads &hp = st.heads[l];
        LatLayerCfg &lc = st.cfg[l];
        bool ok = true;
        LatShape sh;
        for (int w = 0; w < 2; ++w)
            for (int s = 0; s < plans[l].w[w].n_src; ++s) {
                const SourcePlan &sp = plans[l].w[w].src[s];
                ok = ok && sp.compressed && (sp.qparam != nullptr) == st.quant && sp.width == sp.d;
                sh.add(w, sp.d, sp.m);
            }
        if (!ok || !pick_build(cfg, max_m, sh, lc)) continue;
        for (int w = 0; w < 2 && ok; ++w) {
            const WhichPlan &wp = plans[l].w[w];
            ly.list[w].n = hp.n_src[w] = wp.n_src;
            for (int s = 0; s < wp.n_src && ok; ++s) {
                const SourcePlan &sp = wp.src[s];
                LatSrc &d = ly.list[w].src[s];
                d.shift = sp.shift;
                d.rowsum = sp.rowsum;
                const size_t region = (size_t)(w * LT_MAX_SRC + s) * wide_rows;
                d.rowp = st.rowp + region;
                d.c0 = 0;
                d.map = s;
                d.d = sp.d;
                d.m = sp.m;
                d.slope = sp.slope > 1.f ? 1.f / sp.slope : sp.slope;  // see put_signed_fc1
                d.mask = 0;
                hp.src[w][s] = {sp.w2k, sp.w2t, sp.b2, sp.sabs, sp.m, sp.in_dim};
                for (int i = 0; i < sp.n_need; ++i) {
                    const int h = sp.kv_head[i];
                    for (int g = 0; g < group; ++g) d.mask |= 1u << (h * group + g);
                    hp.idx[w][h] = (uint8_t)s;
                    hp.slot[w][h] = (uint8_t)sp.slot[i];
                    hp.cur[w][h] = reinterpret_cast<const __nv_bfloat16 *>(plans[l].cur[w][h]) + plans[l].cur_head[w][h] * 64;
                }
                if (st.quant) {
                    LatCodes &c = st.codes[l];
                    c.codes[w][s] = reinterpret_cast<const int8_t *>(sp.pool);
                    c.qparam[w][s] = sp.qparam;
                    c.d[w][s] = sp.d;
                    c.n_src[w] = wp.n_src;
                }
                ok = (st.quant ? encode_bf16_map(fn, &ly.pool[w][s], reinterpret_cast<__nv_bfloat16 *>(st.wide) + region * max_d, wide_rows, sp.d, max_d)
                               : encode_bf16_map(fn, &ly.pool[w][s], sp.pool, pool_rows, sp.width, sp.width)) &&
                     encode_bf16_map(fn, &ly.w1[w][s], sp.w1n, sp.m, sp.d, sp.d, builds[lc.variant].cn / 2);
            }
        }
        if (!ok) continue;
        if (cudaFuncSetAttribute(builds[lc.variant].kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_MAX) != cudaSuccess) {
            cudaGetLastError();
            continue;
        }
        lc.ok = 1;
        st.available = true;
    }
}

bool lat_layer_supported(const LatState &st, int layer) { return st.available && st.cfg[layer].ok; }

namespace {

// A side's hidden columns in `n` parts of whole chunks of `cn` columns, of about the same number of products each; a part holds one
// range of columns per source at most (the ranges of a source follow one another).  False where a part would be empty.
bool split_side(const LatList &all, int cn, int n, LatList *out) {
    int total = 0, done = 0;
    for (int s = 0; s < all.n; ++s) total += (all.src[s].d + 63) / 64 * ((all.src[s].m + 63) / 64);
    for (int p = 0; p < n; ++p) out[p].n = 0;
    for (int s = 0; s < all.n; ++s)
        for (int c0 = 0; c0 < all.src[s].m; c0 += cn) {
            const int w = std::min(cn, all.src[s].m - c0), cost = (all.src[s].d + 63) / 64 * ((w + 63) / 64);
            LatList &l = out[std::min(n - 1, (int)((int64_t)(2 * done + cost) * n / (2 * total)))];  // by the chunk's middle
            done += cost;
            if (l.n > 0 && l.src[l.n - 1].map == all.src[s].map) {
                l.src[l.n - 1].m += w;
                continue;
            }
            LatSrc &u = l.src[l.n++];
            u = all.src[s];
            u.shift += c0;
            u.rowsum += c0;
            u.c0 = c0;
            u.m = w;
        }
    for (int p = 0; p < n; ++p)
        if (out[p].n == 0) return false;
    return true;
}
int count_chunks(const LatList &l, int cn) {
    int n = 0;
    for (int s = 0; s < l.n; ++s) n += (l.src[s].m + cn - 1) / cn;
    return n;
}

}  // namespace

// `seqs` of a call; `all`: those whose rows the carried encoder takes
static cudaError_t launch_group(LatState &st, const DecodeArgs &a, const SeqList &seqs, const SeqList &all, const int32_t *lens, int layer,
                                const LatEncode *enc_in, cudaStream_t stream, int *n_launches) {
    const LatLayerCfg &lc = st.cfg[layer];
    const LatLayer &ly = st.layer[layer];
    const Build &b = builds[lc.variant];
    Params p;
    fill_seqs(p.sq, seqs, lens, st.n_sms);
    const bool two_k = !(a.flags & KVCAR_ABSORBED), two_v = !((a.flags & KVCAR_ABSORBED) && (a.flags & KVCAR_ABSORBED_V)) && (b.nq <= 16 || b.p2);
    LatEncode e{};
    if (enc_in) e = *enc_in;
    EncodeGrid g{0, 1, 1};
    if (st.quant) {
        const LatCodes &c = st.codes[layer];
        cudaError_t err = launch_pdl(latent_widen_kernel, dim3(p.sq.n_tiles, c.n_src[0] + c.n_src[1], 2), 256, 0, stream, c, p.sq, a.block_table,
                                     a.max_pages_per_seq, a.page_tokens, reinterpret_cast<__nv_bfloat16 *>(st.wide), st.rowp,
                                     st.wide_tiles * TILE, st.max_d);
        if (err != cudaSuccess) return err;
        ++*n_launches;
    }
    // ---- front
    QueryArgs qa;
    qa.q = reinterpret_cast<const __nv_bfloat16 *>(a.q);
    qa.wq = reinterpret_cast<__nv_bfloat16 *>(st.wq);
    qa.qbias = st.qbias;
    qa.n_seqs = seqs.n;
    qa.hq = a.hq;
    qa.group = st.group;
    qa.nq = st.nq;
    qa.m_pad = st.m_pad;
    qa.batch = st.batch;
    qa.two_terms = two_k;
    qa.col_blocks = (lc.max_mk + LQ_COLS - 1) / LQ_COLS;
    qa.scale = a.scale * LOG2E;
    // Features per warp of the encoder: one spreads a few rows' weights over the most warps, two read the rows half as often from
    // shared memory.  12-layer step of the GPT-2 shape over 256 cached tokens: 64 sequences 954 us with one, 817 with two; 256
    // sequences 3093, 2686 (four: 902, 3069, the registers leave one block per SM).
    const int nf = all.n >= 64 ? 2 : 1;
    size_t smem = 0;
    if (enc_in) {
        g.nbx = (std::max(e.max_m, 1) + LF_THREADS / 32 * nf - 1) / (LF_THREADS / 32 * nf);
        g.nby = (all.n + enc::RB - 1) / enc::RB;
        g.n_enc = g.nbx * g.nby * 2;
        smem = (size_t)enc::RB * e.max_in * sizeof(float);
    }
    cudaError_t err = launch_pdl(nf == 2 ? latent_front_kernel<2> : latent_front_kernel<1>, dim3(g.n_enc + a.hq * qa.col_blocks * ((seqs.n + LQ_SB - 1) / LQ_SB)), LF_THREADS,
                                 smem, stream, st.heads[layer], qa, e, all, g);
    if (err != cudaSuccess) return err;
    // ---- tiles
    for (int w = 0; w < 2; ++w)
        for (int s = 0; s < ly.list[w].n; ++s) {
            p.pool[w][s] = ly.pool[w][s];
            p.w1[w][s] = ly.w1[w][s];
        }
    p.tm_wq = st.tm_wq;
    p.block_table = a.block_table;
    p.status = a.status;
    p.upart = st.upart;
    p.ml = st.ml;
    p.score = st.score;
    p.max_pages_per_seq = a.max_pages_per_seq;
    p.page_tokens = a.page_tokens;
    p.hq = a.hq;
    p.m_pad = st.m_pad;
    p.wq_batch = st.batch;
    p.nz = lc.nz;
    p.nh = lc.nh;
    p.nw = lc.nw;
    p.nqs = lc.nqs;
    p.two_terms_k = two_k;
    p.two_terms_v = two_v;
    const int pairs = (((p.sq.n_tiles + p.sq.per - 1) / p.sq.per) + 1) / 2, slots = st.n_sms / 2;
    // Small grids.  Where two clusters per pair of tiles fit on the machine, K and V are two launches and a side's hidden columns
    // are spread over as many clusters as there is room for.  The V launch starts beside the K launch (all of whose blocks run by
    // then), does its hidden layer meanwhile and waits for the K launch only before it sums the parts of the scores.  12-layer step
    // of the GPT-2 shape at 1 / 8 x 1024 tokens: 371 / 649 us, 625 / 712 us with one cluster per pair.
    int kp = std::min({(slots / pairs + 1) / 2, count_chunks(ly.list[0], b.cn), LT_MAX_PARTS});
    int vp = std::min({slots / pairs - kp, count_chunks(ly.list[1], b.cn), LT_MAX_PARTS});
    *n_launches += 3;
    if (p.sq.per == 1 && kp >= 1 && vp >= 1) {
        p.mode = MODE_K;
        while (!split_side(ly.list[0], b.cn, kp, p.list)) --kp;
        p.n_parts = p.k_parts = kp;
        err = launch_pdl(b.kernel, dim3(2 * pairs * kp), n_threads(b.cn), lc.smem, stream, p);
        if (err != cudaSuccess) return err;
        p.mode = MODE_V;
        while (!split_side(ly.list[1], b.cn, vp, p.list)) --vp;
        p.n_parts = vp;
        err = launch_pdl(b.kernel, dim3(2 * pairs * vp), n_threads(b.cn), lc.smem, stream, p);
        ++*n_launches;
    } else {
        p.mode = MODE_BOTH;
        p.n_parts = p.k_parts = 1;
        p.list[0] = ly.list[0];
        p.list[1] = ly.list[1];
        err = launch_pdl(b.kernel, dim3(2 * pairs), n_threads(b.cn), lc.smem, stream, p);
    }
    if (err != cudaSuccess) return err;
    // ---- back
    MergeArgs m;
    m.upart = st.upart;
    m.ml = st.ml;
    m.qbias = st.qbias;
    m.q = qa.q;
    m.out = reinterpret_cast<__nv_bfloat16 *>(a.out);
    m.hq = a.hq;
    m.group = st.group;
    m.kv_width = a.hkv * 64;
    m.m_pad = st.m_pad;
    m.scale = qa.scale;
    m.with_current = (a.flags & KVCAR_INCLUDE_CURRENT_EXACT) != 0;
    const bool wide = a.hq * seqs.n > st.n_sms;
    const int threads = wide ? 256 : 512, sb = wide ? 4 : 1;
    smem = (size_t)sb * st.m_pad * 4 + (wide ? 0 : threads * 16);
    if (enc_in) {
        const int per = threads / 32 * (wide ? nf : 1);
        g.nbx = (std::max(e.max_d, 1) + per - 1) / per;
        g.n_enc = g.nbx * g.nby * 2;
        smem = std::max(smem, (size_t)enc::RB * e.pitch * sizeof(float));
    }
    const dim3 grid(g.n_enc + a.hq * ((seqs.n + sb - 1) / sb));
    return wide ? launch_pdl(nf == 2 ? latent_back_kernel<4, 256, 2> : latent_back_kernel<4, 256, 1>, grid, threads, smem, stream, st.heads[layer], p.sq, m, e, all, g)
                : launch_pdl(latent_back_kernel<1, 512, 1>, grid, threads, smem, stream, st.heads[layer], p.sq, m, e, all, g);
}

cudaError_t lat_launch(LatState &st, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens, int layer, const LatEncode *enc,
                       cudaStream_t stream, int *n_launches) {
    *n_launches = 0;
    if (!st.quant) return launch_group(st, a, seqs, seqs, lens, layer, enc, stream, n_launches);
    // int8 rows: as many sequences at a time as the widened rows have room for; the encoder goes with the first
    for (int i0 = 0; i0 < seqs.n;) {
        SeqList g;
        g.n = 0;
        int tiles = 0, i = i0;
        for (; i < seqs.n; ++i) {
            const int n = (lens[i] + TILE - 1) / TILE;
            if (g.n > 0 && tiles > 0 && tiles + n > st.wide_tiles) break;
            g.id[g.n++] = seqs.id[i];
            tiles += n;
        }
        DecodeArgs ga = a;
        ga.q = reinterpret_cast<const __nv_bfloat16 *>(a.q) + (int64_t)i0 * a.hq * 64;
        ga.out = reinterpret_cast<__nv_bfloat16 *>(a.out) + (int64_t)i0 * a.hq * 64;
        cudaError_t err = launch_group(st, ga, g, seqs, lens + i0, layer, i0 == 0 ? enc : nullptr, stream, n_launches);
        if (err != cudaSuccess) return err;
        i0 = i;
    }
    return cudaSuccess;
}

}  // namespace kvcar

#ifdef KVCAR_TRACE
// out: [2 CTAs][6 roles][4096] records; n: records per CTA and role
extern "C" int kvcar_debug_trace_select(int cluster) { return (int)cudaMemcpyToSymbol(kvcar::g_trace_cluster, &cluster, sizeof(int)); }
extern "C" int kvcar_debug_trace_dump(unsigned long long *out, int *n) {
    cudaError_t e = cudaMemcpyFromSymbol(out, kvcar::g_trace, sizeof(kvcar::g_trace));
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(n, kvcar::g_trace_n, sizeof(kvcar::g_trace_n));
    return (int)e;
}
#endif
