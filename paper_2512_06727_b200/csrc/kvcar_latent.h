// Interface between the host runtime and the latent-attention kernels (kvcar_latent.cu).
#pragma once
#include <vector>

#include "kvcar_internal.h"

namespace kvcar {

constexpr int LT_MAX_SRC = 6;     // distinct source layers per K or V of a layer
constexpr int LT_MAX_Q = 32;      // query heads
constexpr int LT_ENC_SMEM = 160 * 1024;  // what the encoder's input rows may take in the launches that carry it
constexpr int LT_MAX_CTAS = 160;  // blocks of a launch at most (one per SM)

// Place of hidden feature f's shift in the padded array: groups of 32 features, in each the order in which the four lanes of a
// fragment row hold them (features 8 j + 2 c + e of a group at 8 c + 2 j + e).
inline int shift_place(int f) { return (f & ~31) + ((f & 7) >> 1) * 8 + ((f & 31) >> 3) * 2 + (f & 1); }

// Hidden columns c0 .. c0 + m - 1 of one source layer of K or V as the tile kernel sees them (kernel parameter).
struct LatSrc {
    const float *rowsum;  // int8 rows: sums of the rows of the signed first layer, from c0, in the same order
    const float2 *rowp;   // int8 rows: (1/scale, what is left of the zero-point) per widened row
    const float *shift;  // fused bias + BatchNorm shift over the size of its scale, from c0, in fragment order (see shift_place)
    int32_t d, m, c0;
    int32_t map;    // which of the layer's tensor maps
    float slope;
    uint32_t mask;  // query heads whose K (or V) head is served from this source
};
constexpr int LT_WIDE_TILES = 296;  // int8 rows: tiles widened at a time (more if one sequence needs more)
constexpr int LT_MAX_PARTS = 8;  // clusters that share the K (or the V) side of a pair of tiles
struct LatList {
    int32_t n;
    LatSrc src[LT_MAX_SRC];
};

// The listed sequences of a call: device ids, and the first tile of each (low 24 bits) with the valid tokens of its
// last tile minus one in the high 8; first[n] = number of tiles.
struct LatSeqs {
    int32_t n, n_tiles, per, pad_;  // per: consecutive tiles of one block
    int32_t id[KVCAR_MAX_BATCH];
    uint32_t first[KVCAR_MAX_BATCH + 1];
};

// What a layer's launches need; built at bind time, kept on the host and passed to the kernels by value (tensor maps in
// kernel parameters need no acquire, and nothing is found through chains of loads).
struct LatLayer {
    CUtensorMap pool[2][LT_MAX_SRC], w1[2][LT_MAX_SRC];
    LatList list[2];  // K, V: every source whole
};
// The last decoder layer of each source, which source and column slot serves a KV head, the exact current-token rows.
struct LatHeads {
    struct Src {
        const void *w2k, *w2t;  // [in_dim][m] and [m][in_dim], bf16
        const float *b2, *sabs;
        int32_t m, in_dim;
    } src[2][LT_MAX_SRC];
    int32_t n_src[2];
    const void *cur[2][LT_MAX_Q];  // by KV head: its 64 columns of the current-token row of sequence 0
    uint8_t idx[2][LT_MAX_Q], slot[2][LT_MAX_Q];
};
// int8 rows: where a source's codes and its rows' (scale, zero-point) lie, the column sums of its signed first layer
struct LatCodes {
    const int8_t *codes[2][LT_MAX_SRC];
    const float *qparam[2][LT_MAX_SRC];
    int32_t d[2][LT_MAX_SRC];
    int32_t n_src[2];
};

// What decides whether the kernels take a layer: the sources of its K and V heads (all over latent rows).
struct LatShape {
    int n_src[2] = {0, 0}, d = 0, m = 0, mk = 0;  // widest latent, widest hidden layer, widest hidden layer of the K sources
    bool widths_ok = true;
    void add(int which, int latent, int hidden) {
        ++n_src[which];
        d = latent > d ? latent : d;
        m = hidden > m ? hidden : m;
        if (which == 0) mk = hidden > mk ? hidden : mk;
        widths_ok = widths_ok && latent % 16 == 0 && hidden % 16 == 0;
    }
};

struct LatLayerCfg {
    uint8_t ok = 0;
    uint8_t variant = 0;                              // kernel instantiation
    uint8_t nz = 0, nh = 0, nw = 0, nqs = 0;          // staging places: latent, hidden, weight, query slabs
    int32_t smem = 0;
    int32_t max_mk = 0, max_m = 0;  // widest hidden layer of the K sources, of all
};

struct LatState {
    bool available = false;
    std::vector<LatLayer> layer;
    std::vector<LatHeads> heads;
    std::vector<LatCodes> codes;  // int8 rows only
    bool quant = false;
    int wide_tiles = 0, max_d = 0;
    void *wide = nullptr;         // int8 rows: [K, V][source][wide_tiles * 128][max_d] bf16
    float2 *rowp = nullptr;       // [K, V][source][wide_tiles * 128]
    std::vector<LatLayerCfg> cfg;
    int n_sms = 148;
    int nq = 12;      // query heads padded
    int group = 1;    // query heads per KV head
    int m_pad = 0;    // row pitch of the vectors below
    int batch = 0;    // sequences per call at most
    void *wq = nullptr;      // [source][batch][operand rows][m_pad] bf16: W4_h^T q, high parts then low parts
    float *qbias = nullptr;  // [batch][hq]: q . b4_h, in the exponent's base-2 units
    float *upart = nullptr;  // [block + sequence][hq][m_pad]: sum over a run of tiles of p * hidden vector
    float *ml = nullptr;     // [block + sequence][hq][2]: reference maximum and sum of the run
    float *score = nullptr;  // [block][heads padded][128]: parts of the scores (small grids)
    CUtensorMap tm_wq;
};

// bytes of the operands and partial results inside the workspace (0: the shape does not take this path)
size_t lat_ws_bytes(const kvcar_config &cfg, int max_sources, int max_m, int max_d, int batch, int max_len);
// whether the kernels take such a layer (max_m: widest hidden layer of the context)
bool lat_covers(const kvcar_config &cfg, int max_m, const LatShape &sh);
// decide per layer whether the kernels take it, build tensor maps, place the workspace area
void lat_setup(LatState &st, const kvcar_config &cfg, const std::vector<LayerPlan> &plans, size_t pool_rows,
               int max_sources, int max_m, int max_d, int batch, int max_len, char *ws_area);
bool lat_layer_supported(const LatState &st, int layer);
// The encoder of the same step's new rows, carried by the first and the last launch (null: none).
struct LatEncode {
    EncodeArgs a;
    float *hid;
    int32_t pitch, max_batch, max_m, max_d, max_in;
};
// All launches of one call on `stream`.  lens: host copy of the listed sequences' lengths, not all zero.
cudaError_t lat_launch(LatState &st, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens, int layer, const LatEncode *enc,
                       cudaStream_t stream, int *n_launches);

}  // namespace kvcar
