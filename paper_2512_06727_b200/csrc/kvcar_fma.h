// Interface between the host runtime and the fp32-FMA latent-attention kernels (kvcar_fma.cu).
#pragma once
#include <vector>

#include "kvcar_internal.h"

namespace kvcar {

constexpr int FM_MAX_SRC = 8;         // distinct source layers per K or V of a layer
constexpr int FM_TOK = 64;            // tokens of a partial result, whatever the tile of a launch
constexpr int FM_GROUP_TILES = 1024;  // partial results held at a time (more if one sequence needs more)

// One source layer of K or V, by value in the launches' parameters.
struct FmaSrc {
    const void *pool, *w1t, *w2t;
    const float *s1, *t1, *b2, *qparam;  // qparam: (scale, zero-point) per row of int8 codes, else null
    int32_t d, m, in_dim;
    float slope;
    uint32_t kv_mask;  // KV heads of the reading layer served from this source
};
struct FmaLayer {
    FmaSrc src[2][FM_MAX_SRC];
    int32_t n_src[2];
    const void *cur[2][KVCAR_MAX_KV_HEADS];  // by KV head: its columns of the current-token row of sequence 0
    uint8_t idx[2][KVCAR_MAX_KV_HEADS], slot[2][KVCAR_MAX_KV_HEADS];
    uint8_t ok, quant;
};

struct FmaState {
    std::vector<FmaLayer> layer;
    int max_m = 0, batch = 0, n_sms = 148;
    int group_tiles = 0;
    float *wq = nullptr;     // [source][batch][hq][max_m]: W4_h^T q
    float *score = nullptr;  // [chunk of hidden columns][tile of the group][hq][FM_TOK]: parts of the scores
    float *upart = nullptr;  // [tile of the group][hq][max_m]
    float *ml = nullptr;     // [tile of the group][hq][2]
    float *useq = nullptr, *mlseq = nullptr;  // the same per sequence, where a call takes several groups
    bool per_seq = false;                      // what the last tile launches left behind: results per sequence or per tile,
    int last_parts = 1;                        // and pieces of U per tile
};

size_t fma_ws_bytes(const kvcar_config &cfg, int max_k_sources, int max_m, int batch, int max_len);
void fma_setup(FmaState &st, const kvcar_config &cfg, const std::vector<LayerPlan> &plans, int max_k_sources, int max_m, int batch,
               int max_len, char *ws_area);
inline bool fma_layer_supported(const FmaState &st, int layer) { return !st.layer.empty() && st.layer[layer].ok; }
cudaError_t fma_launch_tiles(FmaState &st, const kvcar_config &cfg, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens,
                             int layer, cudaStream_t stream, int *n_launches);
cudaError_t fma_launch_merge(FmaState &st, const kvcar_config &cfg, const DecodeArgs &a, const SeqList &seqs, const int32_t *lens,
                             int layer, cudaStream_t stream);

}  // namespace kvcar
