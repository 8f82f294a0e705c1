// Declarations shared by the scoring kernels.
#pragma once
#include "common.cuh"

namespace lvlm {

// How a scoring call is cut into tiles and work items (score_tc.cu).
struct ScoreShape {
    int box_h, box_p;          // a query tile: box_h heads of a KV group x box_p positions (row = position * box_h + head)
    int copies;                // pass 1: how often the rows of a query tile lie in its 128 rows
    int npt, nh, tpg;          // position tiles of the window; tiles side by side at a position; query tiles of a KV group
    int nkt;                   // tiles of 128 image keys
    bool small1, small2;       // which shape of the kernel runs the passes
    int ksplit;                // pass 1: work items that share the keys of a query tile
    int parts;                 // pass 2: work items that share the query tiles of a key tile and KV group
    int64_t part_tiles, stat_tiles;    // tiles of results the workspace has room for: pass 2 (column sums), pass 1 (max, sum)
};

struct ScoreLayout { ScoreShape shape; size_t off_partial, off_lse, off_nlse, off_stat, total; };
struct ScoreStrides { int64_t q_sb, q_sn, q_sh, kv_sb, kv_sh; };   // elements

ScoreShape score_shape(const lvlm_dims* d);
bool score_layout(const lvlm_dims* d, ScoreLayout* L);

// Tensor-core path: pass 1 (row normalisers, skipped when the caller supplies lse) and pass 2 (column sums, then score
// and score_head).  ws is laid out as L says.
// normalisers_ready: the workspace already holds the log2-domain normalisers of the window rows, [B][H][window] at
// off_lse (the attention kernel of lvlm_prefill_attn wrote them): pass 1 is skipped.
lvlm_status launch_score_tc(const void* Q, const void* K, const float* lse, const lvlm_dims* d,
                            const ScoreStrides& st, float scale, const ScoreLayout& L, char* ws, float* score,
                            float* score_head, int32_t* dev_status, cudaStream_t stream,
                            bool normalisers_ready = false);

}  // namespace lvlm
