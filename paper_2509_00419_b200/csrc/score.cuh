// Declarations shared by the scoring kernels.
#pragma once
#include "common.cuh"
#include "sm100.cuh"

namespace lvlm {

// n / d for 0 <= n < 2^31 by a multiplication: every warp of a CTA takes every work item apart.
struct FastDiv {
    uint32_t d, m, sh;
    FastDiv() = default;
    explicit FastDiv(int div) : d((uint32_t)div), sh(0) {
        while ((1u << sh) < d) ++sh;
        m = (uint32_t)(((((uint64_t)1 << sh) - d) << 32) / d + 1);
    }
    __device__ __forceinline__ int div(int n) const { return (int)((__umulhi(m, (uint32_t)n) + (uint32_t)n) >> sh); }
    __device__ __forceinline__ int divmod(int n, int* rem) const { const int q = div(n); *rem = n - q * (int)d; return q; }
};

// 16 TMEM lanes x 32 fp32 columns: thread l has rows l/4 and l/4 + 8, columns 8 i + 2 (l % 4) + {0, 1}.
__device__ __forceinline__ void tmem_ld_16x256b_x4(uint32_t taddr, float* v) {
    uint32_t* r = reinterpret_cast<uint32_t*>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}

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

// One pass over Q K^T (score_once.cu): key tiles of a CTA, CTAs of a cluster, work items that share the query tiles of a KV
// group, clusters; kt = 0 where the two passes of score_tc.cu are taken.  Leaves column sums for score_sum_kernel,
// [B][Hkv * parts][nkt * 128].
struct OnceScoreShape { int kt, S, parts, clusters; };
OnceScoreShape score_once_shape(const lvlm_dims* d, const ScoreShape& s, float scale);
lvlm_status launch_score_once(const CUtensorMap& qmap, const CUtensorMap& kmap, const lvlm_dims* d, const ScoreShape& s,
                              const OnceScoreShape& o, float scale, float* partial, int32_t* dev_status, cudaStream_t stream);

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
