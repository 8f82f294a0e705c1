// Pieces of lvlm_merge_compact shared between its merge modes.
#pragma once
#include "common.cuh"

namespace lvlm {

constexpr int kMetaInts = 4;           // per sequence: first moved row, ticket counter, merged token, spare

// Launch shape of the kernel that streams the hidden states by input row: 16-byte groups per row, CTAs per
// sequence, cluster size, rows per tile, bytes of a tile's slot in shared memory, tiles in flight.
struct HiddenGrid { int V, cps, cl, rpt, slotB, nstage; };
HiddenGrid hidden_grid(const lvlm_dims* d);

// This layer's K and V for the same launch: the rows merged away are added, times wgt, per (sequence, KV
// head, K|V) into kvP fp32 partial rows (chunks of the image span), kv_partial[b][g][K|V][chunk][128].
struct StreamKv { const void* K; const void* V; int64_t kv_sb, kv_sh; int Hkv, kvP; float* kv_partial; };

// Reads every input row of `hidden` once.  dst_map[b][i] >= 0: the row is copied to that row of
// hidden_out; == -1: it is added, times wgt, to the merged row P_new at row i0+k (wgt != NULL);
// <= -2: it is copied to row -dst-2 of `scratch` (scratch != NULL).  Strides in elements.
// inv_norm (without wgt): [B][k], 1 / |x| of the kept image rows (1 for a zero row), by output row.
// hidden_out == NULL: nothing is stored, only the merged rows are read and one fp32 partial row per cluster
// is left in `partial` ([B][*partials_out][C]) for the in-place compaction that follows.  L gives the launch
// shape at most: fewer CTAs are used when the device cannot run that many clusters at a time.
lvlm_status launch_hidden_rows(const void* hidden, void* hidden_out, int64_t hid_sb, int64_t out_sb,
                               const lvlm_dims* d, const HiddenGrid& L, const int32_t* dst_map,
                               const float* wgt, int32_t* meta, float* partial, void* scratch,
                               int64_t scr_sb, cudaStream_t stream, const StreamKv* kv = nullptr,
                               int32_t* dev_status = nullptr, int* partials_out = nullptr,
                               float* inv_norm = nullptr);

__device__ __forceinline__ float block_sum_fixed(float v, float* scratch) {
    // fixed reduction tree: xor shuffles inside a warp, then warp 0 over the warp sums
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = (threadIdx.x < (blockDim.x >> 5)) ? scratch[threadIdx.x] : 0.f;
    if (threadIdx.x < 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        if (threadIdx.x == 0) scratch[32] = t;
    }
    __syncthreads();
    return scratch[32];
}

// Weight of the merged token at place p of the queue (p = 0 most important), normalised.
__device__ __forceinline__ float merge_weight(int mode, int p, int r1, float inv_sum,
                                              const float* __restrict__ w_custom) {
    switch (mode) {
        case LVLM_W_LINEAR_RANK: return (float)(r1 - p) * inv_sum;
        case LVLM_W_GEOMETRIC: {
            const int q = p < r1 - 1 ? p + 1 : r1 - 1;
            return q <= 126 ? __int_as_float((127 - q) << 23) : ldexpf(1.0f, -q);      // 2^-q
        }
        case LVLM_W_UNIFORM:     return inv_sum;
        default:                 return w_custom[p] * inv_sum;
    }
}

// The rank-weight modes in one launch (merge_once.cu): 16-byte pieces of a row a CTA takes, CTAs of a cluster; P = 0 where the
// launches of merge_compact.cu are taken.  Strides in elements; hidden_out NULL: in place.
struct OnceShape { int P, S; };
struct MergeOnce {
    void* hidden; void* hidden_out; int64_t hid_sb, out_sb; void* K; void* V; int64_t kv_sb, kv_sh;
    int32_t* pos_ids; const int32_t* rank; const float* w_custom; int32_t* new_len; int mode; float inv_sum; int32_t* dev_status;
};
OnceShape merge_once_shape(const lvlm_dims* d);
lvlm_status launch_merge_once(const MergeOnce& m, const lvlm_dims* d, OnceShape s, cudaStream_t stream);

// lvlm_merge_compact in mode LVLM_W_NEAREST_KEPT (nearest_kept.cu).
size_t nearest_kept_workspace(const lvlm_dims* d);
lvlm_status launch_nearest_kept(const void* hidden, void* hidden_out, void* Kc, void* Vc, int32_t* pos_ids,
                                const int32_t* rank, const lvlm_dims* d, float* mass, int32_t* new_len,
                                void* ws, size_t ws_bytes, int32_t* dev_status, cudaStream_t stream);

}  // namespace lvlm
