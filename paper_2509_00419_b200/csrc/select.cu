// lvlm_select_topk: total order of the image tokens by (score descending, index ascending).
// Section 3.2.1, paragraph 4: the tokens with the highest scores form P_unmerged, the others
// form P_merged, "reordered by their importance".
//
// The rank of a token is the number of tokens that come before it in that order, so it can be
// counted directly: nothing iterative, every token independent of the others.  Keys are the
// order-preserving image of the score, and among equal keys the lower index comes first.
// grid (blocks of tokens, S, B): a CTA counts, for its tokens, the keys of one slice of the
// sequence that are smaller; the S CTAs of a cluster (one per slice, along y) add their counts
// through distributed shared memory.
//
// A CTA puts the keys of its slice into bins - linear in the key between the slice's extremes or,
// where that leaves a bin deeper than 128 keys (ties, a handful of distinct scores), bounded by a sorted sample
// of the slice's own (key, index) pairs: those are distinct, so such bins stay a few keys deep whatever the scores
// look like.  All keys of lower bins are smaller, so only the token's own bin is read through; how
// the keys happen to be ordered inside a bin does not matter, the count is the same.  Bound by the chain of passes over a slice
// in shared memory (count, scan, scatter, look up), hence many threads with few keys each.
// us of a call; before (256 threads, short slices read through, two atomics and two 64-bit divisions a key) -> now: 576 tokens
// 4.8 -> 4.7, 6000: 12.5 -> 5.8, 32767: 32.6 -> 11.4, 16 sequences of 1792: 16.8 -> 5.1, 4 of 8000: 55.5 -> 6.4.
// The optional outputs (kept list, near-tie count) come from a second, small kernel.
#include "common.cuh"
#include "sm100.cuh"

namespace lvlm {

constexpr int kRankMaxCluster = 8;
constexpr int kRankMaxSlice = 8192;        // keys of a slice in shared memory
constexpr int kRankMaxKeys = kRankMaxCluster * kRankMaxSlice;     // 65536 keys per sequence
constexpr int kRankThreads = 1024;
constexpr int kRankBins = 2048, kRankSamples = 1024, kRankDeep = 128;
constexpr int kRankKeys = kRankMaxSlice / kRankThreads;           // keys a thread puts into bins at most
constexpr int kRankMaxJT = 4;              // tokens a thread ranks at most


struct RankShape { int S, slice_len, jt; };                           // slices, keys of one, tokens a thread ranks

// As many slices as there are CTAs that run at a time (one per SM; clusters of eight leave more SMs idle), not shorter than
// 256 keys; more tokens a thread only where the CTAs would still need a second wave.  us of a call: 16384 tokens, 8 slices in two
// waves 13.1, with two tokens a thread 8.7, 4 slices 7.7; 32767 tokens: 24.6, (four tokens) 16.6, 11.4.
constexpr int kRankCtas = 136, kRankCtas8 = 112;

inline RankShape rank_shape(int n, int B) {
    RankShape r;
    const int64_t blocks = (int64_t)((n + kRankThreads - 1) / kRankThreads) * B;
    int s = 1;
    while (s < kRankMaxCluster && blocks * (2 * s) <= (s == 4 ? kRankCtas8 : kRankCtas) && n / (2 * s) >= 256) s *= 2;
    while (s < kRankMaxCluster && (n + s - 1) / s > kRankMaxSlice) s *= 2;       // a slice has to fit
    r.S = s;
    r.jt = 1;
    while (r.jt < kRankMaxJT && blocks * s > (int64_t)kRankCtas * r.jt) r.jt *= 2;
    r.slice_len = (n + r.S - 1) / r.S;
    return r;
}
inline size_t rank_smem_bytes(int slice_len) { return (size_t)(slice_len + kRankSamples) * 8 + (size_t)(kRankBins + 1) * 4; }

// Ascending sort of P (a power of two) 64-bit keys in shared memory by the whole CTA.
__device__ __forceinline__ void rank_bitonic_sort(uint64_t* keys, int P) {
    for (int k2 = 2; k2 <= P; k2 <<= 1) {
        for (int j = k2 >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < (P >> 1); t += blockDim.x) {
                const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
                const int l = i | j;
                const bool up = (i & k2) == 0;
                const uint64_t a = keys[i], b = keys[l];
                if ((a > b) == up) { keys[i] = b; keys[l] = a; }
            }
            __syncthreads();
        }
    }
}

// Number of keys of the slice (global indices i_lo ..) that come before each of a thread's jt tokens, j_u = (blockIdx.x * jt + u) * kRankThreads + threadIdx.x.
template <typename KeyFn>
__device__ __forceinline__ void rank_by_bins(KeyFn key_of, int n, int i_lo, int slice_len, int jt, unsigned char* smem, int* count) {
    uint64_t* sb = reinterpret_cast<uint64_t*>(smem);                    // [slice_len] (key, index), bin by bin
    uint64_t* spl = sb + slice_len;                                      // [kRankSamples] sorted sample: bin boundaries
    int* start = reinterpret_cast<int*>(spl + kRankSamples);             // [kRankBins + 1]
    __shared__ int s_scan[33];
    __shared__ uint32_t s_min[32], s_max[32];
    __shared__ int s_deep;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nvalid = max(0, min(slice_len, n - i_lo));
    uint32_t key[kRankKeys], kj[kRankMaxJT];
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
#pragma unroll
    for (int u = 0; u < kRankKeys; ++u) {
        const int i = u * kRankThreads + tid;
        key[u] = 0u;
        if (i < nvalid) { key[u] = key_of(i_lo + i); lo = min(lo, key[u]); hi = max(hi, key[u]); }
    }
#pragma unroll
    for (int u = 0; u < kRankMaxJT; ++u) {
        const int j = (blockIdx.x * jt + u) * kRankThreads + tid;
        kj[u] = u < jt && j < n ? key_of(j) : 0u;
        count[u] = 0;
    }
    lo = __reduce_min_sync(0xFFFFFFFFu, lo);
    hi = __reduce_max_sync(0xFFFFFFFFu, hi);
    if (lane == 0) { s_min[warp] = lo; s_max[warp] = hi; }
    if (tid == 0) s_deep = 0;
    for (int i = tid; i <= kRankBins; i += kRankThreads) start[i] = 0;
    __syncthreads();
    lo = __reduce_min_sync(0xFFFFFFFFu, s_min[lane]);
    hi = __reduce_max_sync(0xFFFFFFFFu, s_max[lane]);
    // Bins linear in the key.  Any function that never falls as the key grows will do: in 32-bit floats.
    const float scale = (float)kRankBins / ((float)(hi - lo) + 1.f);
    auto bin_linear = [&](uint32_t k) { return k <= lo ? 0 : k >= hi ? kRankBins - 1 : min(kRankBins - 1, (int)((float)(k - lo) * scale)); };
    // bin of a pair = number of boundaries spl[1..] that are <= it (binary search)
    auto bin_sampled = [&](uint64_t k) {
        int lo_i = 0, hi_i = kRankSamples - 1;                           // boundaries spl[1 + lo_i .. 1 + hi_i)
        while (lo_i < hi_i) {
            const int mid = (lo_i + hi_i) >> 1;
            if (spl[1 + mid] <= k) lo_i = mid + 1; else hi_i = mid;
        }
        return lo_i;
    };
    auto pair_of = [&](uint32_t k, int i) { return ((uint64_t)k << 32) | (uint32_t)i; };
    int place[kRankKeys];                                                 // place within the bin (16 bits), bin
    bool deep = false;
#pragma unroll
    for (int u = 0; u < kRankKeys; ++u) {
        place[u] = 0;
        if (u * kRankThreads + tid < nvalid) {
            const int bin = bin_linear(key[u]), c = atomicAdd(&start[bin], 1);
            place[u] = (bin << 16) | c;
            deep |= c >= kRankDeep;
        }
    }
    if (deep) s_deep = 1;
    __syncthreads();
    const bool sampled = s_deep != 0;
    if (sampled) {
        for (int t = tid; t < kRankSamples; t += kRankThreads) {
            const int i = nvalid >= kRankSamples ? (int)(((int64_t)t * nvalid) / kRankSamples) : t;
            spl[t] = i < nvalid ? pair_of(key_of(i_lo + i), i_lo + i) : ~0ull;      // padding sorts last and bounds nothing
        }
        for (int i = tid; i <= kRankBins; i += kRankThreads) start[i] = 0;
        __syncthreads();
        rank_bitonic_sort(spl, kRankSamples);
#pragma unroll
        for (int u = 0; u < kRankKeys; ++u) {
            const int i = u * kRankThreads + tid;
            if (i < nvalid) {
                const int bin = bin_sampled(pair_of(key[u], i_lo + i));
                place[u] = (bin << 16) | atomicAdd(&start[bin], 1);
            }
        }
        __syncthreads();
    }
    {   // exclusive scan of the bin counts
        constexpr int kPer = kRankBins / kRankThreads;
        int c[kPer], sum = 0, total;
#pragma unroll
        for (int u = 0; u < kPer; ++u) { c[u] = start[tid * kPer + u]; sum += c[u]; }
        int run = block_exclusive_scan(sum, s_scan, &total);
#pragma unroll
        for (int u = 0; u < kPer; ++u) { start[tid * kPer + u] = run; run += c[u]; }
        if (tid == 0) start[kRankBins] = total;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kRankKeys; ++u) {
        const int i = u * kRankThreads + tid;
        if (i < nvalid) sb[start[place[u] >> 16] + (place[u] & 0xFFFF)] = pair_of(key[u], i_lo + i);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kRankMaxJT; ++u) {
        const int j = (blockIdx.x * jt + u) * kRankThreads + tid;
        if (nvalid > 0 && u < jt && j < n) {
            const uint64_t me = pair_of(kj[u], j);
            const int bin = sampled ? bin_sampled(me) : bin_linear(kj[u]);
            const int p0 = start[bin], p1 = start[bin + 1];
            int cnt = p0;
            for (int p = p0; p < p1; ++p) cnt += (int)(sb[p] < me);
            count[u] = cnt;
        }
    }
}

// grid (blocks of kRankThreads * jt tokens, S, B), clusters (1, S, 1).
__global__ void __launch_bounds__(kRankThreads)
select_count_kernel(const float* __restrict__ score, int64_t stride, int n, int S, int slice_len, int jt,
                    int32_t* __restrict__ rank, int32_t* dev_status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_cnt[kRankMaxJT * kRankThreads];
    pdl_enter();
    const int b = blockIdx.z, s = (int)sm100::cluster_ctarank(), tid = threadIdx.x;
    const float* row = score + (int64_t)b * stride;
    bool nonfinite = false;
    auto key_of = [&](int i) { return desc_key(row[i], &nonfinite); };
    int cnt[kRankMaxJT];
    rank_by_bins(key_of, n, s * slice_len, slice_len, jt, smem_raw, cnt);
    if (S > 1) {
#pragma unroll
        for (int u = 0; u < kRankMaxJT; ++u) s_cnt[u * kRankThreads + tid] = cnt[u];
        sm100::cluster_barrier();
    }
    if (s == 0) {
#pragma unroll
        for (int u = 0; u < kRankMaxJT; ++u) {
            const int j = (blockIdx.x * jt + u) * kRankThreads + tid;
            if (u < jt && j < n) {
                int tot = cnt[u];
                for (int r = 1; r < S; ++r) tot += sm100::cluster_ld(&s_cnt[u * kRankThreads + tid], r);
                rank[(int64_t)b * n + j] = tot;
            }
        }
    }
    // every key is looked at by the CTAs of slice 0 as "their own" key: one report is enough
    if (nonfinite && blockIdx.y == 0 && dev_status) atomicOr(dev_status, LVLM_DEV_NONFINITE);
    if (S > 1) sm100::cluster_barrier();                    // nobody leaves while its counts are read
}

// One CTA per sequence: the kept tokens in ascending order (prefix sum of rank < k over the index) and
// the number of near-ties among neighbours (p, p+1) of the order with p+1 >= k.
__global__ void __launch_bounds__(1024)
select_aux_kernel(const float* __restrict__ score, int64_t stride, int n, int k,
                  const int32_t* __restrict__ rank, int32_t* __restrict__ kept_idx,
                  int32_t* __restrict__ near_tie) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    int32_t* order = reinterpret_cast<int32_t*>(smem_raw);           // [n] token at every place of the order
    __shared__ int scan_scratch[33];
    __shared__ int s_near;
    pdl_enter();
    const int b = blockIdx.x;
    const float* row = score + (int64_t)b * stride;
    const int32_t* rk = rank + (int64_t)b * n;
    if (threadIdx.x == 0) s_near = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int p = rk[j];
        if (p >= 0 && p < n) order[p] = j;
    }
    __syncthreads();
    if (near_tie) {
        int near = 0;
        for (int p = threadIdx.x + max(k - 1, 0); p + 1 < n; p += blockDim.x) {
            const float a = row[order[p]], c = row[order[p + 1]];
            const float dgap = __fsub_rn(a, c);
            const float t = __fmul_rn(1e-4f, fabsf(a));
            if (dgap < t) ++near;
        }
        near = warp_sum(near);
        if ((threadIdx.x & 31) == 0 && near) atomicAdd(&s_near, near);
        __syncthreads();
        if (threadIdx.x == 0) near_tie[b] = s_near;
    }
    if (kept_idx && k > 0) {
        const int per = (n + blockDim.x - 1) / blockDim.x;
        const int j0 = min(n, (int)threadIdx.x * per), j1 = min(n, j0 + per);
        int cnt = 0;
        for (int j = j0; j < j1; ++j) cnt += rk[j] < k;
        int total;
        int off = block_exclusive_scan(cnt, scan_scratch, &total);
        for (int j = j0; j < j1; ++j)
            if (rk[j] < k && off < k) kept_idx[(int64_t)b * k + off++] = j;
    }
}

}  // namespace lvlm

extern "C" lvlm_status lvlm_select_topk(const float* score, int B, int n, int64_t score_stride,
                                         int k, int32_t* rank, int32_t* kept_idx,
                                         int32_t* near_tie, void* ws, size_t ws_bytes,
                                         int32_t* dev_status, void* stream_) {
    using namespace lvlm;
    (void)ws; (void)ws_bytes;
    cudaStream_t stream = (cudaStream_t)stream_;
    if (!score || !rank || B <= 0 || n <= 0 || k < 0 || k > n) return LVLM_ERR_INVALID_ARG;
    if (score_stride == 0) score_stride = n;
    if (score_stride < n) return LVLM_ERR_INVALID_ARG;
    if (n > kRankMaxKeys) return LVLM_ERR_UNSUPPORTED;
    if ((kept_idx || near_tie) && (size_t)n * 4 > (size_t)kMaxDynSmem) return LVLM_ERR_UNSUPPORTED;
    const RankShape r = rank_shape(n, B);
    {
        LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(select_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem));
        const int tokens = kRankThreads * r.jt;
        const lvlm_status st = launch_kernel_cluster(select_count_kernel, dim3((n + tokens - 1) / tokens, r.S, B), dim3(kRankThreads),
                                                     rank_smem_bytes(r.slice_len), stream, dim3(1, r.S, 1),
                                                     score, score_stride, n, r.S, r.slice_len, r.jt, rank, dev_status);
        if (st != LVLM_OK) return st;
    }
    if (!kept_idx && !near_tie) return LVLM_OK;
    LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(select_aux_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem));
    const int threads = n >= 1024 ? 1024 : ((n + 31) / 32) * 32;
    return launch_kernel(select_aux_kernel, dim3(B), dim3(threads), (size_t)n * 4, stream, 1,
                         score, score_stride, n, k, rank, kept_idx, near_tie);
}
