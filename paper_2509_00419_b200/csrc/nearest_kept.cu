// lvlm_merge_compact, mode LVLM_W_NEAREST_KEPT.  Not in the paper (which argues against
// similarity-based merging, Section 3.2.1, paragraph 3): every dropped image token is averaged
// into the kept image token whose hidden row has the highest cosine similarity with its own
// (lower kept index wins ties); masses make repeated merging a true mean.
//
// Launches, all on the caller's stream:
//   plan      a cluster per sequence: kept / dropped token lists, row map, position ids, new length
//   rows      the streaming kernel of the hidden states: kept rows to their place in the output, with 1 / |x_t| on the way,
//             dropped rows side by side into scratch
//   sim       dropped x kept similarity on the tensor cores (tcgen05, accumulators in TMEM, operands by
//             TMA), arg-max per dropped row in the epilogue, merged over column splits with atomicMax
//             on (similarity, ~index) keys
//   group     dropped tokens by kept token: counts, places, and the tokens of a kept token in ascending order
//   merge     every kept row becomes the mass-weighted mean of itself and its segment, in token order
//   K, V      the same mean per KV head, and the rows behind the image, into scratch; then stored in place
//   mass      token masses compacted in place
// us at 16384 + 256 tokens of 6144 channels, 4096 kept: plan 10, similarity 405 (618 GFLOP: 1527 TFLOP/s), group 22, K and V 35;
// rows 64 and merge 46 run at the copy rate.
#include "common.cuh"
#include "merge.cuh"
#include "sm100.cuh"

namespace lvlm {

using namespace sm100;

constexpr int kMaxDropped = 65536;

struct NkLayout {
    int r, Nout, V;
    HiddenGrid grid;
    int rest;                           // rows behind the image
    size_t off_assign, off_dst, off_kept, off_drop, off_inv, off_best, off_place, off_order, off_seg, off_newmass,
           off_scratch, off_kvtmp, total;
};

static bool nk_layout(const lvlm_dims* d, NkLayout* L) {
    if (!d || d->B <= 0 || d->N <= 0 || d->n <= 0 || d->C <= 0 || d->C % 8 || d->i0 < 0 ||
        d->k < 0 || d->k > d->n || (int64_t)d->i0 + d->n > d->N)
        return false;
    const size_t B = d->B, k = d->k, r = d->n - d->k;
    L->r = (int)r;
    L->Nout = d->N - (int)r;
    L->V = d->C / 8;
    L->grid = hidden_grid(d);
    size_t off = 0;
    L->off_assign = off;  off = align_up(off + B * (r ? r : 1) * 4, 256);   // first: callers may read it
    L->rest = d->N - d->i0 - d->n;
    L->off_dst = off;     off = align_up(off + B * d->N * 4, 256);
    L->off_kept = off;    off = align_up(off + B * (k ? k : 1) * 4, 256);
    L->off_drop = off;    off = align_up(off + B * (r ? r : 1) * 4, 256);
    L->off_inv = off;     off = align_up(off + B * (k ? k : 1) * 4, 256);
    L->off_best = off;    off = align_up(off + B * (r ? r : 1) * 8, 256);
    L->off_place = off;   off = align_up(off + B * (r ? r : 1) * 4, 256);
    L->off_order = off;   off = align_up(off + B * (r ? r : 1) * 8, 256);
    L->off_seg = off;     off = align_up(off + B * (k + 1) * 4, 256);
    L->off_newmass = off; off = align_up(off + B * (k ? k : 1) * 4, 256);
    // The dropped hidden rows and, once they are merged, the rows of K and V on their way back into the cache lie in the same
    // place.  (Of these it is k and those behind the image; counted are N, which does not fall as the image span grows.)
    const size_t hid = B * (r ? r : 1) * (size_t)d->C * 2, kv = B * (d->Hkv > 0 ? d->Hkv : 0) * 2 * d->N * (size_t)kHeadDim * 2;
    L->off_scratch = L->off_kvtmp = off; off = align_up(off + (hid > kv ? hid : kv), 256);
    L->total = off;
    return true;
}

size_t nearest_kept_workspace(const lvlm_dims* d) {
    NkLayout L;
    return nk_layout(d, &L) ? L.total : 0;
}

// ---- plan ------------------------------------------------------------------------------------------

// A cluster of P CTAs per sequence (grid (P, B)), CTA c the c-th run of the image tokens: it counts its kept tokens, learns
// from the lower ranks how many came before, then writes its run tile by tile (thread = token, coalesced; one CTA with
// a run of tokens per thread took 39 us for 16384 tokens).  kept[q] / drop[q]: image-token indices in ascending
// order.  dst[i]: output row of input row i, or -2-q for the q-th dropped token.  Position ids are compacted in place in
// rounds (sources lie at or after their destination): every CTA loads its rows of the round, a barrier, then stores.
__global__ void __launch_bounds__(1024)
nk_plan_kernel(const int32_t* __restrict__ rank, int32_t* pos_ids, int N, int i0, int n, int k,
               int32_t* __restrict__ dst_map, int32_t* kept, int32_t* __restrict__ drop,
               unsigned long long* __restrict__ best, int32_t* __restrict__ seg, int32_t* new_len, int32_t* dev_status) {
    __shared__ int scan_scratch[33];
    __shared__ int s_total;
    pdl_enter();
    const int b = blockIdx.y, r = n - k, Nout = N - r, P = (int)gridDim.x, cr = (int)cluster_ctarank();
    const int32_t* rk = rank + (int64_t)b * n;
    int32_t* dst = dst_map + (int64_t)b * N;
    int32_t* kp = kept + (int64_t)b * k;
    const int chunk = (n + P - 1) / P;
    const int c_lo = min(n, cr * chunk), c_hi = min(n, c_lo + chunk);
    if (threadIdx.x == 0) s_total = 0;
    __syncthreads();
    bool bad = false;
    int mine = 0;
    for (int j = c_lo + threadIdx.x; j < c_hi; j += blockDim.x) {
        const int rj = rk[j];
        if (rj < 0 || rj >= n) bad = true;
        mine += rj < k;
    }
    mine = warp_sum(mine);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&s_total, mine);
    cluster_barrier();
    int kq = 0, all = 0;
    for (int c = 0; c < P; ++c) {
        const int t = cluster_ld(&s_total, c);
        kq += c < cr ? t : 0;
        all += t;
    }
    if (all != k) bad = true;
    for (int t0 = c_lo; t0 < c_hi; t0 += blockDim.x) {
        const int j = t0 + threadIdx.x;
        const int is_kept = j < c_hi && rk[j] < k;
        int total;
        const int q = kq + block_exclusive_scan(is_kept, scan_scratch, &total);         // kept tokens before mine
        if (j < c_hi) {
            const int dq = j - q;                                                       // dropped tokens before mine
            if (is_kept) {
                if (q < k) kp[q] = j;
                dst[i0 + j] = q < k ? i0 + q : -2 - min(dq, max(r - 1, 0));              // (inconsistent rank: flagged below)
            } else {
                if (dq < r) { drop[(int64_t)b * r + dq] = j; best[(int64_t)b * r + dq] = 0ull; }
                dst[i0 + j] = dq < r ? -2 - dq : i0;
            }
        }
        kq += total;
    }
    const int first = cr * blockDim.x + threadIdx.x, step = P * blockDim.x;
    for (int o = first; o < i0; o += step) dst[o] = o;
    for (int o = i0 + k + first; o < Nout; o += step) dst[o + r] = o;
    for (int t = first; t <= k; t += step) seg[(int64_t)b * (k + 1) + t] = 0;            // counts, to begin with
    if (bad && dev_status) atomicOr(dev_status, LVLM_DEV_BOUNDS);
    if (cr == 0 && threadIdx.x == 0 && new_len) new_len[b] = Nout;
    cluster_barrier();                                                               // the kept list is complete
    if (pos_ids) {
        int32_t* pid = pos_ids + (int64_t)b * N;
        for (int o0 = i0; o0 < Nout; o0 += step) {
            const int o = o0 + first;
            int val = 0;
            if (o < Nout) val = pid[o < i0 + k ? i0 + (all == k ? kp[o - i0] : o - i0) : o + r];
            cluster_barrier();
            if (o < Nout) pid[o] = val;
        }
    }
    cluster_barrier();                                  // nobody leaves while its shared memory may still be read
}

// ---- group -----------------------------------------------------------------------------------------
// Dropped tokens by the kept token they go to.  count: the assignment, how many go to every kept token (in seg) and a
// place among them, in order of arrival.  place: where every kept token's segment starts, and every dropped token into
// its segment.  sort: the segments, a few tokens each, in ascending token order - so the order of arrival does not matter.
// (Ranking all tokens against each other took 92 us for 12288 of them.)
__global__ void __launch_bounds__(256)
nk_count_kernel(const unsigned long long* __restrict__ best, int r, int k, int32_t* __restrict__ assign,
                int32_t* __restrict__ place, int32_t* seg) {
    pdl_enter();
    const int b = blockIdx.y, q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= r) return;
    uint32_t t = 0xFFFFFFFFu - (uint32_t)(__ldcg(best + (int64_t)b * r + q) & 0xFFFFFFFFull);
    t = t < (uint32_t)k ? t : 0u;                          // nothing won: kept token 0
    assign[(int64_t)b * r + q] = (int)t;
    place[(int64_t)b * r + q] = atomicAdd(seg + (int64_t)b * (k + 1) + t, 1);
}

// One CTA per sequence.  order[p] = (dropped token q, its image-token index).
__global__ void __launch_bounds__(1024)
nk_place_kernel(int32_t* seg, int r, int k, const int32_t* __restrict__ assign, const int32_t* __restrict__ place,
                const int32_t* __restrict__ drop, int2* __restrict__ order) {
    __shared__ int scan_scratch[33];
    pdl_enter();
    const int b = blockIdx.x;
    int32_t* sg = seg + (int64_t)b * (k + 1);
    int before = 0;
    for (int t0 = 0; t0 < k + 1; t0 += 4 * blockDim.x) {   // four consecutive counts a thread
        int c[4], sum = 0, total;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = t0 + threadIdx.x * 4 + u;
            c[u] = t < k ? sg[t] : 0;
            sum += c[u];
        }
        int run = before + block_exclusive_scan(sum, scan_scratch, &total);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int t = t0 + threadIdx.x * 4 + u;
            if (t <= k) sg[t] = run;
            run += c[u];
        }
        before += total;
    }
    __syncthreads();
    for (int q = threadIdx.x; q < r; q += blockDim.x) {
        const int64_t i = (int64_t)b * r + q;
        order[(int64_t)b * r + sg[assign[i]] + place[i]] = make_int2(q, drop[i]);
    }
}

// A warp per kept token; the segments with more than 32 tokens are sorted by the CTA, through a bitmap of the dropped tokens.
constexpr int kSortWarps = 8;
__global__ void __launch_bounds__(kSortWarps * 32)
nk_sort_kernel(const int32_t* __restrict__ seg, int r, int k, const int32_t* __restrict__ drop, int2* __restrict__ order) {
    __shared__ uint32_t bits[kMaxDropped / 32];
    __shared__ int scan_scratch[33];
    __shared__ int s_long[kSortWarps];
    pdl_enter();
    const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * kSortWarps + warp;
    const int32_t* sg = seg + (int64_t)b * (k + 1);
    int2* ord = order + (int64_t)b * r;
    const int p0 = t < k ? sg[t] : 0, len = t < k ? sg[t + 1] - p0 : 0;
    if (lane == 0) s_long[warp] = len > 32;
    if (len > 1 && len <= 32) {
        const int2 mine = lane < len ? ord[p0 + lane] : make_int2(0x7FFFFFFF, 0);
        int at = 0;
        for (int i = 0; i < len; ++i) at += __shfl_sync(0xFFFFFFFFu, mine.x, i) < mine.x;
        __syncwarp();
        if (lane < len) ord[p0 + at] = mine;
    }
    __syncthreads();
    for (int w = 0; w < kSortWarps; ++w) {
        if (!s_long[w]) continue;
        const int tw = blockIdx.x * kSortWarps + w, q0 = sg[tw], q1 = sg[tw + 1];
        const int words = (r + 31) / 32, per = (words + (int)blockDim.x - 1) / (int)blockDim.x;
        for (int i = threadIdx.x; i < words; i += blockDim.x) bits[i] = 0u;
        __syncthreads();
        for (int p = q0 + threadIdx.x; p < q1; p += blockDim.x) { const int q = ord[p].x; atomicOr(&bits[q >> 5], 1u << (q & 31)); }
        __syncthreads();
        const int w0 = min(words, (int)threadIdx.x * per), w1 = min(words, w0 + per);
        int cnt = 0, total;
        for (int i = w0; i < w1; ++i) cnt += __popc(bits[i]);
        int p = q0 + block_exclusive_scan(cnt, scan_scratch, &total);
        for (int i = w0; i < w1; ++i)
            for (uint32_t m = bits[i]; m; m &= m - 1) {
                const int q = i * 32 + __ffs((int)m) - 1;
                ord[p++] = make_int2(q, drop[(int64_t)b * r + q]);
            }
        __syncthreads();
    }
}

// ---- merge of the hidden rows ------------------------------------------------------------------------
// grid (CTAs per sequence, B); a CTA takes kept rows cta, cta + grid.x, ... (segments differ in
// length, striding evens them out).  Thread = 16-byte column group (+256 ...).  Row t of the output
// already holds x_t; its segment's rows come from scratch, four in flight, added in token order.
constexpr int kNkThreads = 256;

template <int CH>
__global__ void __launch_bounds__(kNkThreads)
nk_merge_kernel(uint4* __restrict__ out, int64_t out_stride_b, const uint4* __restrict__ scratch,
                int64_t scr_stride_b, int V, int N, int i0, int k, int r,
                const int32_t* __restrict__ kept, const int2* __restrict__ order, const int32_t* __restrict__ seg,
                const float* __restrict__ mass, float* __restrict__ newmass) {
    pdl_enter();
    const int b = blockIdx.y, tid = threadIdx.x;
    uint4* orow = out + (int64_t)b * out_stride_b + (int64_t)i0 * V;
    const uint4* srow = scratch + (int64_t)b * scr_stride_b;
    const int2* ord = order + (int64_t)b * r;
    const float* ms = mass ? mass + (int64_t)b * N + i0 : nullptr;
    for (int t = blockIdx.x; t < k; t += gridDim.x) {
        const int p0 = seg[(int64_t)b * (k + 1) + t], p1 = seg[(int64_t)b * (k + 1) + t + 1];
        const float mt = ms ? ms[min(max(kept[(int64_t)b * k + t], 0), k + r - 1)] : 1.f;
        float den = mt;
        float acc[CH][8];
#pragma unroll
        for (int ci = 0; ci < CH; ++ci) {
            const int c = tid + ci * kNkThreads;
            const uint4 x = c < V ? orow[(int64_t)t * V + c] : make_uint4(0, 0, 0, 0);
            acc[ci][0] = mt * bf16_lo(x.x); acc[ci][1] = mt * bf16_hi(x.x);
            acc[ci][2] = mt * bf16_lo(x.y); acc[ci][3] = mt * bf16_hi(x.y);
            acc[ci][4] = mt * bf16_lo(x.z); acc[ci][5] = mt * bf16_hi(x.z);
            acc[ci][6] = mt * bf16_lo(x.w); acc[ci][7] = mt * bf16_hi(x.w);
        }
        for (int pb = p0; pb < p1; pb += 4) {
            float md[4];
            uint4 x[4][CH];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = pb + u;
                const int2 e = p < p1 ? ord[p] : make_int2(0, 0);
                const int q = e.x;
                md[u] = p < p1 ? (ms ? ms[min(max(e.y, 0), k + r - 1)] : 1.f) : 0.f;
#pragma unroll
                for (int ci = 0; ci < CH; ++ci) {
                    const int c = tid + ci * kNkThreads;
                    x[u][ci] = (p < p1 && c < V) ? __ldg(srow + (int64_t)q * V + c) : make_uint4(0, 0, 0, 0);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (pb + u < p1) {
                    den += md[u];
#pragma unroll
                    for (int ci = 0; ci < CH; ++ci) {
                        const uint4 xv = x[u][ci];
                        acc[ci][0] = fmaf(md[u], bf16_lo(xv.x), acc[ci][0]); acc[ci][1] = fmaf(md[u], bf16_hi(xv.x), acc[ci][1]);
                        acc[ci][2] = fmaf(md[u], bf16_lo(xv.y), acc[ci][2]); acc[ci][3] = fmaf(md[u], bf16_hi(xv.y), acc[ci][3]);
                        acc[ci][4] = fmaf(md[u], bf16_lo(xv.z), acc[ci][4]); acc[ci][5] = fmaf(md[u], bf16_hi(xv.z), acc[ci][5]);
                        acc[ci][6] = fmaf(md[u], bf16_lo(xv.w), acc[ci][6]); acc[ci][7] = fmaf(md[u], bf16_hi(xv.w), acc[ci][7]);
                    }
                }
            }
        }
        if (p1 > p0) {                                      // a row nothing was merged into stays as it is
            const float inv = 1.0f / den;
#pragma unroll
            for (int ci = 0; ci < CH; ++ci) {
                const int c = tid + ci * kNkThreads;
                if (c < V) {
                    uint4 o;
                    o.x = pack_bf16(acc[ci][0] * inv, acc[ci][1] * inv); o.y = pack_bf16(acc[ci][2] * inv, acc[ci][3] * inv);
                    o.z = pack_bf16(acc[ci][4] * inv, acc[ci][5] * inv); o.w = pack_bf16(acc[ci][6] * inv, acc[ci][7] * inv);
                    orow[(int64_t)t * V + c] = o;
                }
            }
        }
        if (tid == 0) newmass[(int64_t)b * k + t] = den;
    }
}

// ---- K and V ---------------------------------------------------------------------------------------------
// The same mean per (sequence, KV head, tensor), read from the cache as it stands, and the rows behind the image as they
// are, parked in scratch (a row of the cache may be the source of a row before it): 16 threads per 256-byte row, 16
// rows per CTA.  Then stored.
// A thread has the row in kKvSeqs of the Hkv * 2 sequences: they share the segment, whose look-up is a chain of loads.
constexpr int kKvSeqs = 4;
__global__ void __launch_bounds__(kNkThreads)
nk_kv_merge_kernel(const uint4* __restrict__ Kc, const uint4* __restrict__ Vc, int64_t kv_sb, int64_t kv_sh,
                   int Hkv, int N, int i0, int n, int k, int r, int rest, const int32_t* __restrict__ kept,
                   const int2* __restrict__ order, const int32_t* __restrict__ seg, const float* __restrict__ mass,
                   uint4* __restrict__ kvtmp) {
    pdl_enter();
    const int b = blockIdx.z, s0 = blockIdx.y * kKvSeqs;
    const int c = threadIdx.x & 15, t = blockIdx.x * 16 + (threadIdx.x >> 4);
    if (t >= k + rest) return;
    const uint4* rows[kKvSeqs];
    uint4* to = kvtmp + (((int64_t)b * Hkv * 2 + s0) * (k + rest) + t) * 16 + c;
    const int64_t to_step = (int64_t)(k + rest) * 16;
#pragma unroll
    for (int s = 0; s < kKvSeqs; ++s) {                           // (past the last sequence: the last one again, not stored)
        const int sq = min(s0 + s, Hkv * 2 - 1);
        rows[s] = ((sq & 1) ? Vc : Kc) + (int64_t)b * kv_sb + (int64_t)(sq >> 1) * kv_sh + (int64_t)i0 * 16 + c;
    }
    const int p0 = t < k ? seg[(int64_t)b * (k + 1) + t] : 0, p1 = t < k ? seg[(int64_t)b * (k + 1) + t + 1] : 0;
    // (a rank that is no permutation leaves gaps in the list)
    const int jt = t < k ? min(max(kept[(int64_t)b * k + t], 0), n - 1) : n + t - k;
    uint4 own[kKvSeqs];
#pragma unroll
    for (int s = 0; s < kKvSeqs; ++s) own[s] = rows[s][(int64_t)jt * 16];
    if (p1 > p0) {                                                // (otherwise: the row as it is)
        const float* ms = mass ? mass + (int64_t)b * N + i0 : nullptr;
        const int2* ord = order + (int64_t)b * r;
        const float mt = ms ? ms[jt] : 1.f;
        float den = mt, acc[kKvSeqs][8];
#pragma unroll
        for (int s = 0; s < kKvSeqs; ++s) {
            acc[s][0] = mt * bf16_lo(own[s].x); acc[s][1] = mt * bf16_hi(own[s].x); acc[s][2] = mt * bf16_lo(own[s].y); acc[s][3] = mt * bf16_hi(own[s].y);
            acc[s][4] = mt * bf16_lo(own[s].z); acc[s][5] = mt * bf16_hi(own[s].z); acc[s][6] = mt * bf16_lo(own[s].w); acc[s][7] = mt * bf16_hi(own[s].w);
        }
        for (int pb = p0; pb < p1; pb += 2) {
            float md[2];
            uint4 x[2][kKvSeqs];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int p = pb + u;
                const int jd = p < p1 ? min(max(ord[p].y, 0), n - 1) : 0;
                md[u] = p < p1 ? (ms ? ms[jd] : 1.f) : 0.f;
#pragma unroll
                for (int s = 0; s < kKvSeqs; ++s) x[u][s] = p < p1 ? rows[s][(int64_t)jd * 16] : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                if (pb + u < p1) {
                    den += md[u];
#pragma unroll
                    for (int s = 0; s < kKvSeqs; ++s) {
                        const uint4 v = x[u][s];
                        acc[s][0] = fmaf(md[u], bf16_lo(v.x), acc[s][0]); acc[s][1] = fmaf(md[u], bf16_hi(v.x), acc[s][1]);
                        acc[s][2] = fmaf(md[u], bf16_lo(v.y), acc[s][2]); acc[s][3] = fmaf(md[u], bf16_hi(v.y), acc[s][3]);
                        acc[s][4] = fmaf(md[u], bf16_lo(v.z), acc[s][4]); acc[s][5] = fmaf(md[u], bf16_hi(v.z), acc[s][5]);
                        acc[s][6] = fmaf(md[u], bf16_lo(v.w), acc[s][6]); acc[s][7] = fmaf(md[u], bf16_hi(v.w), acc[s][7]);
                    }
                }
            }
        }
        const float inv = 1.0f / den;
#pragma unroll
        for (int s = 0; s < kKvSeqs; ++s) {
            own[s].x = pack_bf16(acc[s][0] * inv, acc[s][1] * inv); own[s].y = pack_bf16(acc[s][2] * inv, acc[s][3] * inv);
            own[s].z = pack_bf16(acc[s][4] * inv, acc[s][5] * inv); own[s].w = pack_bf16(acc[s][6] * inv, acc[s][7] * inv);
        }
    }
#pragma unroll
    for (int s = 0; s < kKvSeqs; ++s)
        if (s0 + s < Hkv * 2) to[s * to_step] = own[s];
}

// grid (CTAs, Hkv * 2, B): four 16-byte words a thread.
__global__ void __launch_bounds__(kNkThreads)
nk_kv_store_kernel(uint4* __restrict__ Kc, uint4* __restrict__ Vc, int64_t kv_sb, int64_t kv_sh, int Hkv,
                   int i0, int rows_out, const uint4* __restrict__ kvtmp) {
    pdl_enter();
    const int b = blockIdx.z, g = blockIdx.y >> 1, which = blockIdx.y & 1, words = rows_out * 16;
    uint4* to = (which ? Vc : Kc) + (int64_t)b * kv_sb + (int64_t)g * kv_sh + (int64_t)i0 * 16;
    const uint4* from = kvtmp + (((int64_t)b * Hkv + g) * 2 + which) * words;
    const int c = blockIdx.x * 4 * kNkThreads + threadIdx.x;
    uint4 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) if (c + u * kNkThreads < words) x[u] = __ldcg(from + c + u * kNkThreads);
#pragma unroll
    for (int u = 0; u < 4; ++u) if (c + u * kNkThreads < words) to[c + u * kNkThreads] = x[u];
}

// Token masses, in place: the kept tokens take their new mass, the rows behind the image move up.
__global__ void __launch_bounds__(1024)
nk_mass_kernel(float* mass, int N, int i0, int k, int r, const float* __restrict__ newmass) {
    pdl_enter();
    const int b = blockIdx.x, Nout = N - r;
    float* m = mass + (int64_t)b * N;
    for (int o0 = i0; o0 < Nout; o0 += blockDim.x) {
        const int o = o0 + threadIdx.x;
        float val = 0.f;
        __syncthreads();
        if (o < Nout) val = o < i0 + k ? newmass[(int64_t)b * k + (o - i0)] : m[o + r];
        __syncthreads();
        if (o < Nout) m[o] = val;
    }
}

// ---- similarity on the tensor cores --------------------------------------------------------------------
// S = X_dropped X_kept^T, K = channels in chunks of 64.  The operands come from L2 faster than it can deliver them: a
// 128x256 tile a time (48 KB a chunk, 424 cycles of MMAs) asked for 30 TB/s over all SMs and got 14.  So a CTA multiplies
// TWO row tiles of 128 with a column tile of 256 at a time (64 KB for twice the work; the two accumulators fill the
// tensor memory).  The kernel is persistent: an item is two neighbouring row tiles (an odd last one alone) and a column tile, and
// the CTAs take the items in turn, so that those under way at a time share few rows and columns and lie in L2 (SimItems).
// The items of a last round that would leave half of the CTAs idle are cut into single row tiles; where that is all there is, the
// stages of the ring hold single tiles and there is one more of them.
// us, with one row tile a time and two accumulators in turn / every CTA a run of neighbouring tiles, in twos where it fits / so:
// 12288 dropped x 4096 kept rows of 6144 channels 522 / 447 / 405; 16 sequences of 732 x 1060 x 4096 115 / 138 / 106; 4 of 1500 x 1500 x
// 3584 51 / 66 / 48; 1985 x 895 x 3584 25 / 28 / 25; 16 of 500 x 500 x 6144 53 / 69 / 57.
// Warp 0 feeds a ring of shared-memory stages by TMA
// across items, warp 1 issues the MMAs, eight epilogue warps scale the columns by 1/|x_t| and find the best (value, kept index)
// of every row.
constexpr int kSimM = 128, kSimN = 256, kSimK = 64;
constexpr int kSimABytes = kSimM * kSimK * 2, kSimBBytes = kSimN * kSimK * 2;
constexpr int kSimRing = 192 * 1024, kSimMaxStages = 4;                  // 3 stages of two row tiles, or 4 of one
constexpr int kSimCtas = 148, kSimWide = 16;                             // column tiles under way at a time
constexpr int kSimThreads = 320, kSimEpi = 256;
constexpr uint32_t kSimTmemCols = 512;

struct SimArgs {
    int r, k, nkc, nrt, nct;
    int npr, wide;                  // row tiles two at a time; column tiles of a group
    int items, whole;               // whole: items taken as they are; those behind go to two CTAs, a row tile each
    int stages, b_off;              // of the ring; where the column tile lies in a stage
    const float* inv_norm;          // [B][k]
    unsigned long long* best;       // [B][r] (orderable similarity << 32) | ~kept index, zero before
    int32_t* dev_status;
};

struct SimSmem {
    uint64_t full[kSimMaxStages], empty[kSimMaxStages], tmem_full, tmem_empty;
    uint32_t tmem_base;
    volatile int abort;
    float inv_s[2][kSimN];          // 1/|x_t| of the columns, per column half (written by its warps for themselves)
    float xv[2][kSimM];             // upper column half's best, handed to the lower half
    int xt[2][kSimM];
};

// The items of a CTA: every gridDim.x-th.  In order: sequence, group of up to kSimWide column tiles, pair of row tiles, column
// tile of the group.  (148 items at a time: 9 pairs of row tiles x 16 column tiles.)
struct SimItems {
    int i, b, ct, rt, n;
    __device__ SimItems() : i((int)blockIdx.x), n(0) {}
    __device__ bool next(const SimArgs& a) {
        int x = i, part = -1;
        if (x >= a.whole) {
            if (x - a.whole >= 2 * (a.items - a.whole)) return false;
            part = (x - a.whole) & 1;
            x = a.whole + ((x - a.whole) >> 1);
        }
        i += (int)gridDim.x;
        const int per_seq = a.nct * a.npr, per_group = a.wide * a.npr;
        b = x / per_seq; x -= b * per_seq;
        const int first = x / per_group * a.wide, width = min(a.wide, a.nct - first);
        x -= first * a.npr;
        rt = 2 * (x / width);
        ct = first + x % width;
        n = min(2, a.nrt - rt);
        if (part >= 0) {
            if (part >= n) return false;                       // (an odd last row tile; nothing follows the items cut in two)
            rt += part;
            n = 1;
        }
        return true;
    }
};

__device__ __forceinline__ bool sim_wait(uint64_t* bar, uint32_t parity, SimSmem* sm, int32_t* dev_status) {
    if (sm->abort) return false;
    if (mbar_wait(bar, parity)) return true;
    sm->abort = 1;
    if (dev_status) atomicOr(dev_status, LVLM_DEV_TIMEOUT);
    return false;
}

__global__ void __launch_bounds__(kSimThreads, 1)
nk_sim_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap bmap, const SimArgs a) {
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
    SimSmem* sm = reinterpret_cast<SimSmem*>(base + kSimRing);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSimMaxStages; ++s) { mbar_init(&sm->full[s], 1); mbar_init(&sm->empty[s], 1); }
        mbar_init(&sm->tmem_full, 1);
        mbar_init(&sm->tmem_empty, kSimEpi);
        sm->abort = 0;
        fence_barrier_init();
        fence_proxy_async();
        prefetch_tmap(&amap);
        prefetch_tmap(&bmap);
    }
    if (warp == 1) tmem_alloc(&sm->tmem_base, kSimTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sm->tmem_base;
    pdl_enter();

    SimItems w;
    const uint32_t stage_bytes = (uint32_t)(a.b_off + kSimBBytes), stages = (uint32_t)a.stages;
    if (warp == 0) {
        if (lane == 0) {
            uint32_t st = 0, phase = 1;                        // (the first lap finds every stage empty)
            bool ok = true;
            while (ok && w.next(a)) {
                for (int kc = 0; kc < a.nkc; ++kc) {
                    if (!(ok = sim_wait(&sm->empty[st], phase, sm, a.dev_status))) break;
                    unsigned char* dst = base + st * stage_bytes;
                    mbar_arrive_expect_tx(&sm->full[st], (uint32_t)(w.n * kSimABytes + kSimBBytes));
                    for (int i = 0; i < w.n; ++i)
                        tma_load_3d(dst + i * kSimABytes, &amap, &sm->full[st], kc * kSimK, (w.rt + i) * kSimM, w.b);
                    tma_load_3d(dst + a.b_off, &bmap, &sm->full[st], kc * kSimK, w.ct * kSimN, w.b);
                    if (++st == stages) { st = 0; phase ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // all lanes run the loop (uniform operands), one elected lane issues
        constexpr uint32_t idesc = idesc_bf16_f32(kSimM, kSimN);
        const uint64_t d0 = smem_desc_sw128(smem_u32(base));
        uint32_t st = 0, phase = 0, it = 0;
        bool ok = true;
        while (ok && w.next(a)) {
            if (it > 0) ok = __all_sync(0xFFFFFFFFu, sim_wait(&sm->tmem_empty, (it - 1) & 1, sm, a.dev_status));
            for (int kc = 0; ok && kc < a.nkc; ++kc) {
                const uint64_t ad = d0 + st * (stage_bytes >> 4), bd = ad + (uint32_t)(a.b_off >> 4);
                ok = __all_sync(0xFFFFFFFFu, sim_wait(&sm->full[st], phase, sm, a.dev_status));
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        mma_bf16_ss(tmem_base, ad + (uint32_t)(kk * 2), bd + (uint32_t)(kk * 2), idesc, (kc > 0 || kk > 0) ? 1u : 0u);
                    if (w.n == 2) {
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_bf16_ss(tmem_base + kSimN, ad + (uint32_t)((kSimABytes >> 4) + kk * 2), bd + (uint32_t)(kk * 2), idesc,
                                        (kc > 0 || kk > 0) ? 1u : 0u);
                    }
                    mma_commit(&sm->empty[st]);
                    if (kc == a.nkc - 1) mma_commit(&sm->tmem_full);
                }
                __syncwarp();
                if (++st == stages) { st = 0; phase ^= 1u; }
            }
            ++it;
        }
    } else {
        const int quarter = warp & 3, half = (warp - 2) >> 2;
        const int row = quarter * 32 + lane;
        const uint32_t my_tmem = tmem_base + ((uint32_t)(quarter * 32) << 16) + half * 128;
        bool ok = true;
        // (every epilogue thread goes through every item, also after a wait has given up: the barriers count them all)
        for (uint32_t it = 0; w.next(a); ++it) {
            // 1/|x_t| of my half's columns, while the item is being multiplied (the four warps write the same values)
            const int t0 = w.ct * kSimN + half * 128;
            const float* inv = a.inv_norm + (int64_t)w.b * a.k;
            asm volatile("bar.sync 1, 256;" ::: "memory");       // the item before has been read
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int t = t0 + u * 32 + lane;
                sm->inv_s[half][u * 32 + lane] = t < a.k ? __ldg(inv + t) : 0.f;
            }
            __syncwarp();
            ok = __all_sync(0xFFFFFFFFu, ok && sim_wait(&sm->tmem_full, it & 1, sm, a.dev_status));
            float best_v[2] = {-INFINITY, -INFINITY};
            int best_t[2] = {-1, -1};
            if (ok) {
                tc_fence_after();
                // (loops, not straight-line code: a CTA with one item runs through it once, and that is fetched slower than executed)
#pragma unroll 1
                for (int i = 0; i < w.n; ++i) {
                    float bv = -INFINITY, v[2][32];
                    int bt = -1;
                    auto pick = [&](const float* x, int c0) {
                        const float* is = &sm->inv_s[half][c0];
#pragma unroll
                        for (int c = 0; c < 32; ++c) {
                            const float val = x[c] * is[c];
                            if (t0 + c0 + c < a.k && val > bv) { bv = val; bt = t0 + c0 + c; }
                        }
                    };
                    // (a chunk is read while the one before is worked on)
                    const uint32_t from = my_tmem + i * kSimN;
                    tmem_ld32(from, v[0]);
#pragma unroll 1
                    for (int c0 = 0; c0 < 128; c0 += 64) {
                        tmem_ld_wait();
                        tmem_ld32(from + c0 + 32, v[1]);
                        pick(v[0], c0);
                        tmem_ld_wait();
                        if (c0 == 0) tmem_ld32(from + 64, v[0]);
                        pick(v[1], c0 + 32);
                    }
                    if (i == 0) { best_v[0] = bv; best_t[0] = bt; } else { best_v[1] = bv; best_t[1] = bt; }
                }
                tc_fence_before();
            }
            mbar_arrive(&sm->tmem_empty);
            // the two column halves of a row meet in shared memory (on equal similarity the lower kept index
            // wins, whichever half and column tile it sits in)
            if (half == 1) {
#pragma unroll
                for (int i = 0; i < 2; ++i) { sm->xv[i][row] = best_v[i]; sm->xt[i][row] = best_t[i]; }
            }
            asm volatile("bar.sync 1, 256;" ::: "memory");
            if (half == 0 && ok && !sm->abort) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int q = (w.rt + i) * kSimM + row;
                    if (i >= w.n || q >= a.r) continue;
                    const float ov = sm->xv[i][row];
                    const int ot = sm->xt[i][row];
                    if (ot >= 0 && (best_t[i] < 0 || ov > best_v[i])) { best_v[i] = ov; best_t[i] = ot; }
                    if (best_t[i] < 0) continue;
                    uint32_t u = __float_as_uint(best_v[i]);
                    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);         // ascending in the value
                    const unsigned long long key = ((unsigned long long)u << 32) | (0xFFFFFFFFu - (uint32_t)best_t[i]);
                    atomicMax(a.best + (int64_t)w.b * a.r + q, key);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (sm->abort) {
#pragma unroll 1
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kSimTmemCols);
    }
}

template <int CH>
static lvlm_status launch_nk_merge(void* out, int64_t out_sb, const void* scratch, int64_t scr_sb, const lvlm_dims* d,
                                   const NkLayout& L, const int32_t* kept, const int2* order, const int32_t* seg,
                                   const float* mass, float* newmass, cudaStream_t stream) {
    int ctas = (4 * 148) / d->B;
    ctas = ctas < 1 ? 1 : (ctas > d->k ? d->k : ctas);
    return launch_kernel(nk_merge_kernel<CH>, dim3(ctas, d->B), dim3(kNkThreads), 0, stream, 1,
                         static_cast<uint4*>(out), out_sb / 8, static_cast<const uint4*>(scratch), scr_sb / 8, L.V,
                         d->N, d->i0, d->k, L.r, kept, order, seg, mass, newmass);
}

lvlm_status launch_nearest_kept(const void* hidden, void* hidden_out, void* Kc, void* Vc, int32_t* pos_ids,
                                const int32_t* rank, const lvlm_dims* d, float* mass, int32_t* new_len,
                                void* ws, size_t ws_bytes, int32_t* dev_status, cudaStream_t stream) {
    NkLayout L;
    if (!nk_layout(d, &L) || d->k < 1) return LVLM_ERR_INVALID_ARG;
    if (!hidden_out || hidden_out == hidden) return LVLM_ERR_UNSUPPORTED;     // out of place only
    if (L.r > kMaxDropped) return LVLM_ERR_UNSUPPORTED;        // the bitmap of the sort
    if (!ws || !aligned256(ws) || ws_bytes < L.total) return LVLM_ERR_WORKSPACE;
    const int64_t hid_sb = d->hid_stride_b ? d->hid_stride_b : (int64_t)d->N * d->C;
    const int64_t out_sb = d->out_stride_b ? d->out_stride_b : (int64_t)L.Nout * d->C;
    const int64_t kv_sh = d->kv_stride_h ? d->kv_stride_h : (int64_t)d->cap * d->D;
    const int64_t kv_sb = d->kv_stride_b ? d->kv_stride_b : (int64_t)d->Hkv * kv_sh;
    const int64_t scr_sb = (int64_t)L.r * d->C;
    char* wsb = static_cast<char*>(ws);
    int32_t* assign = reinterpret_cast<int32_t*>(wsb + L.off_assign);
    int32_t* dst_map = reinterpret_cast<int32_t*>(wsb + L.off_dst);
    int32_t* kept = reinterpret_cast<int32_t*>(wsb + L.off_kept);
    int32_t* drop = reinterpret_cast<int32_t*>(wsb + L.off_drop);
    float* inv_norm = reinterpret_cast<float*>(wsb + L.off_inv);
    unsigned long long* best = reinterpret_cast<unsigned long long*>(wsb + L.off_best);
    int32_t* place = reinterpret_cast<int32_t*>(wsb + L.off_place);
    int2* order = reinterpret_cast<int2*>(wsb + L.off_order);
    int32_t* seg = reinterpret_cast<int32_t*>(wsb + L.off_seg);
    float* newmass = reinterpret_cast<float*>(wsb + L.off_newmass);
    void* scratch = wsb + L.off_scratch;
    uint4* kvtmp = reinterpret_cast<uint4*>(wsb + L.off_kvtmp);

    lvlm_status st;
    const int plan_threads = d->n >= 1024 ? 1024 : (d->n <= 128 ? 128 : ((d->n + 31) / 32) * 32);
    int P = (d->n + 2047) / 2048;                        // CTAs per sequence: about two tiles of tokens each
    P = P < 1 ? 1 : (P > 8 ? 8 : P);
    st = launch_kernel(nk_plan_kernel, dim3(P, d->B), dim3(plan_threads), 0, stream, P, rank, pos_ids, d->N, d->i0,
                       d->n, d->k, dst_map, kept, drop, best, seg, new_len, dev_status);
    if (st != LVLM_OK) return st;
    st = launch_hidden_rows(hidden, hidden_out, hid_sb, out_sb, d, L.grid, dst_map, nullptr, nullptr, nullptr,
                            scratch, scr_sb, stream, nullptr, dev_status, nullptr, inv_norm);
    if (st != LVLM_OK) return st;
    {
        CUtensorMap amap, bmap;
        const uint64_t adims[3] = {(uint64_t)d->C, (uint64_t)L.r, (uint64_t)d->B};
        const uint64_t astr[2] = {(uint64_t)d->C * 2, (uint64_t)scr_sb * 2};
        const uint32_t abox[3] = {(uint32_t)kSimK, (uint32_t)kSimM, 1};
        if (!make_tmap_bf16(&amap, scratch, 3, adims, astr, abox)) return LVLM_ERR_CUDA;
        const uint64_t bdims[3] = {(uint64_t)d->C, (uint64_t)d->k, (uint64_t)d->B};
        const uint64_t bstr[2] = {(uint64_t)d->C * 2, (uint64_t)out_sb * 2};
        const uint32_t bbox[3] = {(uint32_t)kSimK, (uint32_t)kSimN, 1};
        const void* bbase = static_cast<const char*>(hidden_out) + (int64_t)d->i0 * d->C * 2;
        if (!make_tmap_bf16(&bmap, bbase, 3, bdims, bstr, bbox)) return LVLM_ERR_CUDA;
        SimArgs a;
        a.r = L.r; a.k = d->k; a.nkc = (d->C + kSimK - 1) / kSimK; a.nct = (d->k + kSimN - 1) / kSimN;
        a.nrt = (L.r + kSimM - 1) / kSimM; a.npr = (a.nrt + 1) / 2;
        const int groups = (a.nct + kSimWide - 1) / kSimWide;
        a.wide = (a.nct + groups - 1) / groups;
        const int64_t items = (int64_t)d->B * a.nct * a.npr;
        if (items > 0x3FFFFFFFll) return LVLM_ERR_UNSUPPORTED;
        a.items = (int)items;
        const int rest = a.items % kSimCtas;
        a.whole = 2 * rest <= kSimCtas ? a.items - rest : a.items;
        const bool single = a.whole == 0;                        // (then the grid has two CTAs an item)
        a.stages = single ? 4 : 3; a.b_off = single ? kSimABytes : 2 * kSimABytes;
        const int ctas = single ? 2 * a.items : a.items < kSimCtas ? a.items : kSimCtas;
        a.inv_norm = inv_norm; a.best = best; a.dev_status = dev_status;
        const size_t smem = 1024 + (size_t)kSimRing + sizeof(SimSmem);
        LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(nk_sim_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem));
        st = launch_kernel(nk_sim_kernel, dim3((unsigned)ctas), dim3(kSimThreads), smem, stream, 1, amap, bmap, a);
        if (st != LVLM_OK) return st;
    }
    st = launch_kernel(nk_count_kernel, dim3((L.r + 255) / 256, d->B), dim3(256), 0, stream, 1, best, L.r, d->k, assign, place, seg);
    if (st != LVLM_OK) return st;
    st = launch_kernel(nk_place_kernel, dim3(d->B), dim3(1024), 0, stream, 1, seg, L.r, d->k, assign, place, drop, order);
    if (st != LVLM_OK) return st;
    st = launch_kernel(nk_sort_kernel, dim3((d->k + kSortWarps - 1) / kSortWarps, d->B), dim3(kSortWarps * 32), 0, stream, 1,
                       seg, L.r, d->k, drop, order);
    if (st != LVLM_OK) return st;
    const int chunks = (L.V + kNkThreads - 1) / kNkThreads;
    switch (chunks) {
        case 1: st = launch_nk_merge<1>(hidden_out, out_sb, scratch, scr_sb, d, L, kept, order, seg, mass, newmass, stream); break;
        case 2: st = launch_nk_merge<2>(hidden_out, out_sb, scratch, scr_sb, d, L, kept, order, seg, mass, newmass, stream); break;
        case 3: st = launch_nk_merge<3>(hidden_out, out_sb, scratch, scr_sb, d, L, kept, order, seg, mass, newmass, stream); break;
        case 4: st = launch_nk_merge<4>(hidden_out, out_sb, scratch, scr_sb, d, L, kept, order, seg, mass, newmass, stream); break;
        default: return LVLM_ERR_UNSUPPORTED;
    }
    if (st != LVLM_OK) return st;
    if (Kc) {
        const int rows_out = d->k + L.rest;
        st = launch_kernel(nk_kv_merge_kernel, dim3((rows_out + 15) / 16, (d->Hkv * 2 + kKvSeqs - 1) / kKvSeqs, d->B), dim3(kNkThreads), 0,
                           stream, 1, static_cast<const uint4*>(Kc), static_cast<const uint4*>(Vc), kv_sb / 8, kv_sh / 8, d->Hkv, d->N,
                           d->i0, d->n, d->k, L.r, L.rest, kept, order, seg, mass, kvtmp);
        if (st != LVLM_OK) return st;
        st = launch_kernel(nk_kv_store_kernel, dim3((rows_out * 16 + 4 * kNkThreads - 1) / (4 * kNkThreads), d->Hkv * 2, d->B),
                           dim3(kNkThreads), 0, stream, 1, static_cast<uint4*>(Kc), static_cast<uint4*>(Vc), kv_sb / 8,
                           kv_sh / 8, d->Hkv, d->i0, rows_out, kvtmp);
        if (st != LVLM_OK) return st;
    }
    if (mass)
        return launch_kernel(nk_mass_kernel, dim3(d->B), dim3(1024), 0, stream, 1, mass, d->N, d->i0, d->k, L.r,
                             newmass);
    return LVLM_OK;
}

}  // namespace lvlm
