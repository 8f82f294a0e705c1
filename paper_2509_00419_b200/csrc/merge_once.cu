// lvlm_merge_compact in one launch, for sequences whose rows fit the shared memory of a CTA or a cluster of them.
//
// Everything that moves is cut into columns of 16 P bytes: a K or V sequence is 256 bytes wide, the hidden states 2 C, and a
// CTA (a cluster, each CTA with a run of consecutive input rows) takes a column over the WHOLE sequence.
// The rows are brought on chip while every CTA works out for itself, from `rank`, where its rows go and what they weigh; the
// merged rows are added up; then the CTAs meet in a barrier, and since by then every row of the column is on chip, the kept
// rows can be written where they belong, also in place, and the partial sums of the merged row are there to be added
// in rank order.  So no map goes through memory, every row is read once, and nothing is launched behind it.
//
// What bounds it: latency (a chain of load, barrier, store) up to about 20 MB, then the waves of CTAs.  A thread loads, adds and
// stores the same 16-byte pieces of the same rows, so the rows need no block barrier; a row's weight is worked out once.  us of a
// merge, three launches / this: 640 rows of 2 KB and 8 heads 13.9 / 5.7, 1023 rows of 7 KB and 4 heads 14.9 / 7.3, 3008 rows
// 22.1 / 13.4 (2.6 TB/s), 16 x 264 rows of 8 KB and 8 heads 28.8 / 19.5, 2 x 3064 rows (75 MB) 38.6 / 32.6 (3.3 TB/s).  The position ids are one more, narrow
// column.
#include "common.cuh"
#include "exp2.cuh"
#include "merge.cuh"
#include "sm100.cuh"

namespace lvlm {

constexpr int kOnceThreads = 256, kOnceWarps = kOnceThreads / 32;
constexpr int kOnceMaxCluster = 8;
constexpr int kOnceGroups = 4;                           // the rows of a CTA land in so many groups
constexpr int kOnceMaxSmem = 220 * 1024;
constexpr int kMerged = -1, kFirst = -2;                 // rows that go nowhere

struct OnceArgs {
    const char* hid; char* out; int64_t hid_sb, out_sb;  // bytes
    char* K; char* V; int64_t kv_sb, kv_sh;
    int32_t* pos; const int32_t* rank; const float* w_custom; int32_t* new_len; int32_t* dev_status;
    int N, i0, n, k, C, Hkv, cols, S, R, mode;           // cols: columns of the hidden states; R: rows of a CTA
    float inv_sum;
};


// grid (columns * S, B), clusters of S CTAs along x
template <int P>
__global__ void __launch_bounds__(kOnceThreads) merge_once_kernel(const OnceArgs a) {
    constexpr int kLanes = kOnceThreads / P;                             // rows side by side
    extern __shared__ __align__(16) uint4 rows[];                        // [R][P]
    // [R] output row of a kept row, and nothing; kMerged, or kFirst for the first of the queue, and the weight of a merged row
    int2* s_row = reinterpret_cast<int2*>(rows + (size_t)a.R * P);
    int* s_pos = reinterpret_cast<int*>(rows);                           // [R] position ids (last column, in the place of rows)
    __shared__ __align__(16) float s_red[kOnceWarps][P * 8];
    __shared__ __align__(8) float s_part[P * 8];
    __shared__ __align__(16) uint32_t s_new[P * 4];                      // the merged row
    __shared__ float s_scratch[33];
    __shared__ int s_before[kOnceWarps], s_warp[kOnceWarps];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cg = tid % P, rl = tid / P;
    const int S = a.S, cr = (int)sm100::cluster_ctarank(), col = (int)blockIdx.x / S, b = blockIdx.y;
    const int r1 = a.n - a.k, r = r1 - 1;
    // my column: where its rows come from and go to
    const char* from = nullptr; char* to = nullptr; int64_t row_b = 0; int pieces = P;
    const bool last = col == a.cols + a.Hkv * 2 * (kHeadDim * 2 / (16 * P));     // nothing but position ids and the new length
    if (last) {
        pieces = 0;
    } else if (col < a.cols) {
        row_b = (int64_t)a.C * 2;
        from = a.hid + (int64_t)b * a.hid_sb + col * (16 * P);
        to = a.out + (int64_t)b * a.out_sb + col * (16 * P);
        pieces = min(P, a.C / 8 - col * P);
    } else {
        constexpr int kPer = kHeadDim * 2 / (16 * P);                    // columns of a K or V sequence
        const int x = (col - a.cols) / kPer, part = (col - a.cols) % kPer;
        row_b = kHeadDim * 2;
        to = (x & 1 ? a.V : a.K) + (int64_t)b * a.kv_sb + (int64_t)(x >> 1) * a.kv_sh + part * (16 * P);
        from = to;
    }
    const bool in_place = from == to, with_pos = last && a.pos;
    const int lo = min(a.N, cr * a.R), cnt = min(a.N, lo + a.R) - lo;    // my input rows
    const int32_t* rank = a.rank + (int64_t)b * a.n;
    int32_t* pos = with_pos ? a.pos + (int64_t)b * a.N : nullptr;
    pdl_enter();

    // ---- my rows start their way ------------------------------------------------------------------------
    const int rounds = (cnt + kLanes - 1) / kLanes, quarter = (rounds + kOnceGroups - 1) / kOnceGroups;
    {
        const char* f = from + (int64_t)(lo + rl) * row_b + cg * 16;
        uint32_t d = (uint32_t)__cvta_generic_to_shared(&rows[rl * P + cg]);
        const int64_t step = kLanes * row_b;
        int e = rl;
#pragma unroll
        for (int g = 0; g < kOnceGroups; ++g) {
            const int end = cg < pieces ? min(cnt, (g + 1) * quarter * kLanes) : 0;
#pragma unroll 4
            for (; e < end; e += kLanes, f += step, d += kOnceThreads * 16)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(f) : "memory");
            asm volatile("cp.async.commit_group;\n" ::: "memory");
        }
    }
    // ---- where they go: ranks of my tokens, and how many tokens ahead of mine are kept ---------------------------
    // tokens [ja, jb) are mine; a warp has runs of 32 T consecutive ones
    const int ja = min(max(lo - a.i0, 0), a.n), jb = min(max(lo + cnt - a.i0, 0), a.n);
    const int T = (jb - ja + kOnceThreads - 1) / kOnceThreads, jw = ja + warp * T * 32 + lane;
    int mine = 0, before = 0;
    bool bad = false;
    for (int t0 = 0; t0 < T; t0 += 4) {
        int x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = t0 + u < T && jw + (t0 + u) * 32 < jb ? rank[jw + (t0 + u) * 32] : a.n;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = jw + (t0 + u) * 32;
            if (t0 + u < T && j < jb) {
                s_row[a.i0 + j - lo].x = x[u];                           // (read again by this very thread)
                mine += x[u] < a.k;
                bad |= x[u] < 0 || x[u] >= a.n;
            }
        }
    }
    for (int j0 = tid; j0 < ja; j0 += 8 * kOnceThreads) {
        int x[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = j0 + u * kOnceThreads < ja ? rank[j0 + u * kOnceThreads] : a.n;
#pragma unroll
        for (int u = 0; u < 8; ++u) before += j0 + u * kOnceThreads < ja && x[u] < a.k;
    }
    if (with_pos)
        for (int e = tid; e < cnt; e += kOnceThreads) s_pos[e] = pos[lo + e];
    float inv_sum = a.inv_sum;
    if (a.mode == LVLM_W_CUSTOM) {
        float part = 0.f;
        for (int p = tid; p < r1; p += kOnceThreads) part += a.w_custom[p];
        inv_sum = 1.0f / block_sum_fixed(part, s_scratch);
    }
    before = __reduce_add_sync(0xFFFFFFFFu, before);
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if (lane == 0) { s_before[warp] = before; s_warp[warp] = mine; }
    __syncthreads();
    int off = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kOnceWarps; ++w) {
        off += s_before[w] + (w < warp ? s_warp[w] : 0);
        total += s_before[w] + s_warp[w];
    }
    const unsigned lt = (1u << lane) - 1u;
    for (int t = 0; t < T; ++t) {
        const int j = jw + t * 32, e = a.i0 + j - lo;
        const bool on = j < jb;
        const int x = on ? s_row[e].x : a.n;
        const unsigned kept = __ballot_sync(0xFFFFFFFFu, on && x < a.k);
        if (on) {
            const int o = off + __popc(kept & lt);
            int2 to_w = make_int2(a.i0 + o, 0);
            if (x >= a.k) {
                to_w.x = x == a.k ? kFirst : kMerged;
                to_w.y = __float_as_int(merge_weight(a.mode, min(x - a.k, r1 - 1), r1, inv_sum, a.w_custom));
            } else if (o >= a.k) {
                to_w.x = kMerged;                        // (no permutation: too many)
            }
            s_row[e] = to_w;
        }
        off += __popc(kept);
    }
    for (int e = tid; e < cnt; e += kOnceThreads) {      // rows outside the image span
        const int i = lo + e;
        if (i < a.i0) s_row[e].x = i; else if (i >= a.i0 + a.n) s_row[e].x = i - r;
    }
    if (cr == S - 1 && total != a.k) bad = true;         // (its run ends with the sequence)
    if (bad && last && a.dev_status) atomicOr(a.dev_status, LVLM_DEV_BOUNDS);
    if (last && cr == 0 && tid == 0 && a.new_len) a.new_len[b] = a.N - r;
    __syncthreads();

    // ---- my share of the merged row, as the rows come in -----------------------------------------------------------
    f32x2 acc2[4] = {both(0.f), both(0.f), both(0.f), both(0.f)};
    auto add_group = [&](int g) {
        const int end = cg < pieces ? min(cnt, (g + 1) * quarter * kLanes) : 0;
#pragma unroll 2
        for (int e = g * quarter * kLanes + rl; e < end; e += kLanes) {
            const int2 d = s_row[e];
            if (d.x >= 0) continue;
            const f32x2 w = both(__int_as_float(d.y));
            const uint4 x = rows[e * P + cg];
            acc2[0] = fma2(w, pack2(bf16_lo(x.x), bf16_hi(x.x)), acc2[0]);
            acc2[1] = fma2(w, pack2(bf16_lo(x.y), bf16_hi(x.y)), acc2[1]);
            acc2[2] = fma2(w, pack2(bf16_lo(x.z), bf16_hi(x.z)), acc2[2]);
            acc2[3] = fma2(w, pack2(bf16_lo(x.w), bf16_hi(x.w)), acc2[3]);
        }
    };
    asm volatile("cp.async.wait_group 3;\n" ::: "memory"); add_group(0);
    asm volatile("cp.async.wait_group 2;\n" ::: "memory"); add_group(1);
    asm volatile("cp.async.wait_group 1;\n" ::: "memory"); add_group(2);
    asm volatile("cp.async.wait_group 0;\n" ::: "memory"); add_group(3);
    float acc[8];
#pragma unroll
    for (int u = 0; u < 4; ++u) unpack2(acc2[u], acc[2 * u], acc[2 * u + 1]);
#pragma unroll
    for (int o = 16; o >= P; o >>= 1)
#pragma unroll
        for (int u = 0; u < 8; ++u) acc[u] += __shfl_xor_sync(0xFFFFFFFFu, acc[u], o);
    if (lane < P) {
        *reinterpret_cast<float4*>(&s_red[warp][cg * 8]) = make_float4(acc[0], acc[1], acc[2], acc[3]);
        *reinterpret_cast<float4*>(&s_red[warp][cg * 8 + 4]) = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    __syncthreads();
    if (tid < P * 8) {
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < kOnceWarps; ++w) s += s_red[w][tid];
        s_part[tid] = s;
    }
    // ---- every row of the column is on chip, every share is there ----------------------------------------------
    if (S > 1) {
        sm100::cluster_barrier();
    } else {
        __syncthreads();
    }
    if (cr == 0 && tid < pieces * 4) {                   // the merged row: two channels a thread
        float x = 0.f, y = 0.f;
#pragma unroll
        for (int q = 0; q < kOnceMaxCluster; ++q) {
            if (q < S) {
                const float2 v = sm100::cluster_ld(reinterpret_cast<const float2*>(s_part) + tid, q);
                x += v.x; y += v.y;
            }
        }
        s_new[tid] = pack_bf16(x, y);
    }
    // The shares have been read: their sums lie in shared memory before the warp comes together to arrive.  (An arrival with release
    // semantics says the same and waits for a fence: 1023 rows of 7 KB 7.4 -> 8.1 us; shares sent to the first CTA ahead of the barrier
    // need no second one, but make everybody wait for the sending: 4500 rows of 12 KB 36.5 -> 38.3.)
    if (S > 1) sm100::cluster_arrive_exec(); else __syncwarp();
    if (cr == 0 && lane < 8 && warp * 8 + lane < pieces)
        *reinterpret_cast<uint4*>(to + (int64_t)(a.i0 + a.k) * row_b + (warp * 8 + lane) * 16) = reinterpret_cast<const uint4*>(s_new)[warp * 8 + lane];
    if (cg < pieces) {
#pragma unroll 4
        for (int e = rl; e < cnt; e += kLanes) {
            const int d = s_row[e].x;
            if (d >= 0 && !(in_place && d == lo + e)) *reinterpret_cast<uint4*>(to + (int64_t)d * row_b + cg * 16) = rows[e * P + cg];
        }
    }
    if (with_pos) {                                      // P_new takes the id of the first of the queue
        for (int e = tid; e < cnt; e += kOnceThreads) {
            const int d = s_row[e].x;
            if (d != kMerged) pos[d == kFirst ? a.i0 + a.k : d] = s_pos[e];
        }
    }
    if (S > 1) sm100::cluster_wait();                    // nobody leaves while its share is still read
}

static size_t once_smem(int P, int R) { return (size_t)R * (16 * P + 8); }
static int once_rows(int N, int S) { return ((N + S - 1) / S + 3) & ~3; }

// Estimate of the time in us by column width and cluster size, a fit (within 10 %) to 400 measurements of 68 sizes
// (1 to 16 sequences of 214 to 9064 rows, 1024 to 6144 channels, 4 or 8 KV heads).  A wave of CTAs takes a latency and
// what its SM moves, at a lower rate where an SM has one CTA only; a CTA goes through its tokens; clusters meet, and fewer of them
// find room.  What decides: one wave where all rows fit the chip at all (up to about 27 MB), two CTAs an SM rather than one
// (3008 rows of 7 KB and 4 heads, 64-byte columns in clusters of two 13.9 us, 128-byte ones 16.4, 256-byte ones in clusters of eight
// 20.7), beyond that small CTAs in many waves (8 KB and 8 heads, 5564 rows, 50 KB a CTA 35.4, 100 KB 44.6).
// 16-byte pieces 4 << p, CTAs 1 << c, for two numbers of heads at a time: twelve of these are a tenth of a microsecond of every call.
static void once_estimate(const lvlm_dims* d, const int (&heads)[2], int p, int c, double (&t)[2]) {
    static const double kInvCtas[5] = {0.0, 1.0 / 148, 1.0 / 296, 1.0 / 444, 1.0 / 592}, kLast[5] = {0.0, 1.1, 0.55, 1.1 / 3, 0.275};
    static const double kFewer[4] = {1.0, 1.0, 1.0 / 0.91, 1.0 / 0.95};
    const int P = 4 << p, S = 1 << c, R = once_rows(d->N, S);
    const int smem = (int)once_smem(P, R);
    t[0] = t[1] = 1e30;
    if (smem > kOnceMaxSmem) return;
    int per_sm = 227 * 1024 / (smem + 1024 + 512 + 288 * P);
    per_sm = per_sm > 4 ? 4 : per_sm;
    const double kb = R * P * (1.0 / 64), fixed = 0.9 + 0.0019 * d->n / S + (S > 1 ? 1.8 : 0.0);
    for (int h = 0; h < 2; ++h) {
        const int ctas = d->B * (((d->C / 8 + P - 1) >> (p + 2)) + 2 * heads[h] * (4 >> p) + 1) * S;
        const double full = ctas * kInvCtas[per_sm] * kFewer[c], waves = full <= 1 ? 1.0 : full + kLast[per_sm];
        const int here = ctas >= 148 * per_sm ? per_sm : (ctas + 147) / 148;
        t[h] = fixed + waves * (2.5 + kb * (here > 1 ? here * 0.039 : 0.0464));
    }
}

// Neither the path nor the column width and the cluster size may follow K and V: the merged row of the hidden states is added in an
// order that these decide, and it should be the same bits whether a call brings K and V, and however many heads of them.  So
// both rules see batch, rows and channels alone, and take K and V for what GQA models have: 3500 bytes a row for the path; for width and
// size 8 heads up to 2048 channels and 4 beyond, or, where that leaves two choices close, the one that the other number prefers.  By
// the estimate that costs 0 to 0.2 % on average against a choice that knows the heads (1024 to 6144 channels, 4 or 8 of them), 3 %
// with 32 heads or without K and V.
//
// The launches of the general path (plan, row pass, compaction) take over where they are quicker.  us so / here: 2 x 3064 rows of 8 KB and
// 8 heads 38.0 / 36.6, 2 x 3300 39.8 / 43.7; 2 x 3600 of 7 KB and 4 heads 33.9 / 36.9; 4500 of 12 KB and 8 heads 39.0 / 36.5; 2 x 5900 of
// 2 KB and 8 heads 44.2 / 38.4, 3 x 4500 43.1 / 42.8, 3 x 4900 45.4 / 49.2; 9064 rows of 7 KB and 4 heads 39.7 / 59.0.  Short sequences, in
// many small CTAs, gain longer: 16 x 560 of 8 KB and 8 heads 45.6 / 41.7, 16 x 400 of 12 KB 47.2 / 44.8, 16 x 640 of 7 KB and 4 heads 38.5 /
// 37.4.  With 32 heads of 8 KB: 3008 rows 43.1 / 35.6, 2 x 3000 66.2 / 64.5, 5900 67.9 / 70.2.
OnceShape merge_once_shape(const lvlm_dims* d) {
    OnceShape s = {0, 0};
    const double mb = (double)d->B * d->N * (d->C * 2.0 + 3500.0) * 1e-6;
    if (d->N > 6000 || mb > (d->N <= 800 ? 110.0 : 73.0)) return s;
    const int heads[2] = {d->C <= 2048 ? 8 : 4, d->C <= 2048 ? 4 : 8};
    double t[3][4][2], least[2] = {1e29, 1e29};          // [log2 P - 2][log2 S][heads]
    for (int p = 0; p < 3; ++p)
        for (int c = 0; c < 4; ++c) {
            once_estimate(d, heads, p, c, t[p][c]);
            for (int h = 0; h < 2; ++h) least[h] = t[p][c][h] < least[h] ? t[p][c][h] : least[h];
        }
    const double other = 0.1 * least[0] / least[1];
    double best = 1e29;
    for (int p = 2; p >= 0; --p)
        for (int c = 0; c < 4; ++c) {
            const double x = t[p][c][0] + other * t[p][c][1];
            if (x < best) { best = x; s.P = 4 << p; s.S = 1 << c; }
        }
    return s;
}

template <int P>
static lvlm_status launch_once(OnceArgs& a, int B, cudaStream_t stream) {
    a.cols = (a.C / 8 + P - 1) / P;
    const int64_t x = (int64_t)(a.cols + 2 * a.Hkv * (16 / P) + 1) * a.S;
    LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(merge_once_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, kOnceMaxSmem));
    return launch_kernel(merge_once_kernel<P>, dim3((unsigned)x, (unsigned)B), dim3(kOnceThreads), once_smem(P, a.R), stream, a.S, a);
}

lvlm_status launch_merge_once(const MergeOnce& m, const lvlm_dims* d, OnceShape s, cudaStream_t stream) {
    OnceArgs a;
    a.hid = static_cast<const char*>(m.hidden);
    a.out = static_cast<char*>(m.hidden_out ? m.hidden_out : m.hidden);
    a.hid_sb = m.hid_sb * 2; a.out_sb = m.out_sb * 2;
    a.K = static_cast<char*>(m.K); a.V = static_cast<char*>(m.V); a.kv_sb = m.kv_sb * 2; a.kv_sh = m.kv_sh * 2;
    a.pos = m.pos_ids; a.rank = m.rank; a.w_custom = m.w_custom; a.new_len = m.new_len; a.dev_status = m.dev_status;
    a.N = d->N; a.i0 = d->i0; a.n = d->n; a.k = d->k; a.C = d->C; a.Hkv = m.K ? d->Hkv : 0;
    a.S = s.S; a.R = once_rows(d->N, s.S); a.mode = m.mode; a.inv_sum = m.inv_sum;
    switch (s.P) {
        case 4: return launch_once<4>(a, d->B, stream);
        case 8: return launch_once<8>(a, d->B, stream);
        case 16: return launch_once<16>(a, d->B, stream);
    }
    return LVLM_ERR_UNSUPPORTED;
}

}  // namespace lvlm
