// Tensor-core scoring kernels (tcgen05 + TMEM + TMA) for lvlm_score_tokens, where score_once.cu does not do it in one pass.
//
// The score of an image key is a column sum of softmax probabilities (Section 3.2.1,
// paragraph 3), so two passes over Q K^T are needed when the caller has no row normalisers:
//   pass 1 (MODE 0)  S = Q_tile K_tile^T with QUERIES on the TMEM lanes: every epilogue thread owns
//                    one query row and keeps its running max / sum over the key tiles -> normaliser.
//   pass 2 (MODE 1)  S^T = K_tile Q_tile^T with KEYS on the TMEM lanes: every epilogue thread owns
//                    one image key and adds exp2(logit - normaliser[row]) over the query rows of the
//                    heads of the KV group -> group-summed column sums.
// A query tile is 128 positions of one head or, where that wastes fewer rows (a short text window), as many positions
// as fit times all heads of the KV group.  Both orientations are plain K-major operands (D is contiguous in Q and in K),
// so the same pipeline serves both.
//
// What bounds it: one exponential per logit and pass, 1024 cycles of the special-function unit per 128x128 tile against
// 512 of the tensor pipe.  What the epilogue lost beside them, and the answer to each: start-up and drain of a CTA per
// tile or two (the kernel is persistent, a CTA walks over work items, and the roles run ahead of one another ACROSS
// items: a TMA warp through rings of A and B tiles, two MMA-issuing warps through four TMEM accumulators, four sets of
// four epilogue warps, each with an accumulator of its own, and a finisher warp that adds what they left of an item in
// shared memory and parks it in the workspace); operand traffic (an item multiplies TWO A tiles with a run of B tiles, or,
// where the query tiles of a KV group are few, keeps them as B tiles over the items that follow); waiting for
// normalisers (they come with the tile, by bulk copy) and reading one of them per logit (a TMEM load layout in which
// a pair of them serves four keys); rows that a query tile does not have.
// us a call, with a CTA per tile or two / so: all rows of 8448 x 48 heads, pass 2: 1095 / 521, both: 1643 / 1011; 22 layers of
// 3008 keys x 28 heads x 128 rows, pass 2: 135 / 90, both: 214 / 178; 16 sequences of 1888 keys x 32 heads x 96 rows, both:
// 114 / 80; 32933 keys x 28 heads x 131 rows, both: 177 / 100; 640 keys x 8 heads x 64 rows: 12.8 / 13.0 (start-up and
// hand-overs).  Of a tile's 1300 to 2000 cycles the special-function unit is busy for 1024; a polynomial on the FMA pipe for
// a quarter of the exponentials made it 2 to 6 % slower.
// Small launches add the parked sums: normalisers (large shape, where items share a query tile's keys), scores.
#include <type_traits>

#include "common.cuh"
#include "exp2.cuh"
#include "score.cuh"
#include "sm100.cuh"

namespace lvlm {

using namespace sm100;

constexpr int kTile = 128;                 // rows of A, rows of B, and K (= head dim)
constexpr int kHalfBytes = kTile * 64 * 2; // one TMA box: 128 rows x 64 bf16 = 16 KB
constexpr int kTileBytes = 2 * kHalfBytes; // 32 KB
constexpr int kSmCount = 148;
constexpr int kMaxKeep = 4;                // B tiles kept over items at most (two of the six slots are left for A tiles)

// Two shapes of the kernel.  Large: one CTA per SM, everything above.  Small: for calls whose items are few and short,
// where start-up, hand-overs and launches are the time - two CTAs per SM fit side by side, so that the next kernel's CTAs
// set themselves up while this one's still run (programmatic dependent launch); an item has one A tile, one warp
// issues the MMAs, and the other one works the normalisers out of what pass 1 (or the caller) left, which saves a launch.
template <bool SMALL>
struct ScoreCfg {
    static constexpr int kSlots = SMALL ? 3 : 6;           // tiles in shared memory, A and B together
    static constexpr int kAccs = SMALL ? 2 : 4;            // 128-column fp32 accumulators in TMEM
    static constexpr int kSets = kAccs;                    // sets of four epilogue warps, one for each accumulator
    static constexpr int kItemTiles = SMALL ? 1 : 2;       // A tiles of an item
    static constexpr int kIssuers = SMALL ? 1 : 2;         // warps that issue MMAs
    static constexpr int kEpiWarps = 4 * kSets;
    static constexpr int kThreads = (4 + kEpiWarps) * 32;  // warp 0 TMA, 1 (and 3) MMA, 2 finisher, (3 normalisers,) then the epilogue
    static constexpr int kCtas = SMALL ? 2 : 1;            // per SM
    // Normalisers of the last B tiles.  An epilogue set reads those of a tile after its accumulator is free, so their slots
    // outlive the B tile's: when tile c + kNlse is fetched, the MMAs of tile c + kNlse - (B slots) + 1 or so are done, those
    // needed the accumulators of tiles kAccs earlier (two A tiles: half as many) back, and the sets take their tiles in
    // order - whoever read tile c has gone on.
    // (Small shape: the set says so itself.)
    static constexpr int kNlse = SMALL ? 4 : 16;
};
constexpr int kFirstEpiWarp = 4;
// Small shape up to so many 128x128 tiles of a pass, measured with either shape forced: pass 1 as large / small, us of a
// call: 672 tiles (4 KV heads of 7, 3008 keys, 128 rows) 27.2 / 28.7, 924 32.0 / 35.5, 512 26.2 / 29.8, 476 25.1 / 25.3, 256
// 27.7 / 20.5, 40 13.9 / 13.0; pass 2: 1136 tiles 16.9 / 16.4, 896 14.8 / 14.4, 512 14.9 / 12.8, 40 11.8 / 8.2.
constexpr int64_t kSmallTiles1 = 148 * 3, kSmallTiles2 = 148 * 8;
// Most parts of an item, and tiles of 128 results of them in the workspace: 4 MB either way.  The second figures bind where
// there are thousands of items anyhow (an 8 x 48-head window of 5000 rows: five parts instead of six).
constexpr int kMaxSplit = 32, kMaxParts = 16;
constexpr int64_t kMaxStatTiles = 4096, kMaxPartTiles = 8192;
constexpr float kLog2eT = 1.4426950408889634f;

struct ScoreTcArgs {
    int B, H, G, Hkv, N, Nq, i0, n, q_lo, causal;
    ScoreShape s;
    FastDiv by_split, by_hkv, by_b, by_nh, by_box_h, by_box_p;     // by_split: ksplit or parts
    int items, a_slots, keep;
    int from_stat;             // small shape, pass 2: the normalisers come from stat (else, lse given: from lse, times lse_scale)
    const float* lse; float lse_scale;
    float scale_log2;
    float* nlse;               // [B * Hkv * tpg][128] minus the log2-domain normalisers, query tile by query tile; -inf: no row
    float2* stat;              // [B * Hkv * tpg][ksplit][128] (max, sum) of the keys of an item (pass 1, ksplit > 1)
    float* partial;            // [B][Hkv * parts][nkt * 128] column sums of every item (pass 2)
    int32_t* dev_status;
};

struct TcCtl {                                     // what the roles wait on
    uint64_t a_full[6], a_empty[6], b_full[6], b_empty[6], tmem_full[4], tmem_empty[4], nlse_full[16], nlse_empty[4], res_full[2], res_empty[2];
    uint32_t tmem_base;
    volatile int abort;
};
template <bool SMALL>
struct TcSmem : TcCtl {
    alignas(16) float nlse[ScoreCfg<SMALL>::kNlse][kTile];          // the normalisers of the B tiles (pass 2)
    alignas(16) float2 res[2][ScoreCfg<SMALL>::kSets][kTile];       // what the sets leave of an item: (column sum, -) or (max, sum)
};

// Pass 1, one chunk of 32 raw logits of a query row: columns [0, lim) are visible.  Updates the running
// (max, sum of 2^(logit*scale - max)).
__device__ __forceinline__ void rowstat_chunk(float* v, int lim, float scale_log2, float& m_run, float& l_run) {
    if (lim < 32) {
#pragma unroll
        for (int c = 0; c < 32; ++c) v[c] = c < lim ? v[c] : -INFINITY;
    }
    // the maximum of the scaled logits is that of the raw ones scaled (of the smallest for a negative scale)
    float c0, c1, c2, c3;
    if (scale_log2 > 0.f) {
        c0 = v[0]; c1 = v[1]; c2 = v[2]; c3 = v[3];
#pragma unroll
        for (int c = 4; c < 32; c += 4) { c0 = fmaxf(c0, v[c]); c1 = fmaxf(c1, v[c + 1]); c2 = fmaxf(c2, v[c + 2]); c3 = fmaxf(c3, v[c + 3]); }
    } else {
#pragma unroll
        for (int c = 0; c < 32; ++c) v[c] = c < lim ? v[c] * scale_log2 : -INFINITY;
        scale_log2 = 1.f;
        c0 = c1 = c2 = c3 = v[0];
#pragma unroll
        for (int c = 1; c < 32; ++c) c0 = fmaxf(c0, v[c]);
    }
    const float m_new = fmaxf(m_run, fmaxf(fmaxf(c0, c1), fmaxf(c2, c3)) * scale_log2);
    if (m_new == -INFINITY) return;                        // nothing visible yet
    const f32x2 sc = both(scale_log2), mm = both(-m_new);
    f32x2 a0 = both(0.f), a1 = both(0.f);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const f32x2 x = fma2(pack2(v[2 * i], v[2 * i + 1]), sc, mm);
        float x0, x1;
        unpack2(x, x0, x1);
        const f32x2 e = pack2(ex2_fast(x0), ex2_fast(x1));
        if (i & 1) a1 = add2(a1, e); else a0 = add2(a0, e);
    }
    float s0, s1;
    unpack2(add2(a0, a1), s0, s1);
    l_run = l_run * ex2_fast(m_run - m_new) + (s0 + s1);
    m_run = m_new;
}

// Pass 2, 32 raw logits of a thread: four keys (rows r, r+8 of the upper and of the lower 16 TMEM lanes) against four
// pairs of neighbouring query rows (columns 8 i + 2 (lane % 4) of the chunk), as tcgen05.ld.16x256b hands them out.
// nls: (minus) the normalisers of my first pair (log2 domain), 8 floats apart.  The layout is taken because a pair of
// normalisers read from shared memory serves four keys: with a whole TMEM lane a thread every logit needs a normaliser
// of its own, and those broadcast reads took as much of shared memory's bandwidth as the MMAs' operands.
// acc[k] += the probabilities of key k; only those of columns >= first[k] when MASK.
template <bool MASK>
__device__ __forceinline__ void colsum_chunk(const float* v, const float* nls, const int* first, int col0, float scale_log2,
                                             f32x2* acc) {
    const f32x2 sc = both(scale_log2);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const f32x2 n2 = *reinterpret_cast<const f32x2*>(nls + 8 * i);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // registers: [upper or lower 16 lanes][8-column group][row, row + 8][pair]
            const float* e = v + (k >> 1) * 16 + i * 4 + (k & 1) * 2;
            const f32x2 x = fma2(pack2(e[0], e[1]), sc, n2);
            float x0, x1;
            unpack2(x, x0, x1);
            x0 = ex2_fast(x0); x1 = ex2_fast(x1);
            if (MASK) { x0 = col0 + 8 * i >= first[k] ? x0 : 0.f; x1 = col0 + 8 * i + 1 >= first[k] ? x1 : 0.f; }
            acc[k] = add2(acc[k], pack2(x0, x1));
        }
    }
}

__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, TcCtl* sm, int32_t* dev_status) {
    if (mbar_try(bar, parity)) return true;                // (nobody stops for the abort flag while the phases complete)
    if (sm->abort) return false;
    if (mbar_wait(bar, parity)) return true;
    sm->abort = 1;
    if (dev_status) atomicOr(dev_status, LVLM_DEV_TIMEOUT);
    return false;
}

// A work item: one or two A tiles and a run of B tiles.
struct ScoreItem {
    int b, g, part;            // part: of the keys of the query tiles (pass 1), of the query tiles of the key tiles (pass 2)
    int at, na;                // first A tile (query tile of the group, or key tile) and their number
    int t0, nt;                // pass 1: key tiles t0..; pass 2: visible query tiles t0.. of the group
    int v0;                    // pass 2: the first query tile of the group that sees a key of the A tiles
};

// Query tiles of a KV group are numbered position tile by position tile, the heads of one inside it.
struct QTile {
    int hb, pt;
    __device__ QTile(const ScoreTcArgs& a, int i) { pt = a.by_nh.divmod(i, &hb); }
    __device__ void step(const ScoreTcArgs& a, int n) { for (hb += n; hb >= a.s.nh; hb -= a.s.nh) ++pt; }
};

// The items of this CTA: they go round the CTAs in turn, there and back, longest first; with kept B tiles a CTA takes
// consecutive ones instead (the key tiles of a KV group follow one another).
template <int MODE, bool SMALL>
struct ScoreItems {
    static constexpr int kPer = ScoreCfg<SMALL>::kItemTiles;
    const ScoreTcArgs& a;
    int i, end, round;
    __device__ explicit ScoreItems(const ScoreTcArgs& a_) : a(a_), i((int)blockIdx.x), end(a_.items), round(0) {
        if (MODE == 1 && a.keep) {
            i = (int)((int64_t)a.items * blockIdx.x / gridDim.x);
            end = (int)((int64_t)a.items * (blockIdx.x + 1) / gridDim.x);
        }
    }
    __device__ bool next(ScoreItem* w) {
        const bool first = round++ == 0;
        if (i >= end) return false;
        if (MODE == 1 && a.keep && !first && w->at + kPer < a.s.nkt) {      // the next key tiles of the same group
            w->at += kPer;
            w->na = min(kPer, a.s.nkt - w->at);
            ++i;
            return true;
        }
        int x = i;
        if (MODE == 0) {
            x = a.by_split.divmod(x, &w->part);
            x = a.by_hkv.divmod(x, &w->g);
            x = a.by_b.divmod(x, &w->b);
            w->at = max(0, a.s.tpg - kPer * (x + 1));                       // late positions see most keys
            w->na = a.s.tpg - kPer * x - w->at;
            const int last = min(a.Nq, (QTile(a, w->at + w->na - 1).pt + 1) * a.s.box_p);
            const int nt_all = ((a.causal ? min(a.N, a.q_lo + last) : a.N) + kTile - 1) / kTile;
            w->t0 = a.by_split.div(nt_all * w->part);
            w->nt = a.by_split.div(nt_all * (w->part + 1)) - w->t0;
            w->v0 = 0;
        } else {
            if (a.keep) {
                const int per_group = (a.s.nkt + kPer - 1) / kPer;
                w->at = kPer * (x % per_group); x /= per_group;
                x = a.by_split.divmod(x, &w->part);
                w->b = a.by_hkv.divmod(x, &w->g);
            } else {
                x = a.by_split.divmod(x, &w->part);
                x = a.by_hkv.divmod(x, &w->g);
                x = a.by_b.divmod(x, &w->b);
                w->at = kPer * x;                                           // early keys are seen most
            }
            w->na = min(kPer, a.s.nkt - w->at);
            const int j0 = a.i0 + w->at * kTile;
            const int pt_min = a.causal && j0 > a.q_lo ? min(a.by_box_p.div(j0 - a.q_lo), a.s.npt) : 0;
            w->v0 = pt_min * a.s.nh;
            const int all = a.s.tpg - w->v0;
            w->t0 = a.by_split.div(all * w->part);
            w->nt = a.by_split.div(all * (w->part + 1)) - w->t0;
        }
        if (MODE == 1 && a.keep) ++i;
        else i = round * (int)gridDim.x + ((round & 1) ? (int)gridDim.x - 1 - (int)blockIdx.x : (int)blockIdx.x);
        return true;
    }
};

// Minus the normaliser of row r of query tile `qt` of a group, from its (max, sum); -inf where the tile has no such row.
__device__ __forceinline__ float minus_normaliser(const ScoreTcArgs& a, int qt, int r, float M, float Ls) {
    const int p = a.by_box_h.div(r);
    if (p >= a.s.box_p || QTile(a, qt).pt * a.s.box_p + p >= a.Nq) return -INFINITY;
    return -(M + log2f(Ls));
}

// (max, sum) M, Ls and m, l of two sets of keys added.
__device__ __forceinline__ void add_stat(float& M, float& Ls, float m, float l) {
    const float m_new = fmaxf(M, m);
    if (m_new > -INFINITY) { Ls = Ls * exp2f(M - m_new) + l * exp2f(m - m_new); M = m_new; }
}

// The (max, sum) of every `step`-th item of a query tile from `first` on, added in key order, for four rows from `r` on.
// DEEP items' loads are in flight at a time.
template <int DEEP>
__device__ __forceinline__ void add_stats(const ScoreTcArgs& a, int64_t tile, int r, int first, int step, float* M, float* Ls) {
    const float2* st = a.stat + tile * a.s.ksplit * kTile + r;
#pragma unroll
    for (int u = 0; u < 4; ++u) { M[u] = -INFINITY; Ls[u] = 0.f; }
    for (int k0 = first; k0 < a.s.ksplit; k0 += DEEP * step) {
        float4 v[DEEP][2];
#pragma unroll
        for (int k = 0; k < DEEP; ++k) {
            v[k][0] = v[k][1] = make_float4(-INFINITY, 0.f, -INFINITY, 0.f);
            if (k0 + k * step < a.s.ksplit) {
                const float4* x = reinterpret_cast<const float4*>(st + (int64_t)(k0 + k * step) * kTile);
                v[k][0] = __ldcg(x); v[k][1] = __ldcg(x + 1);
            }
        }
#pragma unroll
        for (int k = 0; k < DEEP; ++k) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float4& x = v[k][u >> 1];
                add_stat(M[u], Ls[u], (u & 1) ? x.z : x.x, (u & 1) ? x.w : x.y);
            }
        }
    }
}

// Minus the normalisers of four rows of a query tile from all its items.
template <int DEEP>
__device__ __forceinline__ void norm_of_stat(const ScoreTcArgs& a, int64_t tile, int r, float* out) {
    float M[4], Ls[4];
    add_stats<DEEP>(a, tile, r, 0, 1, M, Ls);
    const int qt = (int)(tile % a.s.tpg);
#pragma unroll
    for (int u = 0; u < 4; ++u) out[u] = minus_normaliser(a, qt, r + u, M[u], Ls[u]);
}

// The same from normalisers somebody else computed, [B][H][Nq], times lse_scale.
__device__ __forceinline__ void norm_of_lse(const ScoreTcArgs& a, int64_t tile, int r0, float* out) {
    const int bg = (int)(tile / a.s.tpg), b = bg / a.Hkv, g = bg - b * a.Hkv;
    const QTile q(a, (int)(tile - (int64_t)bg * a.s.tpg));
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int r = r0 + u, p = a.by_box_h.div(r), pos = q.pt * a.s.box_p + p, h = g * a.G + q.hb * a.s.box_h + r - p * a.s.box_h;
        out[u] = p < a.s.box_p && pos < a.Nq ? __ldcg(a.lse + ((int64_t)b * a.H + h) * a.Nq + pos) * a.lse_scale : -INFINITY;
    }
}

// Slot and phase of a ring.
struct RingPos {
    uint32_t slot = 0, phase = 0;
    bool lapped = false;                                   // somebody has to have emptied the slot before it is filled again
    __device__ void next(uint32_t n) { if (++slot == n) { slot = 0; phase ^= 1u; lapped = true; } }
};

template <int MODE, bool SMALL>
__global__ void __launch_bounds__(ScoreCfg<SMALL>::kThreads, ScoreCfg<SMALL>::kCtas)
score_tc_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                const ScoreTcArgs a) {
    using Cfg = ScoreCfg<SMALL>;
    constexpr int kSlots = Cfg::kSlots, kAccs = Cfg::kAccs, kSets = Cfg::kSets, kNlse = Cfg::kNlse, kThreads = Cfg::kThreads;
    constexpr uint32_t kTmemCols = kAccs * kTile;
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
    const uint32_t a_slots = (uint32_t)a.a_slots, b_slots = kSlots - a_slots;
    unsigned char* sA = base;                              // [a_slots]
    unsigned char* sB = base + a_slots * kTileBytes;       // [b_slots]
    TcSmem<SMALL>* sm = reinterpret_cast<TcSmem<SMALL>*>(base + kTileBytes * kSlots);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int box_rows = a.s.box_h * a.s.box_p;            // rows of a query tile the TMA copy writes

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlots; ++s) {
            mbar_init(&sm->a_full[s], 1); mbar_init(&sm->a_empty[s], Cfg::kIssuers);
            mbar_init(&sm->b_full[s], 1); mbar_init(&sm->b_empty[s], Cfg::kIssuers);
        }
        for (int s = 0; s < kNlse; ++s) { mbar_init(&sm->nlse_full[s], 1); if (SMALL) mbar_init(&sm->nlse_empty[s], 4); }
        for (int s = 0; s < 2; ++s) { mbar_init(&sm->res_full[s], Cfg::kEpiWarps); mbar_init(&sm->res_empty[s], 1); }
        for (int s = 0; s < kAccs; ++s) { mbar_init(&sm->tmem_full[s], 1); mbar_init(&sm->tmem_empty[s], 4); }
        sm->abort = 0;
        fence_barrier_init();
        prefetch_tmap(&qmap);
        prefetch_tmap(&kmap);
    }
    // rows of a query tile that no copy ever writes: their logits are thrown away, but have to be numbers
    const int copies = MODE == 0 ? a.s.copies : 1, row_step = kTile / copies;     // pass 1: the rows of a query tile, so many times
    if (box_rows < row_step) {
        for (int e = threadIdx.x; e < kTile * 8 * kSlots * 2; e += kThreads) {
            const int x = e / (kSlots * 2), r = x >> 3;
            if ((r & (row_step - 1)) >= box_rows)
                *reinterpret_cast<uint4*>(base + (e - x * (kSlots * 2)) * kHalfBytes + r * 128 + (x & 7) * 16) = make_uint4(0, 0, 0, 0);
        }
    }
    fence_proxy_async();
    if (warp == 1) tmem_alloc(&sm->tmem_base, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sm->tmem_base;
    pdl_enter();                               // barriers and tensor memory are set up; now the inputs

    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            const uint32_t q_bytes = (uint32_t)box_rows * 256;
            auto load_q = [&](unsigned char* dst, uint64_t* bar, const ScoreItem& w, const QTile& q) {
                const int hh = w.g * a.G + q.hb * a.s.box_h, pos = q.pt * a.s.box_p;
                tma_load_4d(dst, &qmap, bar, 0, hh, pos, w.b);
                tma_load_4d(dst + kHalfBytes, &qmap, bar, 64, hh, pos, w.b);
            };
            auto load_k = [&](unsigned char* dst, uint64_t* bar, const ScoreItem& w, int row) {
                mbar_arrive_expect_tx(bar, kTileBytes);
                tma_load_4d(dst, &kmap, bar, 0, row, w.g, w.b);
                tma_load_4d(dst + kHalfBytes, &kmap, bar, 64, row, w.g, w.b);
            };
            RingPos ra, rb;
            ScoreItem w;
            int held = -1;                                               // kept B tiles: whose they are
            uint32_t nb = 0;                                             // B tiles fetched so far
            bool ok = true;
            ScoreItems<MODE, SMALL> items(a);
            while (ok && items.next(&w)) {
                if (w.nt == 0) continue;                                  // (its A tiles are not even fetched)
                for (int i = 0; ok && i < w.na; ++i, ra.next(a_slots)) {
                    if (ra.lapped) ok = wait_or_abort(&sm->a_empty[ra.slot], ra.phase ^ 1u, sm, a.dev_status);
                    if (!ok) break;
                    unsigned char* dst = sA + ra.slot * kTileBytes;
                    if (MODE == 0) {
                        const QTile q(a, w.at + i);
                        mbar_arrive_expect_tx(&sm->a_full[ra.slot], q_bytes * (uint32_t)a.s.copies);
                        for (int c = 0; c < a.s.copies; ++c) load_q(dst + c * (kHalfBytes / a.s.copies), &sm->a_full[ra.slot], w, q);
                    }
                    else load_k(dst, &sm->a_full[ra.slot], w, a.i0 + (w.at + i) * kTile);
                }
                if (MODE == 1 && a.keep) {
                    const int who = (w.b * a.Hkv + w.g) * a.s.parts + w.part;
                    if (who == held) continue;                            // they are there already
                    held = who;
                }
                QTile q(a, w.v0 + w.t0);
                for (int t = 0; ok && t < w.nt; ++t) {
                    if (rb.lapped) ok = wait_or_abort(&sm->b_empty[rb.slot], rb.phase ^ 1u, sm, a.dev_status);
                    if (!ok) break;
                    unsigned char* dst = sB + rb.slot * kTileBytes;
                    if (MODE == 0) load_k(dst, &sm->b_full[rb.slot], w, (w.t0 + t) * kTile);
                    else {
                        mbar_arrive_expect_tx(&sm->b_full[rb.slot], q_bytes);
                        load_q(dst, &sm->b_full[rb.slot], w, q);
                        q.step(a, 1);
                    }
                    if (MODE == 1 && !SMALL) {
                        const uint32_t ns = nb % kNlse;
                        mbar_arrive_expect_tx(&sm->nlse_full[ns], kTile * 4);
                        bulk_load(sm->nlse[ns], a.nlse + ((int64_t)(w.b * a.Hkv + w.g) * a.s.tpg + w.v0 + w.t0 + t) * kTile, kTile * 4,
                                  &sm->nlse_full[ns]);
                        ++nb;
                    }
                    rb.next(a.keep ? (uint32_t)w.nt : b_slots);
                }
            }
        }
    } else if (warp == 1 || (warp == 3 && !SMALL)) {
        // ================= MMA issuers =================
        // Two warps take turns at the tiles: issuing the MMAs of a tile keeps a warp for as long as they take, and its waits
        // and bookkeeping another 400 to 700 cycles beside sixteen busy warps - the other warp's MMAs run meanwhile.
        // All lanes run the loop (uniform operands), one elected lane issues.
        constexpr uint32_t idesc = idesc_bf16_f32(kTile, kTile);
        const uint32_t me = warp == 1 ? 0u : 1u;                          // (small shape: one warp takes every tile)
        RingPos ra, rb;
        uint32_t it0 = 0;                                                 // tiles of the items before
        ScoreItem w, wn;
        bool ok = true;
        ScoreItems<MODE, SMALL> items(a);
        bool have = items.next(&w);
        const uint64_t adesc0 = smem_desc_sw128(smem_u32(sA)), bdesc0 = smem_desc_sw128(smem_u32(sB));
        while (ok && have) {
            wn = w;
            have = items.next(&wn);
            // kept B tiles are given up after the last item that reads them
            const bool give_up = !a.keep || !have || wn.g != w.g || wn.b != w.b || wn.part != w.part;
            // of two A tiles I have one with every B tile, of one A tile every other B tile
            const int turn = SMALL ? 0 : (int)((me ^ it0) & 1), ai = w.na == 2 ? turn : 0;
            const RingPos ra0 = ra;
            if (w.nt > 0) ra.next(a_slots);
            const RingPos ra1 = ra;
            if (w.nt > 0 && w.na == 2) ra.next(a_slots);
            const RingPos& r = ai == 1 ? ra1 : ra0;
            const uint64_t ad = adesc0 + r.slot * (uint32_t)(kTileBytes >> 4);
            RingPos rk = rb;                                              // with kept tiles the ring is as long as their number
            // (both warps wait for, and later declare done with, every tile of both rings, also those the other one
            // multiplies: neither can be a generation ahead)
            if (w.nt > 0) {
                ok = wait_or_abort(&sm->a_full[ra0.slot], ra0.phase, sm, a.dev_status);
                if (ok && w.na == 2) ok = wait_or_abort(&sm->a_full[ra1.slot], ra1.phase, sm, a.dev_status);
                ok = __all_sync(0xFFFFFFFFu, ok);
            }
            for (int t = 0; ok && t < w.nt; ++t) {
                const bool mine = SMALL || w.na == 2 || ((t ^ turn) & 1) == 0;
                const uint32_t it = it0 + (uint32_t)(w.na == 2 ? 2 * t + ai : t), buf = it % kAccs;
                const uint64_t bd = bdesc0 + rk.slot * (uint32_t)(kTileBytes >> 4);
                const uint32_t d_tmem = tmem_base + buf * kTile;
                ok = wait_or_abort(&sm->b_full[rk.slot], rk.phase, sm, a.dev_status);
                if (ok && mine && it >= kAccs) ok = wait_or_abort(&sm->tmem_empty[buf], ((it / kAccs) - 1) & 1, sm, a.dev_status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    if (mine) {
#pragma unroll
                        for (int k = 0; k < 8; ++k)                       // 16 channels are 32 bytes, 64 channels a half box
                            mma_bf16_ss(d_tmem, ad + ((k >> 2) * kHalfBytes + (k & 3) * 32) / 16,
                                        bd + ((k >> 2) * kHalfBytes + (k & 3) * 32) / 16, idesc, k > 0 ? 1u : 0u);
                        mma_commit(&sm->tmem_full[buf]);                  // the accumulator may be drained
                    }
                    if (give_up) mma_commit(&sm->b_empty[rk.slot]);       // I am done with the B tile
                }
                __syncwarp();
                rk.next(a.keep ? (uint32_t)w.nt : b_slots);
            }
            if (ok && w.nt > 0 && elect_one()) {                          // I am done with the A tiles
                mma_commit(&sm->a_empty[ra0.slot]);
                if (w.na == 2) mma_commit(&sm->a_empty[ra1.slot]);
            }
            __syncwarp();
            if (give_up) rb = rk;
            it0 += (uint32_t)(w.nt * w.na);
            w = wn;
        }
    } else if (warp == 2) {
        // ================= finisher: lane l has rows 4l .. 4l+3 of an A tile =================
        ScoreItem w;
        uint32_t it0 = 0;
        ScoreItems<MODE, SMALL> items(a);
        for (int round = 0; items.next(&w); ++round) {
            const int rs = round & 1;
            if (!__all_sync(0xFFFFFFFFu, wait_or_abort(&sm->res_full[rs], (round >> 1) & 1, sm, a.dev_status))) break;
            for (int i = 0; i < w.na; ++i) {
                // two A tiles: every other set has worked on tile i; one A tile: all of them have
                const int k0 = w.na == 2 ? (int)((it0 + i) & 1) : 0;
                float x[4], y[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    float2 v = sm->res[rs][k0][lane * 4 + u];
                    for (int k = k0 + w.na; k < kSets; k += w.na) {
                        const float2 o = sm->res[rs][k][lane * 4 + u];
                        if (MODE == 0) {
                            const float M = fmaxf(v.x, o.x);
                            if (M > -INFINITY) { v.y = v.y * exp2f(v.x - M) + o.y * exp2f(o.x - M); v.x = M; }
                        } else {
                            v.x += o.x;
                        }
                    }
                    x[u] = v.x; y[u] = v.y;
                }
                if (MODE == 0) {
                    // the copies of a row: every lane ends up with their sum (the rows past the first copy are not used)
                    for (int o = 16; o >= row_step / 4; o >>= 1) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const float ox = __shfl_xor_sync(0xFFFFFFFFu, x[u], o), oy = __shfl_xor_sync(0xFFFFFFFFu, y[u], o);
                            const float M = fmaxf(x[u], ox);
                            if (M > -INFINITY) { y[u] = y[u] * exp2f(x[u] - M) + oy * exp2f(ox - M); x[u] = M; }
                        }
                    }
                    if (a.s.ksplit > 1) {
                        const int64_t tile = (int64_t)(w.b * a.Hkv + w.g) * a.s.tpg + w.at + i;
                        float4* mine = reinterpret_cast<float4*>(a.stat + (tile * a.s.ksplit + w.part) * kTile + lane * 4);
                        mine[0] = make_float4(x[0], y[0], x[1], y[1]);
                        mine[1] = make_float4(x[2], y[2], x[3], y[3]);
                    } else {
                        const int64_t tile = (int64_t)(w.b * a.Hkv + w.g) * a.s.tpg + w.at + i;
#pragma unroll
                        for (int u = 0; u < 4; ++u) a.nlse[tile * kTile + lane * 4 + u] = minus_normaliser(a, w.at + i, lane * 4 + u, x[u], y[u]);
                    }
                } else {
                    const int64_t prow = ((int64_t)w.b * a.Hkv + w.g) * a.s.parts + w.part;
                    *reinterpret_cast<float4*>(a.partial + (prow * a.s.nkt + w.at + i) * kTile + lane * 4) =
                        make_float4(x[0], x[1], x[2], x[3]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm->res_empty[rs]);
            it0 += (uint32_t)(w.nt * w.na);
        }
    } else if (warp == 3) {
        // ================= small shape, pass 2: the normalisers of the B tiles, lane l those of rows 4l .. 4l+3 =================
        if (MODE == 1) {
            ScoreItem w;
            uint32_t nb = 0;
            bool ok = true;
            ScoreItems<MODE, SMALL> items(a);
            while (ok && items.next(&w)) {
                QTile q(a, w.v0 + w.t0);
                for (int t = 0; t < w.nt; ++t, ++nb, q.step(a, 1)) {
                    const int64_t tile = (int64_t)(w.b * a.Hkv + w.g) * a.s.tpg + w.v0 + w.t0 + t;
                    float v[4];
                    if (a.from_stat) {
                        norm_of_stat<2>(a, tile, lane * 4, v);
                    } else if (a.lse) {
                        norm_of_lse(a, tile, lane * 4, v);
                    } else {
                        const float4 x = __ldcg(reinterpret_cast<const float4*>(a.nlse + tile * kTile) + lane);
                        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
                    }
                    if (nb >= kNlse)
                        ok = __all_sync(0xFFFFFFFFu, wait_or_abort(&sm->nlse_empty[nb % kNlse], ((nb / kNlse) - 1) & 1, sm, a.dev_status));
                    if (!ok) break;
                    *reinterpret_cast<float4*>(&sm->nlse[nb % kNlse][lane * 4]) = make_float4(v[0], v[1], v[2], v[3]);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm->nlse_full[nb % kNlse]);
                }
            }
        }
    } else if (warp >= kFirstEpiWarp) {
        // ===== epilogue: set s of four warps drains accumulator s, a warp its TMEM lanes 32*(warp%4) .. +31 =====
        const int ew = warp - kFirstEpiWarp, quarter = warp & 3, set = ew >> 2;
        const uint32_t my_tmem = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(set * kTile);
        uint32_t it0 = 0, mine = 0;                          // tiles of the items before, tiles my set has taken
        bool ok = true;
        uint32_t nb = 0, gen = 0;                            // MODE 1: B tiles before those of this item; in its generation
        int held = -1;
        ScoreItem w;
        ScoreItems<MODE, SMALL> items(a);
        for (int round = 0; ok && items.next(&w); ++round) {
            // tiles go round the sets; of two A tiles my set has one, with every other B tile
            const int turn = (int)((set - it0) & (kSets - 1)), ai = w.na == 2 ? (turn & 1) : 0, step = kSets / w.na;
            int t = turn / w.na;
            const int rs = round & 1;
            if (MODE == 0) {
                float m_run = -INFINITY, l_run = 0.f;
                // TMEM lane = row of the A tile; of `copies` copies of the rows mine takes every copies-th chunk of columns
                const int row = quarter * 32 + lane, row0 = (quarter * 32) & (row_step - 1), copy = quarter * 32 / row_step;
                const QTile qa(a, w.at + ai);
                const int pos0 = qa.pt * a.s.box_p;              // first window position of my query tile
                const int my_end = a.causal ? min(a.N, a.q_lo + pos0 + a.by_box_h.div(row0 + lane) + 1) : a.N;     // my query sees the keys below
                // nothing to do for a warp whose 32 query rows lie past the window
                const bool idle = row0 >= box_rows || pos0 + a.by_box_h.div(row0) >= a.Nq;
                for (; t < w.nt; t += step, ++mine) {
                    ok = __all_sync(0xFFFFFFFFu, wait_or_abort(&sm->tmem_full[set], mine & 1, sm, a.dev_status));
                    if (!ok) break;
                    tc_fence_after();
                    if (idle) {
                        if (lane == 0) mbar_arrive(&sm->tmem_empty[set]);
                    } else {
#pragma unroll 1
                        for (int c0 = copy * 32; c0 < kTile; c0 += copies * 32) {
                            float v[32];
                            tmem_ld32(my_tmem + c0, v);
                            tmem_ld_wait();
                            if (c0 + copies * 32 >= kTile) {                  // the accumulator may be filled again
                                tc_fence_before();
                                __syncwarp();
                                if (lane == 0) mbar_arrive(&sm->tmem_empty[set]);
                            }
                            rowstat_chunk(v, my_end - (w.t0 + t) * kTile - c0, a.scale_log2, m_run, l_run);
                        }
                    }
                }
                if (!ok) break;
                if (round >= 2) ok = __all_sync(0xFFFFFFFFu, wait_or_abort(&sm->res_empty[rs], ((round >> 1) - 1) & 1, sm, a.dev_status));
                if (!ok) break;
                sm->res[rs][set][row] = make_float2(m_run, l_run);
            } else {
                f32x2 acc[4] = {both(0.f), both(0.f), both(0.f), both(0.f)};
                const int key0 = a.i0 + (w.at + ai) * kTile + quarter * 32 + (lane >> 2);     // my keys: key0 + 0, 8, 16, 24
                const int who = a.keep ? (w.b * a.Hkv + w.g) * a.s.parts + w.part : -2 - round;
                if (who != held) { nb += gen; gen = (uint32_t)w.nt; held = who; }       // kept B tiles are counted once
                QTile q(a, w.v0 + w.t0 + t);
                for (; t < w.nt; t += step, ++mine) {
                    const int qpos = q.pt * a.s.box_p;                                 // first window position of the tile
                    const int rows_here = min(a.s.box_p, a.Nq - qpos) * a.s.box_h;     // ... and its valid rows
                    q.step(a, step);
                    const uint32_t ns = (nb + (uint32_t)t) % kNlse;
                    const float* nls = sm->nlse[ns];
                    // query row c of the tile sees key j iff j <= q_lo + qpos + c / box_h
                    const bool mask = a.causal && a.i0 + (w.at + ai) * kTile + quarter * 32 + 31 > a.q_lo + qpos;
                    f32x2 tile[4] = {both(0.f), both(0.f), both(0.f), both(0.f)};
                    ok = wait_or_abort(&sm->nlse_full[ns], ((nb + (uint32_t)t) / kNlse) & 1, sm, a.dev_status);
                    ok = __all_sync(0xFFFFFFFFu, ok && wait_or_abort(&sm->tmem_full[set], mine & 1, sm, a.dev_status));
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll 1
                    for (int c0 = 0; c0 < rows_here; c0 += 32) {      // (chunks whose 32 query rows lie past the window are left out)
                        float v[32];
                        tmem_ld_16x256b_x4(my_tmem + c0, v);
                        tmem_ld_16x256b_x4(my_tmem + (16u << 16) + c0, v + 16);
                        tmem_ld_wait();
                        if (c0 + 32 >= rows_here) {                  // the accumulator may be filled again
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&sm->tmem_empty[set]);
                        }
                        const int col = c0 + 2 * (lane & 3);
                        if (!mask) {
                            colsum_chunk<false>(v, nls + col, nullptr, col, a.scale_log2, tile);
                        } else {
                            int first[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) first[k] = (key0 + 8 * k - a.q_lo - qpos) * a.s.box_h;
                            colsum_chunk<true>(v, nls + col, first, col, a.scale_log2, tile);
                        }
                    }
                    if (SMALL) {
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sm->nlse_empty[ns]);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[k] = add2(acc[k], tile[k]);
                }
                if (!ok) break;
                if (round >= 2) ok = __all_sync(0xFFFFFFFFu, wait_or_abort(&sm->res_empty[rs], ((round >> 1) - 1) & 1, sm, a.dev_status));
                if (!ok) break;
#pragma unroll
                for (int k = 0; k < 4; ++k) {                        // the four lanes of a key, and the two halves of a pair
                    float s0, s1;
                    unpack2(acc[k], s0, s1);
                    s0 += s1;
                    s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, 1);
                    s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, 2);
                    if ((lane & 3) == 0) sm->res[rs][set][quarter * 32 + (lane >> 2) + 8 * k] = make_float2(s0, 0.f);
                }
            }
            // what my set has of the item goes to the finisher
            it0 += (uint32_t)(w.nt * w.na);
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm->res_full[rs]);
        }
    }
    // ---- common exit: everyone meets, then the allocating warp frees the tensor memory ----------
    tc_fence_before();
    __syncthreads();
    if (sm->abort) {                              // let copies still in flight land before leaving
#pragma unroll 1
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// Large shape: the normalisers of every query tile, from stat or lse, for the bulk copies of pass 2.  A warp per tile; where a
// tile has more items than a warp loads at a time, the four warps of a CTA share it (us of a whole call,
// one warp / four: 4 heads of 7 x 9000 keys x 64 rows, 18 items, 35.4 / 32.3; 8 of 4 x 20000 x 20, 32 items, 41.0 / 37.6).
constexpr int kNormThreads = 128, kNormWarps = kNormThreads / 32, kNormDeep = 8;
template <bool SHARE>
__global__ void __launch_bounds__(kNormThreads) score_norm_kernel(const ScoreTcArgs a, int tiles) {
    __shared__ float4 s_m[kNormWarps][32], s_l[kNormWarps][32];
    pdl_enter();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tile = SHARE ? (int)blockIdx.x : (int)blockIdx.x * kNormWarps + warp;
    float v[4];
    if (SHARE) {
        float M[4], Ls[4];
        add_stats<kNormDeep>(a, tile, lane * 4, warp, kNormWarps, M, Ls);
        s_m[warp][lane] = make_float4(M[0], M[1], M[2], M[3]);
        s_l[warp][lane] = make_float4(Ls[0], Ls[1], Ls[2], Ls[3]);
        __syncthreads();
        if (warp > 0) return;
#pragma unroll
        for (int q = 1; q < kNormWarps; ++q) {
            const float4 m = s_m[q][lane], l = s_l[q][lane];
            add_stat(M[0], Ls[0], m.x, l.x); add_stat(M[1], Ls[1], m.y, l.y);
            add_stat(M[2], Ls[2], m.z, l.z); add_stat(M[3], Ls[3], m.w, l.w);
        }
        const int qt = tile % a.s.tpg;
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = minus_normaliser(a, qt, lane * 4 + u, M[u], Ls[u]);
    } else {
        if (tile >= tiles) return;
        if (a.from_stat) norm_of_stat<kNormDeep>(a, tile, lane * 4, v); else norm_of_lse(a, tile, lane * 4, v);
    }
    reinterpret_cast<float4*>(a.nlse + (int64_t)tile * kTile)[lane] = make_float4(v[0], v[1], v[2], v[3]);
}

// The column sums of the items of a key, added in order: group sums and head mean.  Thread = key.
constexpr int kSumThreads = 128;
__global__ void __launch_bounds__(kSumThreads)
score_sum_kernel(const float* __restrict__ partial, int n, int64_t row_len, int Hkv, int parts, float inv_heads,
                 float* __restrict__ score, float* __restrict__ score_head, int64_t head_stride, int32_t* dev_status) {
    pdl_enter();
    const int b = blockIdx.y, j = blockIdx.x * kSumThreads + threadIdx.x;
    if (j >= n) return;
    const float* col = partial + (int64_t)b * Hkv * parts * row_len + j;
    float tot = 0.f, gs = 0.f;
    int in_group = 0, g = 0;
    const int P = Hkv * parts;
    for (int p0 = 0; p0 < P; p0 += 8) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = p0 + u < P ? __ldcg(col + (p0 + u) * row_len) : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (p0 + u >= P) break;
            gs += v[u];
            if (++in_group == parts) {
                if (score_head) score_head[((int64_t)b * Hkv + g) * head_stride + j] = gs;
                tot += gs;
                gs = 0.f; in_group = 0; ++g;
            }
        }
    }
    const float sc = tot * inv_heads;
    score[(int64_t)b * n + j] = sc;
    if (dev_status && (__float_as_uint(sc) & 0x7F800000u) == 0x7F800000u) atomicOr(dev_status, LVLM_DEV_NONFINITE);
}

ScoreShape score_shape(const lvlm_dims* d) {
    ScoreShape s;
    const int G = d->H / d->Hkv, Nq = d->q_hi - d->q_lo;
    s.box_h = 1; s.box_p = kTile;
    s.npt = (Nq + kTile - 1) / kTile;
    s.tpg = G * s.npt;
    if (G > 1 && G <= kTile) {                   // all heads of the group in one tile, where that makes fewer tiles
        const int bp = kTile / G, npt = (Nq + bp - 1) / bp;
        if (npt < s.tpg) { s.box_h = G; s.box_p = bp; s.npt = s.tpg = npt; }
    }
    // a window of few rows: no rows in a tile that it does not have (less to copy), and in pass 1 their logits several
    // times over, so that all epilogue warps have some
    s.copies = 1;
    if (s.npt == 1) {
        s.box_p = Nq < s.box_p ? Nq : s.box_p;
        while (s.copies < 4 && s.box_h * s.box_p <= kTile / (2 * s.copies)) s.copies *= 2;
    }
    s.nh = G / s.box_h;
    s.nkt = (d->n + kTile - 1) / kTile;
    // The split of either pass, in units of a tile's time: the work of a CTA on average (an item costs `fixed` beside its
    // tiles) and half an item that it may wait for others at the end.
    const int64_t groups = (int64_t)d->B * d->Hkv;
    const int max_kt = (d->N + kTile - 1) / kTile;
    auto split = [&](int64_t a_tiles, int b_tiles, int most, int ctas, int per_item, double fixed, double extra, double each) {
        double best = 1e30;
        int take = 1;
        for (int p = 1; p <= most && p <= b_tiles; ++p) {
            const double items = (double)(groups * ((a_tiles + per_item - 1) / per_item) * p);
            const double item = (a_tiles < per_item ? (double)a_tiles : per_item) * ((b_tiles + p - 1) / p) + fixed;
            const double mean = ((double)(groups * a_tiles * b_tiles) + items * fixed) / ctas;
            const double est = (items <= ctas ? item : (mean + 0.5 * item > item ? mean + 0.5 * item : item)) + (p > 1 ? extra : 0.0) + each * p;
            if (est < best - 1e-9) { best = est; take = p; }
        }
        return take;
    };
    s.small1 = groups * s.tpg * max_kt <= kSmallTiles1;
    s.small2 = groups * s.nkt * s.tpg <= kSmallTiles2;
    // Tiles of results in the workspace.  The splits rise and fall with the size, the workspace may not (a program sizes it
    // once, for its longest prompt and widest batch): it has room for any split up to a limit on the tiles, beyond that
    // for the results without one, and the splits keep to it.
    const int64_t key_tiles = groups * s.nkt, query_tiles = groups * s.tpg, per_head = (int64_t)d->B * d->H * d->n / kTile;
    const int64_t no_split = key_tiles > kMaxPartTiles ? key_tiles : kMaxPartTiles, any_part = key_tiles * (s.tpg < kMaxParts ? s.tpg : kMaxParts);
    const int64_t any_split = query_tiles * (max_kt < kMaxSplit ? max_kt : kMaxSplit);
    s.part_tiles = any_part < no_split ? any_part : no_split;
    s.stat_tiles = any_split < kMaxStatTiles ? any_split : kMaxStatTiles;
    const int most1 = (int)(s.stat_tiles / query_tiles), most2 = (int)((s.part_tiles > per_head ? s.part_tiles : per_head) / key_tiles);
    // (large shape, pass 1: items that share a query tile need a launch that adds their results, about five tiles' time: 16 x 8 heads
    // of 4 x 1230 keys x 96 rows, whole call, without 59.1 us, with three items a tile 63.4)
    s.ksplit = s.small1 ? split(s.tpg, max_kt, most1 < 16 ? most1 : 16, 2 * kSmCount, 1, 4.0, 0.5, 0.3)
                        : split(s.tpg, max_kt, most1 < kMaxSplit ? most1 : kMaxSplit, kSmCount, 2, 1.0, 4.5, 0.02);
    s.parts = split(s.nkt, s.tpg, most2 < kMaxParts ? most2 : kMaxParts, s.small2 ? 2 * kSmCount : kSmCount, s.small2 ? 1 : 2,
                    s.small2 ? 4.0 : 1.0, 0.0, 0.02);
    return s;
}

lvlm_status launch_score_tc(const void* Q, const void* K, const float* lse, const lvlm_dims* d,
                            const ScoreStrides& st, float scale, const ScoreLayout& L, char* ws, float* score,
                            float* score_head, int32_t* dev_status, cudaStream_t stream, bool normalisers_ready) {
    const int Nq = d->q_hi - d->q_lo;
    const ScoreShape& s = L.shape;
    CUtensorMap qmap, kmap;
    {
        const uint64_t dims[4] = {(uint64_t)kHeadDim, (uint64_t)d->H, (uint64_t)Nq, (uint64_t)d->B};
        const uint64_t strides[3] = {(uint64_t)st.q_sh * 2, (uint64_t)st.q_sn * 2, (uint64_t)st.q_sb * 2};
        const uint32_t box[4] = {64, (uint32_t)s.box_h, (uint32_t)s.box_p, 1};
        if (!make_tmap_bf16(&qmap, Q, 4, dims, strides, box)) return LVLM_ERR_CUDA;
    }
    {
        const uint64_t dims[4] = {(uint64_t)kHeadDim, (uint64_t)d->N, (uint64_t)d->Hkv, (uint64_t)d->B};
        const uint64_t strides[3] = {(uint64_t)kHeadDim * 2, (uint64_t)st.kv_sh * 2, (uint64_t)st.kv_sb * 2};
        const uint32_t box[4] = {64, (uint32_t)kTile, 1, 1};
        if (!make_tmap_bf16(&kmap, K, 4, dims, strides, box)) return LVLM_ERR_CUDA;
    }
    auto add_up = [&](int parts) {
        return launch_kernel(score_sum_kernel, dim3((unsigned)((d->n + kSumThreads - 1) / kSumThreads), (unsigned)d->B), dim3(kSumThreads), 0,
                             stream, 1, reinterpret_cast<float*>(ws + L.off_partial), d->n, (int64_t)s.nkt * kTile, d->Hkv, parts,
                             1.0f / (float)d->H, score, score_head, d->head_stride ? d->head_stride : (int64_t)d->n, dev_status);
    };
    if (lse == nullptr && !normalisers_ready) {
        const OnceScoreShape o = score_once_shape(d, s, scale);
        if (o.kt) {
            const lvlm_status r = launch_score_once(qmap, kmap, d, s, o, scale, reinterpret_cast<float*>(ws + L.off_partial), dev_status, stream);
            return r != LVLM_OK ? r : add_up(o.parts);
        }
    }
    ScoreTcArgs a;
    a.B = d->B; a.H = d->H; a.G = d->H / d->Hkv; a.Hkv = d->Hkv; a.N = d->N; a.Nq = Nq; a.i0 = d->i0; a.n = d->n;
    a.q_lo = d->q_lo; a.causal = d->causal; a.scale_log2 = scale * kLog2eT; a.s = s;
    a.by_hkv = FastDiv(d->Hkv); a.by_b = FastDiv(d->B); a.by_nh = FastDiv(s.nh); a.by_box_h = FastDiv(s.box_h); a.by_box_p = FastDiv(s.box_p);
    a.nlse = reinterpret_cast<float*>(ws + L.off_nlse);
    a.partial = reinterpret_cast<float*>(ws + L.off_partial);
    a.dev_status = dev_status;
    a.stat = reinterpret_cast<float2*>(ws + L.off_stat);
    const int64_t groups = (int64_t)d->B * d->Hkv;
    a.a_slots = 3; a.keep = 0; a.from_stat = 0; a.lse = nullptr; a.lse_scale = 0.f;
    auto launch = [&](auto small, void (*kernel)(CUtensorMap, CUtensorMap, ScoreTcArgs), int64_t a_tiles, int split) -> lvlm_status {
        using Cfg = ScoreCfg<decltype(small)::value>;
        const int64_t items = groups * ((a_tiles + Cfg::kItemTiles - 1) / Cfg::kItemTiles) * split, most = Cfg::kCtas * kSmCount;
        if (items > 0x7FFFFFFFll) return LVLM_ERR_UNSUPPORTED;
        const size_t smem = 1024 + (size_t)kTileBytes * Cfg::kSlots + sizeof(TcSmem<decltype(small)::value>);
        LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        a.items = (int)items; a.by_split = FastDiv(split);
        if (decltype(small)::value) { a.a_slots = 1; a.keep = 0; }
        return launch_kernel(kernel, dim3((unsigned)(items < most ? items : most)), dim3(Cfg::kThreads), smem, stream, 1, qmap, kmap, a);
    };
    lvlm_status r = LVLM_OK;
    if (lse == nullptr && !normalisers_ready) {
        r = s.small1 ? launch(std::true_type(), score_tc_kernel<0, true>, s.tpg, s.ksplit)
                     : launch(std::false_type(), score_tc_kernel<0, false>, s.tpg, s.ksplit);
        a.from_stat = s.ksplit > 1;
    } else {
        a.lse = lse ? lse : reinterpret_cast<const float*>(ws + L.off_lse);
        a.lse_scale = lse ? -kLog2eT : -1.f;
    }
    // (Small shape: a warp of every CTA adds the items itself, two loads in flight.  After a small pass 1 that is quicker than a
    // launch - 8 heads x 4000 keys x 32 rows, up to 16 items: 18.4 / 20.5 us - after a large one with many items it is not: 4 heads
    // of 7 x 9000 keys x 32 rows, 24 items: 36.4 / 30.2.)
    if (r == LVLM_OK && (s.small2 ? a.from_stat && !s.small1 && s.ksplit > 4 : a.from_stat || a.lse)) {
        const int64_t tiles = groups * s.tpg;
        if (tiles > 0x7FFFFFFFll) return LVLM_ERR_UNSUPPORTED;
        r = a.from_stat && s.ksplit > kNormDeep
                ? launch_kernel(score_norm_kernel<true>, dim3((unsigned)tiles), dim3(kNormThreads), 0, stream, 1, a, (int)tiles)
                : launch_kernel(score_norm_kernel<false>, dim3((unsigned)((tiles + kNormWarps - 1) / kNormWarps)), dim3(kNormThreads), 0,
                                stream, 1, a, (int)tiles);
        a.from_stat = 0; a.lse = nullptr;
    }
    if (r != LVLM_OK) return r;
    // pass 2: the query tiles of an item stay in shared memory for the next key tiles of the same KV group when they are
    // few and the same for all of them
    const int most = (s.tpg + s.parts - 1) / s.parts;
    a.keep = s.tpg % s.parts == 0 && most <= kMaxKeep && (!d->causal || d->q_lo >= d->i0 + d->n);
    a.a_slots = a.keep && most == kMaxKeep ? 2 : 3;
    r = s.small2 ? launch(std::true_type(), score_tc_kernel<1, true>, s.nkt, s.parts)
                 : launch(std::false_type(), score_tc_kernel<1, false>, s.nkt, s.parts);
    if (r != LVLM_OK) return r;
    return add_up(s.parts);
}

}  // namespace lvlm
