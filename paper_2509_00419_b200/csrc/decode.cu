// lvlm_decode_attn: one generated token attends to every cached key and value of its KV head
// (Section 3.2.2, paragraph 1), over caches whose lengths differ per (sequence, KV head) after
// compression.  HBM-bound: every K and V row is read once and shared by the G query heads of
// the group.
//
// One launch, split-K inside thread-block clusters.  The S CTAs of a cluster share one (sequence,
// KV head): its key tiles are cut into S equal runs, so a ragged cache costs what its own length
// costs.  A CTA is one producer warp and four compute warps around a ring of shared-memory stages
// of 64 keys: the producer fetches the K and V rows of a stage with four TMA tile copies (128-byte
// swizzle, so that ldmatrix is conflict free; completion counted by an mbarrier), a compute warp
// takes 16 keys of the stage, multiplies them with small tensor-core MMAs (the G query heads of the
// group are the rows of a 16-row tile) and keeps an online softmax per head, so the main loop has no
// block barrier.  With d->cache_stable the first lap of the ring is fetched before the kernel waits
// for the one ahead of it in the stream.  The warps of a CTA are merged in warp order
// in shared memory; the CTAs of the cluster then read each other's (max, sum, output) through
// distributed shared memory in rank order, each finishing a slice of the output channels and the
// acc_score entries of its own keys, whose scaled logits it has kept in shared memory (in the
// workspace when a run is too long for that).
//
// Inside a chain of layers the fetches of a layer start while the one ahead finishes; what counts is the time from the
// end of the layer ahead: query, one lap of products, merge of the warps, cluster barrier, output.  So: a warp parks its
// output where its own rows of the last stage lay (one block barrier), no releasing barrier waits for stores (the
// appended row is written last), and few registers live across the loop (they spilled).  us per layer, before -> now:
// 4 heads of 216 rows 4.5 -> 4.0, with acc_score 5.65 -> 4.9; 64 heads of 1100 rows 12.1 -> 11.3 (acc_score), 216 rows 7.3 -> 6.2;
// 128 heads of 1100 rows 19.9 -> 17.5.  Tried and slower: 8 or 16 compute warps a CTA (5.7 to 20 us), acc_score
// fetched ahead of the cluster barrier (5.2 -> 5.6).
//
// Few heads with long caches (a video prompt's first layers: one sequence, 4 KV heads, 32898 rows) leave most of the
// GPU idle that way: a cluster has at most 8 CTAs.  There (parts_from_tiles) the run of a head is cut into as many parts as fill the GPU
// twice, without clusters; every part leaves its (max, sum, output) in the workspace, and a second, small launch adds
// the parts in order, finishes acc_score and bumps len.  HBM-bound either way.  That shape, per layer (67 MB):
// 53.6 us with 8 CTAs a head, 17.8 us as 74 parts a head
// (3.8 TB/s; the start-up, the merge and the second launch are 6 us of it).
#include <mutex>

#include "common.cuh"
#include "sm100.cuh"

namespace lvlm {

using namespace sm100;

constexpr int kDecWarps = 4;                         // compute warps
constexpr int kDecThreads = (kDecWarps + 1) * 32;    // ... and the producer warp
constexpr int kTileKeys = 16;                        // keys per warp tile
constexpr int kStageKeys = kDecWarps * kTileKeys;    // keys per stage
constexpr int kBoxBytes = kStageKeys * 128;          // one TMA box: 64 keys x 64 channels
constexpr int kStageBytes = 4 * kBoxBytes;           // K low half, K high half, V low half, V high half
constexpr int kStagesDec = 3;
constexpr int kRingBytes = kStagesDec * kStageBytes;
constexpr int kDecTargetCtas = 2 * 148;              // CTAs wanted in flight: two per SM of a 148-SM part
constexpr int kDecMaxCluster = 8;                    // portable cluster size
constexpr int kDecMinTiles = 2;                      // a CTA's run is not made shorter than this by splitting
constexpr int kDecPartTiles = 4;                     // a part's run is not made shorter than this
constexpr int kDecLogitBytes = 12 * 1024;            // scaled logits of a CTA's own keys kept in shared memory
constexpr float kLog2e = 1.4426950408889634f;

// S CTAs a head form a cluster; P > 0: as many independent CTAs a head whose results a second launch adds.
// Bytes of workspace: `logits` always, `used` by the form taken, `total` what a caller is told: room for the parts of any number of
// heads, so that it never shrinks as the problem grows.
struct DecodeLayout { int S, P; size_t off_s, off_ml, off_o, off_len, logits, used, total; };

// Rows, in tiles, from which the heads are cut into parts where a cluster of 8 a head leaves SMs idle.  us per layer as
// cluster / as parts, inside a chain of layers:
//   from 32 heads the clusters of 8 no longer fit the GPU side by side: 36 heads of 216 rows 9.3 / 6.9, 2500 18.0 / 14.0,
//   9000 45 / 33; 32 heads of 216 rows 6.5 / 5.7, 9000 32 / 29;
//   without acc_score the cluster's one launch wins while the runs are short: 4 heads of 600 rows 4.8 / 5.4, 1100 5.4 / 5.5,
//   2100 7.1 / 5.9, 8200 16.4 / 9.5; 8 heads of 2100 rows 7.1 / 7.0, 4100 10.3 / 9.0; 16 heads of 4100 rows 12.7 / 12.0, 16400 36 / 26;
//   24 heads of 16400 rows 37.5 / 35.6;
//   with it the second launch takes the update of acc_score off the cluster's tail: 4 heads of 600 rows 5.8 / 5.7, 1100
//   6.6 / 5.9; 8 heads of 600 rows 5.7 / 5.3; 16 heads of 2100 rows 9.2 / 8.9, 4100 14.0 / 12.1.
// The lengths themselves are only known on the device.  Where the caller gives a bound of them, that decides (known).
// Where only the capacity is known, the cache may be short - after the compaction of a prompt it is - and then the
// second launch is lost time (4 heads of 216 rows in 33000: 4.1 / 5.6, with acc_score 5.3 / 6.1; 16 heads 4.4 / 6.3, 5.6 / 6.2).  The
// line lies where a full cache gains in proportion what such a short one loses: without acc_score 4 heads of 6200 rows 13.4 / 8.7,
// 8 of 8200 16.5 / 11.8, 16 of 25000 52 / 36, more never; with it 4 heads of 2100 rows 8.3 / 6.8, 8 of 4100 11.4 / 9.0, 20 of
// 4100 16.1 / 14.1.
static int parts_from_tiles(int64_t heads, bool acc, bool known) {
    constexpr int kNever = 1 << 28;
    if (heads >= 32) return 14;
    if (known && acc) return heads <= 8 ? 36 : heads <= 20 ? 192 : 800;
    if (known) return heads <= 4 ? 96 : heads <= 8 ? 192 : heads <= 20 ? 320 : 800;
    if (acc) return heads <= 4 ? 128 : heads <= 8 ? 192 : heads <= 20 ? 256 : 800;
    return heads <= 4 ? 384 : heads <= 8 ? 512 : heads <= 16 ? 1536 : kNever;
}

// may_split: the caller's workspace has room for the parts.
static bool decode_layout(const lvlm_dims* d, DecodeLayout* L, bool acc, bool may_split) {
    if (!d || d->B <= 0 || d->H <= 0 || d->Hkv <= 0 || d->H % d->Hkv || d->cap <= 0) return false;
    // cluster size: the power of two that brings the grid closest to the target without going
    // over it, as long as a full cache still gives every CTA a few tiles
    const int64_t heads = (int64_t)d->B * d->Hkv;
    const int tiles = (d->cap + kTileKeys - 1) / kTileKeys;
    int S = 1;
    while (S < kDecMaxCluster && heads * (2 * S) <= kDecTargetCtas && tiles / (2 * S) >= kDecMinTiles) S *= 2;
    L->S = S;
    L->P = 0;
    const int rows = d->N > 0 && d->N < d->cap ? d->N : d->cap, row_tiles = (rows + kTileKeys - 1) / kTileKeys;
    if (may_split && S == kDecMaxCluster && row_tiles >= parts_from_tiles(heads, acc, d->N > 0)) {
        const int fill = (int)(kDecTargetCtas / heads), most = (row_tiles + kDecPartTiles - 1) / kDecPartTiles;   // (a whole stage each)
        L->P = fill < most ? fill : most;
    }
    size_t off = 0;
    L->off_s = off; off = align_up(off + (size_t)d->B * d->H * d->cap * 4, 256);
    L->logits = L->off_ml = L->off_o = L->off_len = off;
    if (L->P > 0) {
        L->off_ml = off;  off = align_up(off + (size_t)d->B * d->H * L->P * 8, 256);
        L->off_o = off;   off = align_up(off + (size_t)d->B * d->H * L->P * kHeadDim * 4, 256);
        L->off_len = off; off = align_up(off + (size_t)heads * 4, 256);
    }
    L->used = off;
    // (heads * P <= kDecTargetCtas; shorter caches are never cut)
    const size_t part_rows = (size_t)(d->H / d->Hkv) * kDecTargetCtas;
    L->total = L->logits;
    if (tiles >= kDecMaxCluster * kDecMinTiles)
        L->total += align_up(part_rows * 8, 256) + align_up(part_rows * kHeadDim * 4, 256) + align_up((size_t)heads * 4, 256);
    return true;
}

size_t decode_attn_workspace(const lvlm_dims* d) {
    DecodeLayout L;
    return decode_layout(d, &L, false, false) ? L.total : 0;
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
// D (16x8 fp32) += A (16x16 bf16, row) * B (16x8 bf16, col)
__device__ __forceinline__ void mma_16816(float* d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

struct DecodeArgs {
    const __nv_bfloat16* q; __nv_bfloat16* Kc; __nv_bfloat16* Vc; int32_t* len;
    const __nv_bfloat16* k_new; const __nv_bfloat16* v_new; float* acc_score; __nv_bfloat16* out;
    int H, Hkv, cap, S;
    int early;               // the cache and len are not written by the kernel ahead: fetch before waiting for it
    int logit_keys;          // keys of a run whose logits fit in shared memory (0: they go to ws_s)
    int64_t kv_sb, kv_sh;
    float scale_log2;
    float2* part_ml;         // parts: [B*Hkv][S][G] (max, sum), [B*Hkv][S][G][128] output relative to it,
    float* part_o;           //        and [B*Hkv] length before the append, -1 = nothing was appended
    int32_t* part_len;
    float* ws_s;             // [B*H][cap] scaled logits (log2 domain), only with acc_score and a long run
    int32_t* dev_status;
#ifdef LVLM_TEST_HOOKS
    int starve;
#endif
};

// The test build can keep the producer from fetching anything, so that the waits for the stages run out.
#ifdef LVLM_TEST_HOOKS
static int g_decode_starve = 0;
__device__ __forceinline__ bool starved(const DecodeArgs& a) { return a.starve != 0; }
#else
__device__ __forceinline__ bool starved(const DecodeArgs&) { return false; }
#endif

// Offset inside a stage of the 16-byte chunk `ch` (0..15) of key row `r` (0..63): K or V half boxes of 64
// channels, rows of 128 bytes, chunks XOR-swizzled with the row as the TMA copy wrote them.
__device__ __forceinline__ uint32_t stage_off(int r, int ch) {
    return (uint32_t)((ch >> 3) * kBoxBytes + r * 128 + (((ch & 7) ^ (r & 7)) << 4));
}

// grid.x = heads * S, clusters of S CTAs along x: cluster = (sequence, KV head), rank = run of tiles.
// kDecSolo: one CTA per head and no cluster instruction in the kernel at all.  kDecParts: S CTAs that know nothing of
// each other leave their results in the workspace.
enum { kDecSolo = 0, kDecCluster = 1, kDecParts = 2 };

template <int G, int MODE>
__global__ void __launch_bounds__(kDecThreads, 2)
decode_cluster_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                      const DecodeArgs a) {
    constexpr bool CL = MODE == kDecCluster;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float2* s_wml = reinterpret_cast<float2*>(smem + kRingBytes);       // [4 warps][8 heads] (max, sum)
    float2* s_ML = s_wml + kDecWarps * 8;                               // [8] this CTA's (max, sum) per head
    float* s_FM = reinterpret_cast<float*>(s_ML + 8);                   // [8] cluster-wide max
    float* s_FI = s_FM + 8;                                             // [8] 1 / cluster-wide sum
    float2* s_res = reinterpret_cast<float2*>(smem + 2 * kBoxBytes);    // [G][64] this CTA's output (the ring, once it is done)
    uint64_t* s_full = reinterpret_cast<uint64_t*>(s_FI + 8);                    // [kStagesDec]
    uint64_t* s_empty = s_full + kStagesDec;                            // [kStagesDec]
    float* s_logit = reinterpret_cast<float*>(s_empty + kStagesDec + 1);          // [G][logit_keys]
    __shared__ int s_abort;
    __shared__ __align__(16) uint4 s_app[32];                          // the appended row: K, then V

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 32) { prefetch_tmap(&kmap); prefetch_tmap(&vmap); }     // the descriptors start their way first
    if (tid == 0) {
        for (int s = 0; s < kStagesDec; ++s) { mbar_init(&s_full[s], 1); mbar_init(&s_empty[s], kDecWarps); }
        s_abort = 0;
        fence_barrier_init();
    }
    __syncthreads();
    // With a.early the first key/value stages and the length are fetched while the kernel ahead in the
    // stream is still finishing; q, k_new, v_new and every write come after the wait in any case.
    if (!a.early) pdl_enter();
    const int S = MODE == kDecSolo ? 1 : a.S, H = a.H, cap = a.cap;
    const int hd = blockIdx.x / S;
    const int rank = MODE == kDecParts ? (int)(blockIdx.x % S) : CL ? (int)cluster_ctarank() : 0;
    const int b = hd / a.Hkv, g = hd % a.Hkv, h0 = g * G;

    // ---- this head's length; every CTA of the cluster takes the same decisions ---------------------------
    int ln = a.len[hd];
    const bool bad = ln < 0 || ln > cap;
    if (bad) ln = 0;
    const bool app = a.k_new != nullptr && !bad && ln < cap;
    if (rank == 0 && tid == 0 && a.dev_status && (bad || (a.k_new != nullptr && !bad && !app)))
        atomicOr(a.dev_status, LVLM_DEV_BOUNDS);                        // bad length, or append at capacity
    const int lne = ln + (app ? 1 : 0);
    if (lne == 0) {                                                     // no key at all: zeros
        if (a.early) pdl_enter();
        if (MODE == kDecParts) {
            if (tid < G) a.part_ml[((int64_t)hd * S + rank) * G + tid] = make_float2(-INFINITY, 0.f);
            if (rank == 0 && tid == 0) a.part_len[hd] = -1;
            return;
        }
        if (rank == 0)
            for (int i = tid; i < G * kHeadDim; i += kDecThreads)
                a.out[(int64_t)(b * H + h0) * kHeadDim + i] = __float2bfloat16_rn(0.f);
        return;
    }
    const int nt = (lne + kTileKeys - 1) / kTileKeys;
    int per = (nt + S - 1) / S;
    if (per >= kDecWarps) per = (per + kDecWarps - 1) / kDecWarps * kDecWarps;   // whole stages where the run is long enough
    const int t_lo = min(nt, rank * per), t_hi = min(nt, t_lo + per);   // my run of tiles
    const int nstage = (t_hi - t_lo + kDecWarps - 1) / kDecWarps;
    if (MODE == kDecParts && nstage == 0) {                             // a part without keys: no weight, no output
        if (a.early) pdl_enter();
        if (tid < G) a.part_ml[((int64_t)hd * S + rank) * G + tid] = make_float2(-INFINITY, 0.f);
        return;
    }
    const uint32_t ring = smem_u32(smem);
    volatile int* abort_flag = &s_abort;
    auto wait_on = [&](uint64_t* bar, uint32_t parity) -> bool {
        if (*abort_flag) return false;
        if (mbar_wait(bar, parity)) return true;
        *abort_flag = 1;
        if (a.dev_status) atomicOr(a.dev_status, LVLM_DEV_TIMEOUT);
        return false;
    };

    float o[16][2];                            // head `row`, columns nt*8 + qd*2 + {0,1}
#pragma unroll
    for (int i = 0; i < 16; ++i) o[i][0] = o[i][1] = 0.f;
    float m_run = -INFINITY, l_run = 0.f;      // of head `row`; l_run is this lane's share of the sum
    const int row = lane >> 2, qd = lane & 3;
    // the warp of this CTA whose tile takes the appended row, or -1
    const int app_warp = app && ln / kTileKeys >= t_lo && ln / kTileKeys < t_hi ? (ln / kTileKeys - t_lo) % kDecWarps : -1;
    auto store_appended = [&]() {
        if (warp != app_warp) return;
        // (a warp whose wait has given up comes here without having patched its tile: the copy of the row is waited for here too,
        // so that the cache never takes a row that has not landed)
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        *reinterpret_cast<uint4*>((lane < 16 ? a.Kc : a.Vc) + (int64_t)b * a.kv_sb + (int64_t)g * a.kv_sh + (int64_t)ln * kHeadDim + (lane & 15) * 8) = s_app[lane];
    };

    if (warp == kDecWarps) {
        // ---- producer: four tile copies per stage ---------------------------------------------------------
        auto issue = [&](int s) {
            unsigned char* st = smem + (s % kStagesDec) * kStageBytes;
            const int j0 = (t_lo + s * kDecWarps) * kTileKeys;
            mbar_arrive_expect_tx(&s_full[s % kStagesDec], kStageBytes);
            tma_load_4d(st, &kmap, &s_full[s % kStagesDec], 0, j0, g, b);
            tma_load_4d(st + kBoxBytes, &kmap, &s_full[s % kStagesDec], 64, j0, g, b);
            tma_load_4d(st + 2 * kBoxBytes, &vmap, &s_full[s % kStagesDec], 0, j0, g, b);
            tma_load_4d(st + 3 * kBoxBytes, &vmap, &s_full[s % kStagesDec], 64, j0, g, b);
        };
        if (lane == 0 && !starved(a)) {
            for (int s = 0; s < kStagesDec && s < nstage; ++s) issue(s);
        }
        if (a.early) pdl_enter();
        if (lane == 0 && !starved(a)) {
            for (int s = kStagesDec; s < nstage; ++s) {
                if (!wait_on(&s_empty[s % kStagesDec], (uint32_t)(s / kStagesDec - 1) & 1u)) break;
                issue(s);
            }
        }
    } else {
        if (a.acc_score) {                     // my keys' acc_score entries: needed at the very end, fetched now
            const float* acc = a.acc_score + (int64_t)hd * cap;
            const int j_lo = t_lo * kTileKeys, j_hi = min(lne, t_hi * kTileKeys);
            for (int j = j_lo + tid * 32; j < j_hi; j += kDecWarps * 32 * 32) prefetch_l2(acc + j);
        }
        if (a.early) pdl_enter();
        const __nv_bfloat16* kn = app ? a.k_new + (int64_t)hd * kHeadDim : nullptr;
        const __nv_bfloat16* vn = app ? a.v_new + (int64_t)hd * kHeadDim : nullptr;
        // the appended row: fetched now, patched into its tile below, written to the cache at the very end (a store
        // before the cluster barrier would be waited for there)
        if (app_warp == warp) {
            asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"((uint32_t)__cvta_generic_to_shared(&s_app[lane])),
                         "l"((lane < 16 ? kn : vn) + (lane & 15) * 8) : "memory");
        }
        // query fragments: heads of the group are rows 0..G-1 of a 16-row A tile
        uint32_t qa[8][2];
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            qa[ks][0] = qa[ks][1] = 0u;
            if (row < G) {
                const uint32_t* qp = reinterpret_cast<const uint32_t*>(a.q + (int64_t)(b * H + h0 + row) * kHeadDim);
                qa[ks][0] = __ldg(qp + ks * 8 + qd);
                qa[ks][1] = __ldg(qp + ks * 8 + 4 + qd);
            }
        }
        for (int s = 0; s < nstage; ++s) {
            const bool ok = wait_on(&s_full[s % kStagesDec], (uint32_t)(s / kStagesDec) & 1u);
            const int t = t_lo + s * kDecWarps + warp;
            if (ok && t < t_hi) {
                const uint32_t st = ring + (s % kStagesDec) * kStageBytes;      // K boxes; the V boxes follow
                const int r0 = warp * kTileKeys;                               // my rows of the stage
                const int j0 = t * kTileKeys;
                if (app && ln >= j0 && ln < j0 + kTileKeys) {
                    // the appended row: into its place of the tile
                    const int rr = r0 + ln - j0, ch = lane & 15;
                    const uint32_t off = (lane < 16 ? 0 : 2 * kBoxBytes) + stage_off(rr, ch);
                    asm volatile("cp.async.wait_all;\n" ::: "memory");
                    const uint4 x = s_app[lane];             // (copied by this very lane)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(st + off), "r"(x.x), "r"(x.y), "r"(x.z), "r"(x.w) : "memory");
                }
                if (j0 + kTileKeys > lne) {
                    // V rows past the last key hold whatever the cache holds: zero them, their weight is zero
                    for (int e = lane; e < (j0 + kTileKeys - lne) * 16; e += 32) {
                        const int rr = r0 + (lne - j0) + (e >> 4), ch = e & 15;
                        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(st + 2 * kBoxBytes + stage_off(rr, ch)), "r"(0u) : "memory");
                    }
                }
                __syncwarp();
                // ---- S = Q K^T for 16 keys -------------------------------------------------------------------
                float sc[2][4];
#pragma unroll
                for (int i = 0; i < 2; ++i) sc[i][0] = sc[i][1] = sc[i][2] = sc[i][3] = 0.f;
                {
                    const int mi = lane >> 3, r8 = lane & 7;
                    const int key = r0 + (mi >> 1) * 8 + r8;
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks) {
                        const int chunkc = 2 * ks + (mi & 1);
                        uint32_t b0, b1, b2, b3;
                        ldmatrix_x4(st + stage_off(key, chunkc), b0, b1, b2, b3);
                        mma_16816(sc[0], qa[ks][0], 0u, qa[ks][1], 0u, b0, b1);
                        mma_16816(sc[1], qa[ks][0], 0u, qa[ks][1], 0u, b2, b3);
                    }
                }
                // ---- online softmax of head `row` over the tile's keys -------------------------------------------
                float tmax = -INFINITY;
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int cc = 0; cc < 2; ++cc) {
                        const int j = j0 + i * 8 + qd * 2 + cc;
                        float v = sc[i][cc] * a.scale_log2;
                        if (j >= lne) v = -INFINITY;
                        sc[i][cc] = v;
                        tmax = fmaxf(tmax, v);
                        if (a.acc_score && row < G && j < lne) {
                            if (a.logit_keys) s_logit[row * a.logit_keys + (j - t_lo * kTileKeys)] = v;
                            else a.ws_s[(int64_t)(b * H + h0 + row) * cap + j] = v;
                        }
                    }
                tmax = fmaxf(tmax, __shfl_xor_sync(0xFFFFFFFFu, tmax, 1));
                tmax = fmaxf(tmax, __shfl_xor_sync(0xFFFFFFFFu, tmax, 2));
                const float m_new = fmaxf(m_run, tmax);          // finite: every tile has a valid key
                const float corr = exp2f(m_run - m_new);
                m_run = m_new;
                float p[2][2];
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int cc = 0; cc < 2; ++cc) p[i][cc] = exp2f(sc[i][cc] - m_new);
                l_run = l_run * corr + (p[0][0] + p[0][1]) + (p[1][0] + p[1][1]);
#pragma unroll
                for (int i = 0; i < 16; ++i) { o[i][0] *= corr; o[i][1] *= corr; }
                // ---- O += P V -----------------------------------------------------------------------------------
                // P is split into a bf16 head and a bf16 remainder so that the product keeps ~16 bits
                const uint32_t pa0 = pack_bf16(p[0][0], p[0][1]), pa2 = pack_bf16(p[1][0], p[1][1]);
                const uint32_t pr0 = pack_bf16(p[0][0] - bf16_lo(pa0), p[0][1] - bf16_hi(pa0));
                const uint32_t pr2 = pack_bf16(p[1][0] - bf16_lo(pa2), p[1][1] - bf16_hi(pa2));
                {
                    const int mi = lane >> 3, r8 = lane & 7;
                    const int key = r0 + (mi & 1) * 8 + r8;
#pragma unroll
                    for (int dp = 0; dp < 8; ++dp) {
                        const int chunkc = 2 * dp + (mi >> 1);
                        uint32_t b0, b1, b2, b3;
                        ldmatrix_x4_trans(st + 2 * kBoxBytes + stage_off(key, chunkc), b0, b1, b2, b3);
                        // rows 8..15 of the MMA tile are padding: their accumulators are thrown away
                        float d0[4] = {o[2 * dp][0], o[2 * dp][1], 0.f, 0.f};
                        float d1[4] = {o[2 * dp + 1][0], o[2 * dp + 1][1], 0.f, 0.f};
                        mma_16816(d0, pa0, 0u, pa2, 0u, b0, b1);
                        mma_16816(d1, pa0, 0u, pa2, 0u, b2, b3);
                        mma_16816(d0, pr0, 0u, pr2, 0u, b0, b1);
                        mma_16816(d1, pr0, 0u, pr2, 0u, b2, b3);
                        o[2 * dp][0] = d0[0]; o[2 * dp][1] = d0[1];
                        o[2 * dp + 1][0] = d1[0]; o[2 * dp + 1][1] = d1[1];
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_empty[s % kStagesDec]);
        }
    }
    // ---- merge the four warps in warp order ------------------------------------------------------------
    // A warp parks its output where its own K rows of the last stage lay (nobody else reads those, and nothing is fetched there
    // any more): heads 0..3 in the box of the low channels, heads 4..7 in the other; pairs of channels, XOR-swizzled by head.
    l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 1);
    l_run += __shfl_xor_sync(0xFFFFFFFFu, l_run, 2);
    const uint32_t last = (uint32_t)((nstage > 0 ? nstage - 1 : 0) % kStagesDec) * kStageBytes;
    auto slot_of = [&](int w, int hh, int pair) {
        return reinterpret_cast<float2*>(smem + last + (hh >> 2) * kBoxBytes + w * kTileKeys * 128 + (hh & 3) * 512) + (pair ^ ((hh & 3) * 4));
    };
    if (warp < kDecWarps && row < G) {
        if (qd == 0) s_wml[warp * 8 + row] = make_float2(m_run, l_run);
#pragma unroll
        for (int i = 0; i < 16; ++i) *slot_of(warp, row, i * 4 + qd) = make_float2(o[i][0], o[i][1]);
    }
    __syncthreads();
    if (s_abort) {                             // a wait gave up: copies may still be in flight, let them land
#pragma unroll 1
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
        __syncthreads();
    }
    for (int idx = tid; idx < G * (kHeadDim / 2); idx += kDecThreads) {
        const int hh = idx >> 6, pair = idx & 63;
        float2 ml[kDecWarps], x[kDecWarps];
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) { ml[w] = s_wml[w * 8 + hh]; x[w] = *slot_of(w, hh, pair); }
        float M2 = -INFINITY, Ls = 0.f;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) M2 = fmaxf(M2, ml[w].x);
        float2 v = make_float2(0.f, 0.f);
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) {
            const float f = ml[w].x > -INFINITY ? exp2f(ml[w].x - M2) : 0.f;
            v.x += x[w].x * f; v.y += x[w].y * f; Ls += ml[w].y * f;
        }
        if (MODE == kDecParts) reinterpret_cast<float2*>(a.part_o)[((int64_t)hd * S + rank) * (G * 64) + idx] = v;
        else s_res[idx] = v;
        if (pair == 0) {
            if (MODE == kDecParts) a.part_ml[((int64_t)hd * S + rank) * G + hh] = make_float2(M2, Ls);
            s_ML[hh] = make_float2(M2, Ls);
        }
    }
    if (MODE == kDecParts) {
        if (rank == 0 && tid == 0) a.part_len[hd] = app ? ln : -1;
        store_appended();
        return;
    }

    // ---- combine the CTAs of the cluster in rank order through distributed shared memory ----------------
    if (CL) cluster_barrier(); else __syncthreads();
    // my slice of the output: pairs of channels rank * kDecThreads + tid (+ S * kDecThreads ...) of the G heads.  A thread fetches
    // what it needs from every CTA in one go (max, sum and its channels) and works out the weights itself, so there is one
    // round trip and no block barrier on this path.
    for (int idx = rank * kDecThreads + tid; idx < G * (kHeadDim / 2); idx += S * kDecThreads) {
        const int hh = idx >> 6;
        float2 x[kDecMaxCluster], ml[kDecMaxCluster];
#pragma unroll
        for (int r = 0; r < kDecMaxCluster; ++r) {
            x[r] = make_float2(0.f, 0.f); ml[r] = make_float2(-INFINITY, 0.f);
            if (r < S) {
                if (CL) {
                    x[r] = cluster_ld(s_res + idx, r);
                    ml[r] = cluster_ld(s_ML + hh, r);
                } else {                       // a head with one CTA: its own shared memory, read directly
                    x[r] = s_res[idx]; ml[r] = s_ML[hh];
                }
            }
        }
        float FM = -INFINITY;
#pragma unroll
        for (int r = 0; r < kDecMaxCluster; ++r) FM = fmaxf(FM, ml[r].x);
        float2 v = make_float2(0.f, 0.f);
        float Ls = 0.f;
#pragma unroll
        for (int r = 0; r < kDecMaxCluster; ++r) {
            const float w = ml[r].x > -INFINITY ? exp2f(ml[r].x - FM) : 0.f;
            v.x += x[r].x * w; v.y += x[r].y * w;
            Ls += ml[r].y * w;
        }
        const float inv = Ls > 0.f ? 1.0f / Ls : 0.f;
        reinterpret_cast<uint32_t*>(a.out + (int64_t)(b * H + h0) * kHeadDim)[idx] = pack_bf16(v.x * inv, v.y * inv);
    }
    if (a.acc_score && tid < 64) {             // cluster-wide (max, 1 / sum) of every head: thread = (head, CTA)
        const int hh = tid >> 3, r = tid & 7;
        float2 ml = make_float2(-INFINITY, 0.f);
        if (hh < G && r < S) ml = CL ? cluster_ld(s_ML + hh, r) : s_ML[hh];
        float FM = ml.x;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) FM = fmaxf(FM, __shfl_xor_sync(0xFFFFFFFFu, FM, o));
        float Ls = ml.x > -INFINITY ? ml.y * exp2f(ml.x - FM) : 0.f;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) Ls += __shfl_xor_sync(0xFFFFFFFFu, Ls, o);
        if (r == 0) { s_FM[hh] = FM; s_FI[hh] = Ls > 0.f ? 1.0f / Ls : 0.f; }
    }
    if (CL) cluster_arrive_exec();             // my reads of the other CTAs' shared memory are done
    store_appended();
    // the probabilities of my own keys go to acc_score
    if (a.acc_score) {
        __syncthreads();
        float* acc = a.acc_score + (int64_t)hd * cap;
        float il[G], mx[G];
#pragma unroll
        for (int hh = 0; hh < G; ++hh) { mx[hh] = s_FM[hh]; il[hh] = s_FI[hh]; }
        const int j_lo = t_lo * kTileKeys, j_hi = min(lne, t_hi * kTileKeys);
        // four keys per thread per round (past the end: the last key again, not stored): 4 (G + 1) independent loads in flight
        const float* ws = a.ws_s + (int64_t)(b * H + h0) * cap;
        for (int j0 = j_lo + tid; j0 < j_hi; j0 += 4 * kDecThreads) {
            float lg[4][G], old[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) old[u] = __ldcg(acc + min(j0 + u * kDecThreads, j_hi - 1));
            if (a.logit_keys) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int hh = 0; hh < G; ++hh) lg[u][hh] = s_logit[hh * a.logit_keys + min(j0 + u * kDecThreads, j_hi - 1) - j_lo];
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int hh = 0; hh < G; ++hh) lg[u][hh] = __ldcg(ws + (int64_t)hh * cap + min(j0 + u * kDecThreads, j_hi - 1));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + u * kDecThreads;
                float pr = 0.f;
#pragma unroll
                for (int hh = 0; hh < G; ++hh) pr += exp2f(lg[u][hh] - mx[hh]) * il[hh];
                if (j < j_hi) acc[j] = (app && j == ln ? 0.f : old[u]) + pr;         // a new entry starts at zero
            }
        }
    }
    if (app && rank == 0 && tid == 0) a.len[hd] = lne;    // every CTA of the cluster read it before the barrier
    if (CL) cluster_wait();                               // nobody leaves while its shared memory is still read
}

// Adds the parts of every head.  grid (G + CTAs for the keys, heads): CTA x < G finishes the output of query head x of the
// group, the others add the probabilities of the keys to acc_score, a slice at a time in turn: as many CTAs as fit the GPU
// beside the others, but eight, not one for every slice of the capacity (us a layer in a capacity of 32898 rows: 36 heads of 216
// rows 16.3 so, 8.2 now; of 32000 rows 118.8 / 118.0, with four CTAs 122.8; 16 heads of 216 rows 8.2 / 6.2).  Latency-bound (0.3 to 1 MB in all): every
// weight is worked out first, so that the loads of the parts depend on nothing - a warp takes every 16th part, a lane
// four channels - and the warps are added in warp order.
constexpr int kDecCombineThreads = 512;
constexpr int kDecSliceKeys = 2 * kDecCombineThreads;
constexpr int kDecLeastSliceCtas = 8;

template <int G>
__global__ void __launch_bounds__(kDecCombineThreads) decode_combine_kernel(const DecodeArgs a) {
    constexpr int kWarps = kDecCombineThreads / 32;
    __shared__ float s_M[G], s_I[G];
    __shared__ float s_w[kDecTargetCtas];                  // this query head's weight of every part
    __shared__ float4 s_o[kWarps][32];
    pdl_enter();
    const int hd = blockIdx.y, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, S = a.S;
    const float2* ml = a.part_ml + (int64_t)hd * S * G;
    const int app_at = a.part_len[hd];
    // every warp takes one of the query heads this CTA needs: (max, 1/sum) over the parts
    const bool finish = (int)blockIdx.x < G;
    const int first_key = ((int)blockIdx.x - G) * kDecSliceKeys, key_step = ((int)gridDim.x - G) * kDecSliceKeys;
    // (a.acc_score) where a row was appended another CTA bumps len meanwhile: part_len tells the keys then
    const int lne = finish ? 0 : app_at >= 0 ? app_at + 1 : a.len[hd];
    if (!finish && (lne <= first_key || lne > a.cap)) return;          // no keys for this CTA, or the head was skipped
    const int hh_w = finish ? (int)blockIdx.x : warp;
    if (finish ? warp == 0 : warp < G) {
        float m[(kDecTargetCtas + 31) / 32], l[(kDecTargetCtas + 31) / 32], M = -INFINITY, Ls = 0.f;
#pragma unroll
        for (int u = 0; u < (kDecTargetCtas + 31) / 32; ++u) {
            const int p = u * 32 + lane;
            const float2 v = p < S ? ml[p * G + hh_w] : make_float2(-INFINITY, 0.f);
            m[u] = v.x; l[u] = v.y;
            M = fmaxf(M, v.x);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
#pragma unroll
        for (int u = 0; u < (kDecTargetCtas + 31) / 32; ++u) {
            const int p = u * 32 + lane;
            const float w = m[u] > -INFINITY ? exp2f(m[u] - M) : 0.f;
            Ls += l[u] * w;
            if (finish && p < S) s_w[p] = w;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) Ls += __shfl_xor_sync(0xFFFFFFFFu, Ls, o);
        if (lane == 0) { s_M[hh_w] = M; s_I[hh_w] = Ls > 0.f ? 1.0f / Ls : 0.f; }
    }
    __syncthreads();
    const int b = hd / a.Hkv, h0 = (hd % a.Hkv) * G;
    if (finish) {
        const int hh = blockIdx.x;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int p0 = warp; p0 < S; p0 += 8 * kWarps) {
            float4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int p = p0 + u * kWarps;
                x[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (p < S && s_w[p] > 0.f)                 // (a part without keys has written no output)
                    x[u] = __ldcg(reinterpret_cast<const float4*>(a.part_o + (((int64_t)hd * S + p) * G + hh) * kHeadDim) + lane);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int p = p0 + u * kWarps;
                const float w = p < S ? s_w[p] : 0.f;
                v.x += x[u].x * w; v.y += x[u].y * w; v.z += x[u].z * w; v.w += x[u].w * w;
            }
        }
        s_o[warp][lane] = v;
        __syncthreads();
        if (tid < kHeadDim) {
            float r = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) r += reinterpret_cast<const float*>(s_o[w])[tid];
            a.out[(int64_t)(b * a.H + h0 + hh) * kHeadDim + tid] = __float2bfloat16_rn(r * s_I[hh]);
        }
        if (hh == 0 && tid == 0 && app_at >= 0) a.len[hd] = app_at + 1;
        return;
    }
    float* acc = a.acc_score + (int64_t)hd * a.cap;
    for (int j0 = first_key; j0 < lne; j0 += key_step) {
        float lg[2][G], old[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int j = j0 + u * kDecCombineThreads + tid;
            old[u] = 0.f;
#pragma unroll
            for (int hh = 0; hh < G; ++hh) lg[u][hh] = j < lne ? __ldcg(a.ws_s + (int64_t)(b * a.H + h0 + hh) * a.cap + j) : 0.f;
            if (j < lne && j != app_at) old[u] = acc[j];   // a new entry starts at zero
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int j = j0 + u * kDecCombineThreads + tid;
            float pr = 0.f;
#pragma unroll
            for (int hh = 0; hh < G; ++hh) pr += exp2f(lg[u][hh] - s_M[hh]) * s_I[hh];
            if (j < lne) acc[j] = old[u] + pr;
        }
    }
}

template <int G>
static lvlm_status launch_decode(const void* q, void* Kc, void* Vc, int32_t* len, const void* k_new,
                                 const void* v_new, float* acc_score, const lvlm_dims* d, float scale,
                                 void* out, char* wsb, const DecodeLayout& L, int64_t kv_sb,
                                 int64_t kv_sh, int32_t* dev_status, cudaStream_t stream) {
    // scaled logits of a CTA's own keys stay in shared memory when the longest run fits the budget
    const int nt_max = (d->cap + kTileKeys - 1) / kTileKeys;
    const bool parts = L.P > 0;
    const int S = parts ? L.P : L.S;
    int per = (nt_max + S - 1) / S;
    if (per >= kDecWarps) per = (per + kDecWarps - 1) / kDecWarps * kDecWarps;
    const int run_keys = per * kTileKeys;
    const int logit_keys = acc_score && !parts && (size_t)G * run_keys * 4 <= (size_t)kDecLogitBytes ? run_keys : 0;
    const size_t smem = 1024 + (size_t)kRingBytes + (size_t)(2 * kDecWarps * 8 + 4 * 8) * 4 +
                        (size_t)(2 * kStagesDec + 1) * 8 + (size_t)G * logit_keys * 4;
    CUtensorMap kmap, vmap;
    {
        const uint64_t dims[4] = {(uint64_t)kHeadDim, (uint64_t)d->cap, (uint64_t)d->Hkv, (uint64_t)d->B};
        const uint64_t strides[3] = {(uint64_t)kHeadDim * 2, (uint64_t)kv_sh * 2, (uint64_t)kv_sb * 2};
        const uint32_t box[4] = {64, (uint32_t)kStageKeys, 1, 1};
        if (!make_tmap_bf16(&kmap, Kc, 4, dims, strides, box) || !make_tmap_bf16(&vmap, Vc, 4, dims, strides, box))
            return LVLM_ERR_CUDA;
    }
    const int64_t ctas = (int64_t)d->B * d->Hkv * S;
    if (ctas > 0x7FFFFFFFll) return LVLM_ERR_UNSUPPORTED;
    DecodeArgs a;
    a.q = static_cast<const __nv_bfloat16*>(q);
    a.Kc = static_cast<__nv_bfloat16*>(Kc);
    a.Vc = static_cast<__nv_bfloat16*>(Vc);
    a.len = len;
    a.k_new = static_cast<const __nv_bfloat16*>(k_new);
    a.v_new = static_cast<const __nv_bfloat16*>(v_new);
    a.acc_score = acc_score;
    a.out = static_cast<__nv_bfloat16*>(out);
    a.H = d->H; a.Hkv = d->Hkv; a.cap = d->cap; a.S = S;
    a.early = d->cache_stable != 0 && pdl_enabled();
    a.kv_sb = kv_sb; a.kv_sh = kv_sh; a.scale_log2 = scale * kLog2e;
    a.ws_s = acc_score ? reinterpret_cast<float*>(wsb + L.off_s) : nullptr;
    a.logit_keys = logit_keys;
    a.dev_status = dev_status;
#ifdef LVLM_TEST_HOOKS
    a.starve = g_decode_starve;
#endif
    a.part_ml = reinterpret_cast<float2*>(wsb + L.off_ml);
    a.part_o = reinterpret_cast<float*>(wsb + L.off_o);
    a.part_len = reinterpret_cast<int32_t*>(wsb + L.off_len);
    void (*kernel)(CUtensorMap, CUtensorMap, DecodeArgs) =
        parts ? decode_cluster_kernel<G, kDecParts> : S == 1 ? decode_cluster_kernel<G, kDecSolo> : decode_cluster_kernel<G, kDecCluster>;
    LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem));
    const lvlm_status st = launch_kernel(kernel, dim3((unsigned)ctas), dim3(kDecThreads), smem, stream, parts ? 1 : S, kmap, vmap, a);
    if (st != LVLM_OK || !parts) return st;
    const int heads = d->B * d->Hkv;                       // (at most kDecTargetCtas / kDecMaxCluster here)
    int slices = 0;
    if (acc_score) {
        const int most = (d->cap + kDecSliceKeys - 1) / kDecSliceKeys, room = kDecTargetCtas / heads - G;
        slices = room > kDecLeastSliceCtas ? room : kDecLeastSliceCtas;
        slices = slices < most ? slices : most;
    }
    return launch_kernel(decode_combine_kernel<G>, dim3((unsigned)(G + slices), (unsigned)heads), dim3(kDecCombineThreads),
                         0, stream, 1, a);
}

static lvlm_status decode_attn(const void* q, void* Kc, void* Vc, int32_t* len, const void* k_new, const void* v_new,
                               float* acc_score, const lvlm_dims* d, float scale, void* out, void* ws, size_t ws_bytes,
                               int32_t* dev_status, cudaStream_t stream) {
    DecodeLayout L;
    if (!q || !Kc || !Vc || !len || !out || !decode_layout(d, &L, acc_score != nullptr, true)) return LVLM_ERR_INVALID_ARG;
    if ((k_new == nullptr) != (v_new == nullptr)) return LVLM_ERR_INVALID_ARG;
    const int G = d->H / d->Hkv;
    if (d->D != kHeadDim || G > kMaxGroup) return LVLM_ERR_UNSUPPORTED;
    const int64_t kv_sh = d->kv_stride_h ? d->kv_stride_h : (int64_t)d->cap * d->D;
    const int64_t kv_sb = d->kv_stride_b ? d->kv_stride_b : (int64_t)d->Hkv * kv_sh;
    if (!aligned16(q) || !aligned16(Kc) || !aligned16(Vc) || !aligned16(out) || !aligned16(k_new) ||
        !aligned16(v_new) || kv_sh % 8 || kv_sb % 8)
        return LVLM_ERR_ALIGNMENT;
    if (!ws || !aligned256(ws) || ws_bytes < L.logits) return LVLM_ERR_WORKSPACE;
    if (ws_bytes < L.used) decode_layout(d, &L, acc_score != nullptr, false);        // without room for parts: no parts
    char* wsb = static_cast<char*>(ws);
#define LVLM_DEC_CASE(GG)                                                                         \
    case GG: return launch_decode<GG>(q, Kc, Vc, len, k_new, v_new, acc_score, d, scale, out, wsb, \
                                      L, kv_sb, kv_sh, dev_status, stream)
    switch (G) {
        LVLM_DEC_CASE(1); LVLM_DEC_CASE(2); LVLM_DEC_CASE(3); LVLM_DEC_CASE(4);
        LVLM_DEC_CASE(5); LVLM_DEC_CASE(6); LVLM_DEC_CASE(7); LVLM_DEC_CASE(8);
    }
#undef LVLM_DEC_CASE
    return LVLM_ERR_UNSUPPORTED;
}

}  // namespace lvlm

#ifdef LVLM_TEST_HOOKS
extern "C" void lvlm_debug_starve_decode(int on) { lvlm::g_decode_starve = on ? 1 : 0; }
#endif

extern "C" lvlm_status lvlm_decode_attn(const void* q, void* Kc, void* Vc, int32_t* len,
                                         const void* k_new, const void* v_new, float* acc_score,
                                         const lvlm_dims* d, float scale, void* out, void* ws,
                                         size_t ws_bytes, int32_t* dev_status, void* stream_) {
    return lvlm::decode_attn(q, Kc, Vc, len, k_new, v_new, acc_score, d, scale, out, ws, ws_bytes, dev_status,
                             (cudaStream_t)stream_);
}

// ---- decode attention for callers that cannot allocate ------------------------------------------
// Scratch of lvlm_decode_attn_static: one array per GPU that loads the library, held until the
// process exits.  In host code the name below is only a handle for cudaGetSymbolAddress, never a
// pointer a kernel may be given.
static __device__ __align__(256) unsigned char g_decode_static_scratch[LVLM_STATIC_SCRATCH_BYTES];

namespace lvlm {

constexpr int kMaxStaticDevices = 64;
static void* g_static_scratch_ptr[kMaxStaticDevices];     // device address of the array, per device
static std::mutex g_static_scratch_mutex;

// Device address of the scratch array on the current device, looked up once per device.
static lvlm_status static_scratch_address(void** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxStaticDevices) return LVLM_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
    if (!g_static_scratch_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_decode_static_scratch) != cudaSuccess || !p) return LVLM_ERR_CUDA;
        g_static_scratch_ptr[dev] = p;
    }
    *out = g_static_scratch_ptr[dev];
    return LVLM_OK;
}

}  // namespace lvlm

extern "C" lvlm_status lvlm_decode_attn_static(const void* q, void* Kc, void* Vc, int32_t* len,
                                                const void* k_new, const void* v_new,
                                                float* acc_score, const lvlm_dims* d, float scale,
                                                void* out, int32_t* dev_status, void* stream) {
    using namespace lvlm;
    DecodeLayout L;
    if (!decode_layout(d, &L, false, false)) return LVLM_ERR_INVALID_ARG;
    if (L.logits > (size_t)LVLM_STATIC_SCRATCH_BYTES) return LVLM_ERR_WORKSPACE;
    void* scratch = nullptr;
    const lvlm_status st = static_scratch_address(&scratch);
    if (st != LVLM_OK) return st;
    return decode_attn(q, Kc, Vc, len, k_new, v_new, acc_score, d, scale, out, scratch,
                       (size_t)LVLM_STATIC_SCRATCH_BYTES, dev_status, (cudaStream_t)stream);
}
