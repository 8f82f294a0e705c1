// lvlm_score_tokens with ONE pass over Q K^T: a cluster of CTAs holds all logits of a query tile in its tensor memory.
//
// A CTA has up to four tiles of 128 keys.  For a tile of 128 query rows
//   S = Q_tile K_tile^T on tcgen05, queries on the TMEM lanes,
//   every logit is replaced in tensor memory by E = 2^(logit - m), m the largest one that the same thread has of the row,
//   (max, sum) of every row go to all CTAs of the cluster (st.async into their shared memory),
//   from those of all keys follows what the E of a thread's part of a row have to be weighted with, and the weighted column sums
//   are the scores.
// So a logit costs one exponential and one MMA instead of two, and two launches (this one and score_sum_kernel) do instead
// of four.  A thread has four rows x 32 columns of a tile, in pairs of columns (tcgen05.ld.16x256b): maxima and sums of a row are its
// own but for four shuffles, and a column takes four multiplications and 7/8 of a shuffle.
//
// Against sums in 64 bits the scores are off by 6e-8 to 1.2e-7 of their norm (nine sizes of 300 to 4096 keys), those of two passes by 8e-8 to
// 1.5e-7: an exponential's argument is small where the exponential is not.  (test_score_one_pass and test_score_two_passes hold both
// below 2^-21.)
//
// Roles as in score_tc.cu: a TMA warp, two MMA-issuing warps, a finisher warp, and sixteen epilogue warps in four sets, each
// with an accumulator.  With few key tiles a CTA the sets form teams that work on query tiles in turn, so that the exponentials
// of one run while another waits for its sums.  The K tiles of a KV group stay for all its query tiles.
#include <mutex>

#include "common.cuh"
#include "exp2.cuh"
#include "score.cuh"
#include "sm100.cuh"

namespace lvlm {

using namespace sm100;

constexpr int kOTile = 128;
constexpr int kOHalf = kOTile * 64 * 2, kOTileBytes = 2 * kOHalf;
constexpr int kOSets = 4, kOEpiWarps = 4 * kOSets, kOThreads = (4 + kOEpiWarps) * 32;   // warps: TMA, MMA, finisher, MMA, epilogue
constexpr int kOMaxCluster = 8;
constexpr int kOQSlots = 2;
constexpr int kOSmCount = 148;
constexpr int kOnceScoreSmem = 227 * 1024;
constexpr float kLog2eO = 1.4426950408889634f;

struct OnceScoreArgs {
    int G, Hkv, N, Nq, i0, n, q_lo, causal;
    int box_h, box_p, nh, tpg;
    int S, kt, teams, k_slots, parts, runs, clusters;
    FastDiv by_nh, by_box_h, by_parts, by_hkv;
    float scale_log2;
    float* partial; int64_t row_len;   // [B][Hkv * parts][row_len] column sums
    int32_t* dev_status;
#ifdef LVLM_TEST_HOOKS
    int starve;
#endif
};

// The test build can keep the first CTA of every cluster from sending, so that all of them wait for sums that never come.
#ifdef LVLM_TEST_HOOKS
static int g_score_starve = 0;
__device__ __forceinline__ bool once_starved(const OnceScoreArgs& a, int cr) { return a.starve != 0 && cr == 0; }
#else
__device__ __forceinline__ bool once_starved(const OnceScoreArgs&, int) { return false; }
#endif

struct OnceCtl {
    uint64_t q_full[kOQSlots], q_empty[kOQSlots], k_full[4], k_empty[4], acc_full[kOSets], acc_empty[kOSets];
    uint64_t recv[kOSets][2][4];       // [team][buffer][quarter of the rows]
    uint64_t meet[kOSets][4];          // the kt warps of a team that have the same rows
    uint64_t res_full[2], res_empty[2];
    uint32_t tmem_base;
    volatile int abort;
};

__device__ __forceinline__ void tmem_st_16x256b_x4(uint32_t taddr, const float* v) {
    const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// 32 TMEM lanes x 32 columns: v[16 (half of the lanes) + 4 (8-column group) + 2 (row, row + 8) + pair].
__device__ __forceinline__ void once_ld(uint32_t taddr, float* v) {
    tmem_ld_16x256b_x4(taddr, v);
    tmem_ld_16x256b_x4(taddr + (16u << 16), v + 16);
}
__device__ __forceinline__ constexpr int once_at(int k, int i) { return (k >> 1) * 16 + (i >> 1) * 4 + (k & 1) * 2 + (i & 1); }

__device__ __forceinline__ bool once_give_up(OnceCtl* sm, int32_t* dev_status) {
    sm->abort = 1;
    if (dev_status) atomicOr(dev_status, LVLM_DEV_TIMEOUT);
    return false;
}
__device__ __forceinline__ bool once_wait(uint64_t* bar, uint32_t parity, OnceCtl* sm, int32_t* dev_status) {
    if (mbar_try(bar, parity)) return true;
    if (sm->abort) return false;
    return mbar_wait(bar, parity) || once_give_up(sm, dev_status);
}

// The query tiles of my cluster, in order: runs [run, end) of query tiles of a KV group.
struct OnceTiles {
    const OnceScoreArgs& a;
    int run, end;
    int bg = -1, t = 0, t1 = 0;        // KV group (all sequences), query tile of it, end of the run
    bool new_group = false, last_of_run = false, last_of_group = false;
    __device__ explicit OnceTiles(const OnceScoreArgs& a_) : a(a_) {
        const int c = (int)blockIdx.x / a.S;
        run = (int)((int64_t)a.runs * c / a.clusters) - 1;
        end = (int)((int64_t)a.runs * (c + 1) / a.clusters);
    }
    __device__ bool next() {
        new_group = false;
        if (t + 1 < t1) {
            ++t;
        } else {
            if (++run >= end) return false;
            int part;
            const int x = a.by_parts.divmod(run, &part);
            new_group = x != bg;
            bg = x;
            t = a.by_parts.div(a.tpg * part);
            t1 = a.by_parts.div(a.tpg * (part + 1));
        }
        last_of_run = t + 1 >= t1;
        last_of_group = last_of_run && (run + 1 >= end || a.by_parts.div(run + 1) != bg);
        return true;
    }
};

// (max, sum) of a row over `cnt` <= MOST sets of keys, `step` apart.
template <int MOST>
__device__ __forceinline__ float2 join_stats(const float2* st, int step, int cnt) {
    float2 e[MOST];
#pragma unroll
    for (int i = 0; i < MOST; ++i) e[i] = i < cnt ? st[i * step] : make_float2(-INFINITY, 0.f);
    float M = e[0].x, L = 0.f;
#pragma unroll
    for (int i = 1; i < MOST; ++i) M = fmaxf(M, e[i].x);
    const float ref = M == -INFINITY ? 0.f : M;
#pragma unroll
    for (int i = 0; i < MOST; ++i)
        if (i < cnt) L = fmaf(e[i].y, ex2_fast(e[i].x - ref), L);
    return make_float2(M, L);
}

__global__ void __launch_bounds__(kOThreads, 1)
score_once_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap, const OnceScoreArgs a) {
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
    const int kt = a.kt, teams = a.teams, S = a.S, k_slots = a.k_slots;
    unsigned char* sQ = base;                                            // [kOQSlots] tiles
    unsigned char* sK = sQ + kOQSlots * kOTileBytes;                     // [k_slots] tiles
    float2* s_recv = reinterpret_cast<float2*>(sK + k_slots * kOTileBytes);              // [teams][2][S][128]
    float2* s_stat = s_recv + (size_t)teams * 2 * S * kOTile;                            // [2][sets][128]
    float* s_res = reinterpret_cast<float*>(s_stat + 2 * kOSets * kOTile);               // [res_bufs][sets][4][128]
    const int res_bufs = teams > 1 ? 2 : 1;
    OnceCtl* sm = reinterpret_cast<OnceCtl*>(s_res + (size_t)res_bufs * kOSets * 4 * kOTile);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cr = (int)cluster_ctarank(), sets = teams * kt;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kOQSlots; ++s) { mbar_init(&sm->q_full[s], 1); mbar_init(&sm->q_empty[s], 2); }
        for (int s = 0; s < 4; ++s) { mbar_init(&sm->k_full[s], 1); mbar_init(&sm->k_empty[s], 2); }
        for (int s = 0; s < kOSets; ++s) {
            mbar_init(&sm->acc_full[s], 1); mbar_init(&sm->acc_empty[s], 4);
            for (int x = 0; x < 8; ++x) mbar_init(&sm->recv[s][x >> 2][x & 3], 1);
            for (int x = 0; x < 4; ++x) mbar_init(&sm->meet[s][x], (uint32_t)kt);
        }
        for (int s = 0; s < 2; ++s) { mbar_init(&sm->res_full[s], (uint32_t)(sets * 4)); mbar_init(&sm->res_empty[s], 1); }
        sm->abort = 0;
        fence_barrier_init();
        prefetch_tmap(&qmap);
        prefetch_tmap(&kmap);
    }
    // rows of a query tile that no copy ever writes: their logits count for nothing, but have to be numbers
    const int box_rows = a.box_h * a.box_p;
    if (box_rows < kOTile) {
        for (int e = threadIdx.x; e < (kOTile - box_rows) * 8 * kOQSlots * 2; e += kOThreads) {
            const int x = e / (kOQSlots * 2);
            *reinterpret_cast<uint4*>(sQ + (e - x * (kOQSlots * 2)) * kOHalf + (box_rows + (x >> 3)) * 128 + (x & 7) * 16) = make_uint4(0, 0, 0, 0);
        }
    }
    fence_proxy_async();
    if (warp == 1) tmem_alloc(&sm->tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (S > 1)                                 // (a CTA's barriers are there before anybody sends to them)
        cluster_barrier();
    const uint32_t tmem_base = sm->tmem_base;
    pdl_enter();

    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            const uint32_t q_bytes = (uint32_t)box_rows * 256;
            OnceTiles w(a);
            int kslot = 0, kround = 0;
            bool ok = true;
            for (int x = 0; ok && w.next(); ++x) {
                int g, hb;
                const int b = a.by_hkv.divmod(w.bg, &g), qs = x % kOQSlots;
                if (x >= kOQSlots) ok = once_wait(&sm->q_empty[qs], ((x / kOQSlots) - 1) & 1, sm, a.dev_status);
                if (!ok) break;
                const int pt = a.by_nh.divmod(w.t, &hb), hh = g * a.G + hb * a.box_h, pos = pt * a.box_p;
                mbar_arrive_expect_tx(&sm->q_full[qs], q_bytes);
                tma_load_4d(sQ + qs * kOTileBytes, &qmap, &sm->q_full[qs], 0, hh, pos, b);
                tma_load_4d(sQ + qs * kOTileBytes + kOHalf, &qmap, &sm->q_full[qs], 64, hh, pos, b);
                if (!w.new_group) continue;
                for (int i = 0; i < kt; ++i) {
                    if (kround > 0) ok = once_wait(&sm->k_empty[kslot], (kround - 1) & 1, sm, a.dev_status);
                    if (!ok) break;
                    unsigned char* dst = sK + kslot * kOTileBytes;
                    const int row = (cr * kt + i) * kOTile;
                    mbar_arrive_expect_tx(&sm->k_full[kslot], kOTileBytes);
                    tma_load_4d(dst, &kmap, &sm->k_full[kslot], 0, row, g, b);
                    tma_load_4d(dst + kOHalf, &kmap, &sm->k_full[kslot], 64, row, g, b);
                    if (++kslot == k_slots) { kslot = 0; ++kround; }
                }
                // the next group's tiles into L2 meanwhile: their slots are free only once this group's MMAs are done
                if ((w.bg + 1) * a.parts < w.end) {
                    int g2;
                    const int b2 = a.by_hkv.divmod(w.bg + 1, &g2);
                    for (int i = 0; i < kt; ++i) {
                        const int row = (cr * kt + i) * kOTile;
                        if (row >= a.N) break;
                        tma_prefetch_4d(&kmap, 0, row, g2, b2);
                        tma_prefetch_4d(&kmap, 64, row, g2, b2);
                    }
                    tma_prefetch_4d(&qmap, 0, g2 * a.G, 0, b2);
                    tma_prefetch_4d(&qmap, 64, g2 * a.G, 0, b2);
                }
            }
        }
    } else if (warp == 1 || warp == 3) {
        // ================= MMA issuers =================
        // One has the accumulators of even, the other those of odd number: issuing the MMAs of a tile keeps a warp for as long as
        // they take, and its waits another few hundred cycles.  Both wait for, and declare done with, every tile of both rings, so
        // that neither can be a generation ahead.  (All lanes run the loop, one elected lane issues.)
        constexpr uint32_t idesc = idesc_bf16_f32(kOTile, kOTile);
        const uint64_t qd0 = smem_desc_sw128(smem_u32(sQ)), kd0 = smem_desc_sw128(smem_u32(sK));
        const int me = warp == 1 ? 0 : 1;
        OnceTiles w(a);
        int first = 0, first_round = 0, nslot = 0, nround = 0;           // ring position of the group's first K tile, and behind its last
        int team = 0, y = 0;                                             // whose turn it is, and how many it has had
        bool ok = true;
        for (int x = 0; ok && w.next(); ++x) {
            const int qs = x % kOQSlots;
            if (w.new_group) { first = nslot; first_round = nround; }
            ok = once_wait(&sm->q_full[qs], (x / kOQSlots) & 1, sm, a.dev_status);
            int slot = first, round = first_round;
            for (int i = 0; i < kt; ++i) {
                const int s = team * kt + i;
                const bool mine = (s & 1) == me;
                if (ok && w.new_group) ok = once_wait(&sm->k_full[slot], round & 1, sm, a.dev_status);
                if (ok && mine && y > 0) ok = once_wait(&sm->acc_empty[s], (y - 1) & 1, sm, a.dev_status);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) break;
                tc_fence_after();
                if (elect_one()) {
                    if (mine) {
                        const uint64_t qd = qd0 + (uint32_t)(qs * (kOTileBytes >> 4)), kd = kd0 + (uint32_t)(slot * (kOTileBytes >> 4));
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            const uint32_t off = ((k >> 2) * kOHalf + (k & 3) * 32) >> 4;
                            mma_bf16_ss(tmem_base + s * kOTile, qd + off, kd + off, idesc, k > 0 ? 1u : 0u);
                        }
                        mma_commit(&sm->acc_full[s]);
                    }
                    if (w.last_of_group) mma_commit(&sm->k_empty[slot]);
                    if (i + 1 == kt) mma_commit(&sm->q_empty[qs]);
                }
                __syncwarp();
                if (++slot == k_slots) { slot = 0; ++round; }
            }
            nslot = slot; nround = round;
            if (++team == teams) { team = 0; ++y; }
        }
    } else if (warp == 2) {
        // ================= finisher: column sums of a run, all row quarters and teams, in a fixed order =================
        OnceTiles w(a);
        int rr = 0;
        while (w.next()) {
            if (!w.last_of_run) continue;
            const int rb = res_bufs > 1 ? (rr & 1) : 0, use = res_bufs > 1 ? rr >> 1 : rr;
            ++rr;
            if (!__all_sync(0xFFFFFFFFu, once_wait(&sm->res_full[rb], use & 1, sm, a.dev_status))) break;
            int part;
            a.by_parts.divmod(w.run, &part);
            float* row = a.partial + ((int64_t)w.bg * a.parts + part) * a.row_len;
            for (int i = 0; i < kt; ++i) {
                float sum[4] = {0.f, 0.f, 0.f, 0.f};
                for (int tm = 0; tm < teams; ++tm) {
                    const float* r = s_res + (size_t)((rb * kOSets + tm * kt + i) * 4) * kOTile + lane;
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int u = 0; u < 4; ++u) sum[u] += r[q * kOTile + u * 32];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int j = (cr * kt + i) * kOTile + u * 32 + lane - a.i0;
                    if (j >= 0 && j < a.n) row[j] = sum[u];
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm->res_empty[rb]);
        }
    } else if (((warp - 4) >> 2) < sets) {
        // ================= epilogue: set s has accumulator s; a warp the TMEM lanes 32 (warp % 4) .. + 31 =================
        const int quarter = warp & 3, s = (warp - 4) >> 2, team = s / kt, tile = s - team * kt, row0 = quarter * 32;
        const uint32_t acc = tmem_base + ((uint32_t)row0 << 16) + (uint32_t)(s * kOTile);
        const int key0 = (cr * kt + tile) * kOTile, col0 = 2 * (lane & 3);
        const f32x2 sc = both(a.scale_log2);
        OnceTiles w(a);
        float col[4] = {0.f, 0.f, 0.f, 0.f};       // column sums of the run: of column 32 c + 8 (lane / 8) + 2 (lane % 4) + (lane / 4 % 2)
        int turn = 0, y = 0, z = 0, rr = 0;        // z: query tiles of which my quarter has rows
        bool ok = true;
        while (ok && w.next()) {
            if (turn == team) {
                int hb;
                const int pt = a.by_nh.divmod(w.t, &hb), pos0 = pt * a.box_p;
                // my rows row0 + lane / 4 + 8 k see the columns below lim[k]; all rows of the warp those below `some`, one or another
                // those below `any` (rows that are not there may see what they like: they are weighted with 0)
                int lim[4], some = kOTile, any = 0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int p = a.by_box_h.div(row0 + (lane >> 2) + 8 * k);
                    const bool there = p < a.box_p && pos0 + p < a.Nq;
                    lim[k] = there ? min(max((a.causal ? min(a.N, a.q_lo + pos0 + p + 1) : a.N) - key0, 0), kOTile) : kOTile;
                    some = min(some, lim[k]);
                    any = max(any, there ? lim[k] : 0);
                }
                some = __reduce_min_sync(0xFFFFFFFFu, some);
                any = __reduce_max_sync(0xFFFFFFFFu, any);
                const int p_first = a.by_box_h.div(row0);
                const bool idle = p_first >= a.box_p || pos0 + p_first >= a.Nq;         // no such rows
                ok = __all_sync(0xFFFFFFFFu, once_wait(&sm->acc_full[s], y & 1, sm, a.dev_status));
                if (!ok) break;
                tc_fence_after();
                if (!idle) {
                    auto hide = [&](float* v, int c) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                v[once_at(k, i)] = c + 8 * (i >> 1) + col0 + (i & 1) < lim[k] ? v[once_at(k, i)] : -INFINITY;
                    };
                    // ---- the largest logit of every row among my columns ----
                    float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
                    for (int c = 0; c < any; c += 32) {
                        float v[32];
                        once_ld(acc + c, v);
                        tmem_ld_wait();
                        if (c + 32 > some) hide(v, c);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
#pragma unroll
                            for (int i = 0; i < 8; ++i) m[k] = fmaxf(m[k], v[once_at(k, i)]);
                    }
                    f32x2 neg[4], l2[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        m[k] *= a.scale_log2;                              // (a positive scale keeps the order)
                        neg[k] = both(m[k] == -INFINITY ? 0.f : -m[k]);
                        l2[k] = both(0.f);
                    }
                    // ---- 2^(logit - m), in its place ----
#pragma unroll 1
                    for (int c = 0; c < any; c += 32) {
                        float v[32];
                        once_ld(acc + c, v);
                        tmem_ld_wait();
                        if (c + 32 > some) hide(v, c);
#pragma unroll
                        for (int k = 0; k < 4; ++k)
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                float* e = v + once_at(k, 2 * i);
                                float x0, x1;
                                unpack2(fma2(pack2(e[0], e[1]), sc, neg[k]), x0, x1);
                                e[0] = ex2_fast(x0); e[1] = ex2_fast(x1);
                                l2[k] = add2(l2[k], pack2(e[0], e[1]));
                            }
                        tmem_st_16x256b_x4(acc + c, v);
                        tmem_st_16x256b_x4(acc + (16u << 16) + c, v + 16);
                    }
                    // ---- (max, sum) of a row over the tile, over the tiles of the CTA, to all CTAs ----
                    float2* stat = s_stat + ((z & 1) * kOSets + team * kt) * kOTile + row0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        float M = m[k], L, L1;
                        unpack2(l2[k], L, L1);
                        M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, 1));
                        M = fmaxf(M, __shfl_xor_sync(0xFFFFFFFFu, M, 2));
                        L = (L + L1) * ex2_fast(m[k] - (M == -INFINITY ? 0.f : M));
                        L += __shfl_xor_sync(0xFFFFFFFFu, L, 1);
                        L += __shfl_xor_sync(0xFFFFFFFFu, L, 2);
                        if ((lane & 3) == 0) stat[tile * kOTile + (lane >> 2) + 8 * k] = make_float2(M, L);
                    }
                    __syncwarp();
                    if (kt > 1) {
                        if (lane == 0) mbar_arrive(&sm->meet[team][quarter]);
                        ok = __all_sync(0xFFFFFFFFu, once_wait(&sm->meet[team][quarter], z & 1, sm, a.dev_status));
                        if (!ok) break;
                    }
                    float2 mine = join_stats<4>(stat + lane, kOTile, kt);  // row row0 + lane
                    if (S > 1) {
                        uint64_t* bar = &sm->recv[team][z & 1][quarter];
                        float2* to = s_recv + (size_t)((team * 2 + (z & 1)) * S) * kOTile + row0 + lane;
                        if (tile == 0 && lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)(S * 256));
                        const uint32_t addr = smem_u32(to + cr * kOTile), bar_addr = smem_u32(bar);
                        for (int d = once_starved(a, cr) ? S : tile; d < S; d += kt) st_async8(cluster_map(addr, (uint32_t)d), mine, cluster_map(bar_addr, (uint32_t)d));
                        ok = sm->abort ? false : mbar_wait_cluster(bar, (z >> 1) & 1) || once_give_up(sm, a.dev_status);
                        ok = __all_sync(0xFFFFFFFFu, ok);
                        if (!ok) break;
                        mine = join_stats<kOMaxCluster>(to, kOTile, S);
                    }
                    float nn = -(mine.x + log2f(mine.y));                  // minus the normaliser of the row (log2 domain)
                    {
                        const int p = a.by_box_h.div(row0 + lane);
                        if (p >= a.box_p || pos0 + p >= a.Nq) nn = -INFINITY;           // (no such row)
                    }
                    f32x2 wgt[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        wgt[k] = both(ex2_fast(m[k] + __shfl_sync(0xFFFFFFFFu, nn, (lane >> 2) + 8 * k)));
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    // ---- the column sums of my 32 rows ----
                    const bool up16 = lane & 16, up8 = lane & 8, up4 = lane & 4;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        if (c * 32 >= any) continue;
                        float u[32];
                        once_ld(acc + c * 32, u);
                        tmem_ld_wait();
                        f32x2 t[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            t[i] = mul2(pack2(u[i * 4], u[i * 4 + 1]), wgt[0]);
                            t[i] = fma2(pack2(u[i * 4 + 2], u[i * 4 + 3]), wgt[1], t[i]);
                            t[i] = fma2(pack2(u[16 + i * 4], u[16 + i * 4 + 1]), wgt[2], t[i]);
                            t[i] = fma2(pack2(u[16 + i * 4 + 2], u[16 + i * 4 + 3]), wgt[3], t[i]);
                        }
                        float f[8];
#pragma unroll
                        for (int i = 0; i < 4; ++i) unpack2(t[i], f[2 * i], f[2 * i + 1]);
                        float h[4], g[2];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {                      // upper lanes take the upper column groups
                            const float give = up16 ? f[e] : f[4 + e], keep = up16 ? f[4 + e] : f[e];
                            h[e] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, 16);
                        }
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float give = up8 ? h[e] : h[2 + e], keep = up8 ? h[2 + e] : h[e];
                            g[e] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, 8);
                        }
                        col[c] += (up4 ? g[1] : g[0]) + __shfl_xor_sync(0xFFFFFFFFu, up4 ? g[0] : g[1], 4);
                    }
                    ++z;
                }
                tc_fence_before();                                         // the accumulator may be filled again
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm->acc_empty[s]);
                ++y;
            }
            if (++turn == teams) turn = 0;
            if (w.last_of_run) {
                const int rb = res_bufs > 1 ? (rr & 1) : 0, use = res_bufs > 1 ? rr >> 1 : rr;
                ++rr;
                if (use > 0) ok = __all_sync(0xFFFFFFFFu, once_wait(&sm->res_empty[rb], (use - 1) & 1, sm, a.dev_status));
                if (!ok) break;
                float* r = s_res + (size_t)((rb * kOSets + s) * 4 + quarter) * kOTile + (lane >> 3) * 8 + col0 + ((lane >> 2) & 1);
#pragma unroll
                for (int c = 0; c < 4; ++c) { r[c * 32] = col[c]; col[c] = 0.f; }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm->res_full[rb]);
            }
        }
    }
    // ---- common exit ----
    tc_fence_before();
    __syncthreads();
    if (sm->abort) {                              // let copies still in flight land before leaving
#pragma unroll 1
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    if (S > 1)                                    // (nobody leaves while somebody may still send to it)
        cluster_barrier();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

// ---- host -------------------------------------------------------------------------------------------------------
static size_t once_smem(int k_slots, int teams, int S) {
    return 1024 + (size_t)(kOQSlots + k_slots) * kOTileBytes +
           sizeof(float2) * kOTile * ((size_t)teams * 2 * S + 2 * kOSets) + sizeof(float) * kOTile * 4 * kOSets * (teams > 1 ? 2 : 1) +
           sizeof(OnceCtl);
}
static int once_k_slots(int kt) { return kt == 1 ? 2 : kt == 2 ? 3 : 4; }
static int once_teams(int kt) { return kOSets / kt; }

// How many clusters of S CTAs the current device runs at a time; looked up once per device and size.
static int once_clusters(int S) {
    static std::mutex mu;
    static int cache[64][kOMaxCluster + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return kOSmCount / (2 * S);
    std::lock_guard<std::mutex> lock(mu);
    if (cache[dev][S] == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(S * 256));
        cfg.blockDim = dim3(kOThreads);
        cfg.dynamicSmemBytes = once_smem(4, 1, kOMaxCluster);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)S; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(score_once_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kOnceScoreSmem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, score_once_kernel, &cfg) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 128 / S;                                    // a safe guess
        }
        cache[dev][S] = n;
    }
    return cache[dev][S];
}

// Estimates in us, a fit to 17 sizes with every shape forced (1 to 16 sequences of 300 to 4096 keys, 8 to 48 heads, 17 to 256 rows).
// One pass: a query tile takes a cluster a chain of steps (MMAs, maxima, exponentials, the meeting of the CTAs, column
// sums: 7000 cycles and more with one key tile a CTA), teams overlap theirs.  Two passes: start-up and hand-overs of four launches, then 1600
// cycles a tile and SM.  us measured, two passes / one: 8 heads x 640 keys x 64 rows 12.4 / 9.2, 28 x 406 x 128 15.0 / 10.4, 28 x 1023 x
// 128 17.2 / 11.6, 28 x 3008 x 128 26.6 / 18.0, 3 sequences of 28 x 2846 x 50 29.1 / 19.9, 16 of 8 x 400 x 17 22.9 / 12.2, 16 of 32 x 1156 x
// 96 57.5 / 50.0, 2 of 32 x 4000 x 100 43.9 / 39.4; where a cluster has many query tiles the chains lose: 16 of 32 x 1888 x 96 78.9 / 82.6,
// 16 of 48 x 2000 x 100 125 / 132.  One pass has to be ahead by 7 %: between other launches it gains less than in a loop of its own (the
// 57.5 / 50.0 above made a whole two-stage reduction of 16 x 1888 rows 367 / 370 us; the reason is not measured).
OnceScoreShape score_once_shape(const lvlm_dims* d, const ScoreShape& s, float scale) {
    static const double chain[4] = {3700, 5800, 10300, 12000};             // cycles a query tile in a row of them, by key tiles a CTA
    OnceScoreShape best = {0, 0, 0, 0};
    const int keys = d->causal && d->q_hi < d->N ? d->q_hi : d->N, tiles = (keys + kOTile - 1) / kOTile;
    // (a window that starts among the scored keys sees less of them: the two passes leave out the tiles it does not see)
    if (!(scale > 0.f) || tiles > 4 * kOMaxCluster || (d->causal && d->q_lo < d->i0 + d->n)) return best;
    const int64_t groups = (int64_t)d->B * d->Hkv, key_tiles = groups * s.nkt, per_head = (int64_t)d->B * d->H * d->n / kOTile;
    const int64_t room = (s.part_tiles > per_head ? s.part_tiles : per_head) / key_tiles;
    const int most = (int)(room < 64 ? room : 64);
    double best_t = 0.93 * (14.5 + 0.85 * (double)groups * s.tpg * (tiles + s.nkt) / kOSmCount);
    for (int kt = 1; kt <= 4; ++kt) {
        const int S = (tiles + kt - 1) / kt;
        if (S > kOMaxCluster) continue;
        const int nc = once_clusters(S);
        for (int p = 1; p <= most && p <= s.tpg; ++p) {
            const int64_t runs = groups * p, rounds = (runs + nc - 1) / nc;
            const double q = (double)rounds * ((s.tpg + p - 1) / p);
            const double t = 6.5 + (5700.0 + 1300.0 * kt + (q - 1) * chain[kt - 1] + 500.0 * rounds + 10.0 * S) / 1900.0;
            if (t < best_t) { best_t = t; best.kt = kt; best.S = S; best.parts = p; best.clusters = (int)(runs < nc ? runs : nc); }
        }
    }
    return best;
}

lvlm_status launch_score_once(const CUtensorMap& qmap, const CUtensorMap& kmap, const lvlm_dims* d, const ScoreShape& s,
                              const OnceScoreShape& o, float scale, float* partial, int32_t* dev_status, cudaStream_t stream) {
    OnceScoreArgs a;
    a.G = d->H / d->Hkv; a.Hkv = d->Hkv; a.N = d->N; a.Nq = d->q_hi - d->q_lo; a.i0 = d->i0; a.n = d->n; a.q_lo = d->q_lo;
    a.causal = d->causal;
    a.box_h = s.box_h; a.box_p = s.box_p; a.nh = s.nh; a.tpg = s.tpg;
    a.S = o.S; a.kt = o.kt; a.teams = once_teams(o.kt); a.k_slots = once_k_slots(o.kt); a.parts = o.parts; a.clusters = o.clusters;
    const int64_t runs = (int64_t)d->B * d->Hkv * o.parts;
    if (runs > 0x7FFFFFFFll) return LVLM_ERR_UNSUPPORTED;
    a.runs = (int)runs;
    a.by_nh = FastDiv(s.nh); a.by_box_h = FastDiv(s.box_h); a.by_parts = FastDiv(o.parts); a.by_hkv = FastDiv(d->Hkv);
    a.scale_log2 = scale * kLog2eO;
#ifdef LVLM_TEST_HOOKS
    a.starve = g_score_starve;
#endif
    a.partial = partial; a.row_len = (int64_t)s.nkt * kOTile; a.dev_status = dev_status;
    LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(score_once_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kOnceScoreSmem));
    return launch_kernel(score_once_kernel, dim3((unsigned)(o.clusters * o.S)), dim3(kOThreads), once_smem(a.k_slots, a.teams, a.S), stream,
                         o.S, qmap, kmap, a);
}

}  // namespace lvlm

#ifdef LVLM_TEST_HOOKS
extern "C" void lvlm_debug_starve_score(int on) { lvlm::g_score_starve = on ? 1 : 0; }
#endif
