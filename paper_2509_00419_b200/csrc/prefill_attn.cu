// lvlm_prefill_attn: the causal attention of a prefill layer that hands the token reduction its scores as a
// by-product (Section 3.2.1, paragraph 3 and its footnote: the per-key summed attention comes out of the
// attention kernel that runs anyway, so no separate pass over Q K^T is paid for the row normalisers).
//
// One CTA per pair of tiles of 128 query rows that read the same keys (two heads of a KV group at the same rows, or two
// neighbouring tiles of the odd head out) or, where query tiles are few, one query tile whose key tiles are split between
// the two halves of the CTA; tcgen05 MMAs, accumulators in tensor memory.  The two tiles take turns: while
// the softmax of one works, the tensor cores multiply for the other.
//   S = Q K_j^T      A = Q tile, B = K tile, both K-major from TMA (128-byte swizzle), 128x128 fp32 in TMEM
//   softmax          four warps a tile: thread = query row; running max m and sum l in the log2 domain.  The
//                    probabilities 2^(s - m) go back into the tensor-memory columns the logits came from, as
//                    bf16 pairs (head and remainder of every probability: a plain bf16 would miss the output
//                    tolerance on rows that see few keys), so P never touches shared memory.  They are handed over in two
//                    halves of 64 keys, so that the product starts while the second half is still exponentiated.  The
//                    output accumulator is rescaled only when the maximum has grown by more than 2^8 (the stale maximum
//                    keeps every probability below 2^8, well inside bf16 and fp32); the products before are complete
//                    by then, since the MMAs of S that the softmax has waited for were issued behind them
//   O += P V_j       A = P from tensor memory, B = V tile as it lies in memory (keys x channels: an MN-major
//                    operand), 128x128 fp32 in TMEM; the next S of the tile is issued right behind it, over the P it reads
//                    (MMAs of a CTA execute in the order of their issue)
// What bounds it: the MMAs.  With P in two bf16 parts a pair of key tiles takes 3072 cycles of the tensor pipe at least;
// it takes 3960, because the MMAs of S read both operands from shared memory (104 cycles instead of 53: tensor memory
// is full with S, P and O of the two tiles, there is no room for Q) - and over milliseconds the power limit.  With one
// query tile a CTA (S, then softmax, then P V, in turns) a key tile took 2800.  us, before -> now: 28 heads x 3008 rows 131 -> 95,
// 48 x 16640 4400 -> 3900 (872 TFLOP/s), 16 sequences of 32 x 1888 950 -> 753, 28 x 600 16 -> 16.5, 28 x 1000 31 -> 25.
// At the end a thread divides its row by l, writes it, writes lse = ln sum exp of the row, and - for the rows
// of the scoring window - the log2-domain normaliser the column-sum pass of lvlm_score_tokens reads; that pass then
// runs on the same stream (keys on the TMEM lanes, see score_tc.cu) and produces score and score_head.
#include "common.cuh"
#include "exp2.cuh"
#include "score.cuh"
#include "sm100.cuh"

namespace lvlm {

using namespace sm100;

constexpr int kAT = 128;                     // query rows per CTA, keys per tile, head dim
constexpr int kAHalf = kAT * 64 * 2;         // one TMA box: 128 rows x 64 bf16 = 16 KB
constexpr int kATile = 2 * kAHalf;           // 32 KB
constexpr int kAStages = 2;                  // K ring and V ring (released separately: K after S, V after O)
constexpr int kAThreads = 128 + 2 * kAT;     // warp 0 TMA, warp 1 MMA, (2, 3 idle,) four softmax warps for each of the two tiles
// A softmax thread holds a row of 128 logits: the first warpgroup hands registers over to the other two.  Launched with
// 168 a thread (65536 / 384, rounded down to 8): 3 * 168 = 104 + 2 * 200.  What the kernel is launched with is the compiler's
// choice; with less, the two would wait for registers that nobody has, so a call looks it up first (attn_registers_fit).
constexpr int kARegsLaunch = 168, kARegsFew = 104, kARegsMany = 200;
static_assert(3 * kARegsLaunch >= kARegsFew + 2 * kARegsMany, "the split has to fit the registers the block is launched with");
constexpr uint32_t kATmemCols = 512;         // S/P of the two tiles | O of the two tiles
constexpr float kLog2eA = 1.4426950408889634f;
constexpr float kLn2A = 0.6931471805599453f;
constexpr float kRescaleStep = 8.0f;         // the output is rescaled when the row maximum has grown by more (log2)

struct AttnArgs {
    int B, H, G, Hkv, N, causal, q_lo, q_hi;
    int nqt, split;            // query tiles of a head; 1 = one query tile a CTA, its key tiles split
    float scale_log2;
    __nv_bfloat16* out; int64_t out_sb, out_sn, out_sh;   // elements
    float* lse;                // [B][H][N] natural log
    float* lse_win;            // [B][H][q_hi-q_lo] log2 domain, or NULL
    int32_t* dev_status;
};

struct AttnSmem {
    uint64_t q_full, k_full[kAStages], k_empty[kAStages], v_full[kAStages], v_empty[kAStages], s_full[2], p_ready[2][2], o_done[2];
    uint32_t tmem_base;
    volatile int abort;
    float xm[2][kAT], xl[2][kAT];   // split: (max, sum) of a row over the key tiles of either half
};

// D[tmem] (+)= A[tmem] * B[smem]^T, issued by one thread: A is 128 rows (lanes) of bf16 pairs, two K indices a column.
__device__ __forceinline__ void mma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(tmem_d), "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}

// Shared-memory descriptor of an MN-major bf16 operand stored as rows of 128 bytes (64 elements of the M or N
// dimension) with the 128-byte swizzle, one row per K index: 8 rows are one swizzle atom (stride byte offset 1024
// between atoms along K), the next 64 elements of M/N start `lbo` bytes further (leading byte offset).
__device__ __forceinline__ uint64_t smem_desc_mn_sw128(uint32_t addr, uint32_t lbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// 32 consecutive fp32 columns of this thread's TMEM lane, written back.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float* v) {
    const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
          "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
          "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
          "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ bool attn_wait(uint64_t* bar, uint32_t parity, AttnSmem* sm, int32_t* dev_status) {
    if (mbar_try(bar, parity)) return true;
    if (sm->abort) return false;
    if (mbar_wait(bar, parity)) return true;
    sm->abort = 1;
    if (dev_status) atomicOr(dev_status, LVLM_DEV_TIMEOUT);
    return false;
}

// The (up to two) tiles of a CTA: head and query tile (split: one, twice).  CTAs are numbered longest first, over all heads and sequences.
struct AttnTiles { int b, g, h[2], qt[2], n; };

__device__ __forceinline__ AttnTiles attn_tiles(const AttnArgs& a) {
    AttnTiles w;
    int i = (int)blockIdx.x;
    if (a.split) {
        const int per = a.B * a.H, t = a.nqt - 1 - i / per;
        i %= per;
        w.b = i / a.H; w.h[0] = w.h[1] = i % a.H; w.g = w.h[0] / a.G;
        w.qt[0] = w.qt[1] = t; w.n = 2;
        return w;
    }
    // two query tiles t, t-1 at a time: the pairs of heads at t, the last head's tiles t and t-1 where the heads are odd in
    // number, the pairs of heads at t-1
    const int groups = a.B * a.Hkv, hp = a.G / 2, odd = a.G & 1, per = groups * (2 * hp + odd);
    int t = a.nqt - 1 - 2 * (i / per);
    i %= per;
    w.n = 2;
    if (i >= groups * hp && i < groups * (hp + odd)) {
        i -= groups * hp;
        w.h[0] = w.h[1] = a.G - 1;
        w.qt[0] = t; w.qt[1] = t - 1;
        if (t == 0) w.n = 1;
    } else {
        if (i >= groups * hp) { i -= groups * (hp + odd); --t; }
        const int pair = i / groups;
        i %= groups;
        w.h[0] = 2 * pair; w.h[1] = w.h[0] + 1;
        w.qt[0] = w.qt[1] = t;
    }
    w.b = i / a.Hkv; w.g = i % a.Hkv;
    w.h[0] += w.g * a.G; w.h[1] += w.g * a.G;
    return w;
}

__global__ void __launch_bounds__(kAThreads, 1)
prefill_attn_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                    const __grid_constant__ CUtensorMap vmap, const AttnArgs a) {
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* base = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
    unsigned char* sQ = base;                                     // [2] tiles
    unsigned char* sK = base + 2 * kATile;                        // [kAStages] tiles
    unsigned char* sV = sK + kAStages * kATile;                   // [kAStages] tiles
    AttnSmem* sm = reinterpret_cast<AttnSmem*>(sV + kAStages * kATile);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const AttnTiles w = attn_tiles(a);
    int nk = 0, nk2[2];                                          // key tiles in all, and of either half of the CTA
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int key_end = a.causal ? min(a.N, (w.qt[u] + 1) * kAT) : a.N;
        nk2[u] = u < w.n ? (key_end + kAT - 1) / kAT : 0;
        nk = max(nk, nk2[u]);
    }
    // the i-th key tile of half u is i, or with the key tiles split 2 i + u
    const int split = a.split, nq = split ? 1 : w.n;
    if (split) { nk2[0] = (nk + 1) / 2; nk2[1] = nk / 2; }

    if (threadIdx.x == 0) {
        mbar_init(&sm->q_full, 1);
        for (int s = 0; s < kAStages; ++s) {
            mbar_init(&sm->k_full[s], 1); mbar_init(&sm->k_empty[s], 1);
            mbar_init(&sm->v_full[s], 1); mbar_init(&sm->v_empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&sm->s_full[s], 1); mbar_init(&sm->o_done[s], 1);
            mbar_init(&sm->p_ready[s][0], 4); mbar_init(&sm->p_ready[s][1], 4);
        }
        sm->abort = 0;
        fence_barrier_init();
        fence_proxy_async();
        prefetch_tmap(&qmap);
        prefetch_tmap(&kmap);
        prefetch_tmap(&vmap);
    }
    if (warp == 1) tmem_alloc(&sm->tmem_base, kATmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = sm->tmem_base;
    pdl_enter();

    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kARegsFew));
    if (warp == 0) {
        // ================= TMA producer =================
        if (lane == 0) {
            mbar_arrive_expect_tx(&sm->q_full, (uint32_t)(nq * kATile));
            for (int u = 0; u < nq; ++u) {
                tma_load_4d(sQ + u * kATile, &qmap, &sm->q_full, 0, w.h[u], w.qt[u] * kAT, w.b);
                tma_load_4d(sQ + u * kATile + kAHalf, &qmap, &sm->q_full, 64, w.h[u], w.qt[u] * kAT, w.b);
            }
            for (int j = 0; j < nk; ++j) {
                const int st = j % kAStages;
                if (j >= kAStages && !attn_wait(&sm->k_empty[st], ((j / kAStages) - 1) & 1, sm, a.dev_status)) break;
                mbar_arrive_expect_tx(&sm->k_full[st], kATile);
                tma_load_4d(sK + st * kATile, &kmap, &sm->k_full[st], 0, j * kAT, w.g, w.b);
                tma_load_4d(sK + st * kATile + kAHalf, &kmap, &sm->k_full[st], 64, j * kAT, w.g, w.b);
                if (j >= kAStages && !attn_wait(&sm->v_empty[st], ((j / kAStages) - 1) & 1, sm, a.dev_status)) break;
                mbar_arrive_expect_tx(&sm->v_full[st], kATile);
                tma_load_4d(sV + st * kATile, &vmap, &sm->v_full[st], 0, j * kAT, w.g, w.b);
                tma_load_4d(sV + st * kATile + kAHalf, &vmap, &sm->v_full[st], 64, j * kAT, w.g, w.b);
            }
        }
    } else if (warp == 1) {
        // ================= MMA issuer =================
        // The whole warp runs the loop (same values in every lane, so that they can live in uniform registers); one
        // elected lane issues the MMAs and the commits.
        constexpr uint32_t idesc_qk = idesc_bf16_f32(kAT, kAT);
        constexpr uint32_t idesc_pv = idesc_bf16_f32(kAT, kAT) | (1u << 16);     // B (the V tile) is MN-major
        const uint64_t qd0 = smem_desc_sw128(smem_u32(sQ)), kd0 = smem_desc_sw128(smem_u32(sK));
        const uint64_t vd0 = smem_desc_mn_sw128(smem_u32(sV), kAHalf);
        // S of half u for its i-th key tile, over the P of the one before
        auto issue_qk = [&](int u, int i) -> bool {
            const int j = split ? 2 * i + u : i, st = j % kAStages;
            if (!__all_sync(0xFFFFFFFFu, attn_wait(&sm->k_full[st], (j / kAStages) & 1, sm, a.dev_status))) return false;
            tc_fence_after();
            const uint64_t qd = qd0 + (uint32_t)((split ? 0 : u) * (kATile >> 4)), kd = kd0 + (uint32_t)(st * (kATile >> 4));
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {               // 16 channels are 32 bytes, 64 channels a half tile
                    const uint32_t off = ((k >> 2) * kAHalf + (k & 3) * 32) >> 4;
                    mma_bf16_ss(tmem_base + u * kAT, qd + off, kd + off, idesc_qk, k > 0 ? 1u : 0u);
                }
                mma_commit(&sm->s_full[u]);
                if (split || u == 1 || i >= nk2[1]) mma_commit(&sm->k_empty[st]);       // nobody needs the K tile any more
            }
            __syncwarp();
            return true;
        };
        bool ok = __all_sync(0xFFFFFFFFu, attn_wait(&sm->q_full, 0, sm, a.dev_status));
        for (int u = 0; u < 2; ++u)
            if (ok && nk2[u] > 0) ok = issue_qk(u, 0);
        for (int i = 0; ok && i < nk2[0]; ++i) {            // (half 0 has the longer run)
            for (int u = 0; ok && u < 2; ++u) {
                if (i >= nk2[u]) continue;
                const int j = split ? 2 * i + u : i, st = j % kAStages;
                const uint64_t vd = vd0 + (uint32_t)(st * (kATile >> 4));
                const uint32_t p_tmem = tmem_base + u * kAT, o_tmem = tmem_base + (2 + u) * kAT;
                ok = attn_wait(&sm->v_full[st], (j / kAStages) & 1, sm, a.dev_status);
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    ok = __all_sync(0xFFFFFFFFu, ok && attn_wait(&sm->p_ready[u][half], i & 1, sm, a.dev_status));
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
#pragma unroll
                        for (int k = half * 4; k < half * 4 + 4; ++k) {   // 16 keys: heads in 8 columns, remainders 16 columns on
                            const uint32_t pa = p_tmem + (k >> 1) * 32 + (k & 1) * 8;
                            mma_bf16_ts(o_tmem, pa, vd + (uint32_t)(k * (2048 >> 4)), idesc_pv, i > 0 || k > 0 ? 1u : 0u);
                            mma_bf16_ts(o_tmem, pa + 16, vd + (uint32_t)(k * (2048 >> 4)), idesc_pv, 1u);
                        }
                        if (half == 1) {
                            if (split || u == 1 || i >= nk2[1]) mma_commit(&sm->v_empty[st]);
                            if (i + 1 == nk2[u]) mma_commit(&sm->o_done[u]);
                        }
                    }
                    __syncwarp();
                }
                if (ok && i + 1 < nk2[u]) ok = issue_qk(u, i + 1);
            }
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kARegsMany));
        // ================= softmax: thread = query row of tile u =================
        const int u = (warp - 4) >> 2, quarter = warp & 3;   // (a warp reads the tensor-memory lanes 32 (warp % 4) .. + 31)
        const int row = quarter * 32 + lane;
        const int pos = w.qt[u] * kAT + row;                 // sequence position of my query
        const uint32_t s_addr = tmem_base + ((uint32_t)(quarter * 32) << 16) + u * kAT, o_addr = s_addr + 2 * kAT;
        const int n_mine = nk2[u], key_end = min(a.N, a.causal ? pos + 1 : a.N);
        const f32x2 sc = both(a.scale_log2);
        float m_used = -INFINITY;
        f32x2 l_run = both(0.f);
        bool ok = true;
        for (int j = 0; j < n_mine; ++j) {
            ok = __all_sync(0xFFFFFFFFu, attn_wait(&sm->s_full[u], j & 1, sm, a.dev_status));
            if (!ok) break;
            tc_fence_after();
            float v[4][32];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + c * 32, v[c]);
            tmem_ld_wait();
            const int lim = key_end - (split ? 2 * j + u : j) * kAT;      // my columns c < lim are visible
            // off the diagonal every lane of the warp sees all keys: no masks then
            if (!__all_sync(0xFFFFFFFFu, lim >= kAT)) {
#pragma unroll
                for (int c = 0; c < 4; ++c)
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[c][e] = c * 32 + e < lim ? v[c][e] : -INFINITY;
            }
            float t0 = v[0][0], t1 = v[1][0], t2 = v[2][0], t3 = v[3][0];
#pragma unroll
            for (int e = 1; e < 32; ++e) {
                t0 = fmaxf(t0, v[0][e]); t1 = fmaxf(t1, v[1][e]); t2 = fmaxf(t2, v[2][e]); t3 = fmaxf(t3, v[3][e]);
            }
            const float tmax = fmaxf(fmaxf(t0, t1), fmaxf(t2, t3)) * a.scale_log2;       // a positive scale keeps the order
            const bool grow = tmax > -INFINITY && (m_used == -INFINITY || tmax > m_used + kRescaleStep);
            // O is touched only when some row of the warp moves its reference
            if (__any_sync(0xFFFFFFFFu, grow)) {
                float corr = 1.f;
                if (grow) { corr = m_used == -INFINITY ? 0.f : ex2_fast(m_used - tmax); m_used = tmax; }
                if (j > 0) {
                    const f32x2 corr2 = both(corr);
                    l_run = mul2(l_run, corr2);
#pragma unroll 1
                    for (int c = 0; c < 4; ++c) {
                        float o[32];
                        tmem_ld32(o_addr + c * 32, o);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] *= corr;
                        tmem_st32(o_addr + c * 32, o);
                    }
                }
            }
            // probabilities relative to m_used, written over the logits they came from: 32 logits become 16 columns
            // of bf16 pairs (the bf16 rounding of every probability) and 16 columns of what the rounding left
            const f32x2 mneg = both(m_used == -INFINITY ? 0.f : -m_used);
            f32x2 ps0 = both(0.f), ps1 = both(0.f);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t pk[32];
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    float x0, x1;
                    unpack2(fma2(pack2(v[c][2 * e], v[c][2 * e + 1]), sc, mneg), x0, x1);
                    x0 = ex2_fast(x0); x1 = ex2_fast(x1);
                    const f32x2 p = pack2(x0, x1);
                    const uint32_t hi = pack_bf16(x0, x1);
                    float r0, r1;
                    unpack2(add2(p, pack2(-bf16_lo(hi), -bf16_hi(hi))), r0, r1);
                    pk[e] = hi;
                    pk[16 + e] = pack_bf16(r0, r1);
                    if (e & 1) ps1 = add2(ps1, p); else ps0 = add2(ps0, p);
                }
                tmem_st32(s_addr + c * 32, reinterpret_cast<const float*>(pk));
                if (c & 1) {                                 // half of the keys: the product may start on them
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm->p_ready[u][c >> 1]);
                }
            }
            l_run = add2(l_run, add2(ps0, ps1));
        }
        // ---- the output row --------------------------------------------------------------------------------
        float l0, l1;
        unpack2(l_run, l0, l1);
        float l_row = l0 + l1;
        // The rows of a warp go through shared memory (the Q tile is not needed any more): written row by row from the threads,
        // 32 rows side by side, every store instruction would touch 32 lines.  A row of 16-byte chunks, XOR-swizzled.
        unsigned char* stage = sQ + u * kATile + quarter * (kATile / 4);
        const int rowB = split ? 128 : 256, ch_mask = rowB / 16 - 1;
        auto stage32 = [&](int c, const float* o, float f) {         // 32 channels: chunks 4 c .. 4 c + 3 of my row
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4*>(stage + lane * rowB + (((4 * c + q) ^ (lane & ch_mask)) << 4)) =
                    make_uint4(pack_bf16(o[8 * q] * f, o[8 * q + 1] * f), pack_bf16(o[8 * q + 2] * f, o[8 * q + 3] * f),
                               pack_bf16(o[8 * q + 4] * f, o[8 * q + 5] * f), pack_bf16(o[8 * q + 6] * f, o[8 * q + 7] * f));
        };
        auto store_rows = [&](int c0) {                             // from channel c0 on
            __syncwarp();
            const int per = 512 / rowB, ch = lane & ch_mask;
            const int pos0 = w.qt[u] * kAT + quarter * 32;
            __nv_bfloat16* to = a.out + (int64_t)w.b * a.out_sb + (int64_t)w.h[u] * a.out_sh + c0 + ch * 8;
#pragma unroll 4
            for (int r = lane / (rowB / 16); r < 32; r += per) {
                const uint4 x = *reinterpret_cast<const uint4*>(stage + r * rowB + ((ch ^ (r & ch_mask)) << 4));
                if (pos0 + r < a.N) *reinterpret_cast<uint4*>(to + (int64_t)(pos0 + r) * a.out_sn) = x;
            }
        };
        if (!split) {
            if (n_mine > 0) {
                ok = __all_sync(0xFFFFFFFFu, ok && attn_wait(&sm->o_done[u], 0, sm, a.dev_status));
                tc_fence_after();
                const float inv = l_row > 0.f ? 1.0f / l_row : 0.f;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float o[32];
                    tmem_ld32(o_addr + c * 32, o);
                    tmem_ld_wait();
                    stage32(c, o, inv);
                }
                if (ok && !sm->abort) store_rows(0);
            }
        } else {
            // the two halves of the keys meet: a thread of half u finishes channels 64 u .. 64 u + 63 of its row
            sm->xm[u][row] = m_used;
            sm->xl[u][row] = l_row;
            asm volatile("bar.sync 1, %0;" ::"n"(2 * kAT) : "memory");
            const float m0 = sm->xm[0][row], m1 = sm->xm[1][row], ls0 = sm->xl[0][row], ls1 = sm->xl[1][row];
            m_used = fmaxf(m0, m1);
            const float f0 = m0 > -INFINITY ? exp2f(m0 - m_used) : 0.f, f1 = m1 > -INFINITY ? exp2f(m1 - m_used) : 0.f;
            l_row = ls0 * f0 + ls1 * f1;
            const float inv = l_row > 0.f ? 1.0f / l_row : 0.f;
            for (int x = 0; x < 2; ++x)
                ok = ok && (nk2[x] == 0 || attn_wait(&sm->o_done[x], 0, sm, a.dev_status));
            ok = __all_sync(0xFFFFFFFFu, ok);
            tc_fence_after();
            const uint32_t o0_addr = o_addr - u * kAT;
#pragma unroll 1
            for (int c = 2 * u; c < 2 * u + 2; ++c) {
                float o[32];
                tmem_ld32(o0_addr + c * 32, o);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 32; ++e) o[e] *= f0;
                if (nk2[1] > 0) {
                    float p[32];
                    tmem_ld32(o0_addr + kAT + c * 32, p);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; ++e) o[e] = f1 > 0.f ? fmaf(p[e], f1, o[e]) : o[e];
                }
                stage32(c - 2 * u, o, inv);
            }
            if (ok && !sm->abort) store_rows(64 * u);
        }
        if (n_mine > 0 && (!split || u == 0) && ok && pos < a.N && !sm->abort) {
            const float lse2 = m_used + log2f(l_row);        // log2 of the row's sum of 2^(scaled logits)
            a.lse[((int64_t)w.b * a.H + w.h[u]) * a.N + pos] = lse2 * kLn2A;
            if (a.lse_win && pos >= a.q_lo && pos < a.q_hi)
                a.lse_win[((int64_t)w.b * a.H + w.h[u]) * (a.q_hi - a.q_lo) + (pos - a.q_lo)] = lse2;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (sm->abort) {                              // let copies still in flight land before leaving
#pragma unroll 1
        for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, kATmemCols);
    }
}

// Two query tiles a CTA that take turns, or one whose key tiles are split between the two halves: as much work a CTA and
// key tile, but twice the CTAs, half as long.  The estimate of either, in units of a turn of both halves (4000 cycles):
// a CTA's turns and what its start and end take, shared out over the SMs, and a quarter of the longest CTA for the last
// wave.  us measured as pairs / split: 28 heads x 600 rows 22.7 / 16.6, 28 x 1000 28.9 / 24.8, 32 x 1500 39.1 / 43.5,
// 16 (no groups) x 5000 135 / 144, 28 x 3008 95 / 103.
static bool attn_split(int64_t tiles, int64_t pairs, double heads, int nqt, int causal) {
    const double turns = heads * (causal ? 0.5 * nqt * (nqt + 1.0) : (double)nqt * nqt) / 2;
    auto estimate = [&](double ctas, double longest, double each) {
        return ctas <= 148 ? longest + each : (turns + each * ctas) / 148 + 0.25 * (longest + each);
    };
    return estimate((double)tiles, 0.5 * nqt, 3.0) < estimate((double)pairs, nqt, 3.5);
}

#ifdef LVLM_TEST_HOOKS
static int g_attn_regs = 0;                  // the test build's idea of the registers a thread, 0 = the kernel's own
#endif

// The registers that the kernel is launched with cover the split of its warpgroups.
static lvlm_status attn_registers_fit() {
    cudaFuncAttributes f;
    LVLM_RETURN_IF_CUDA(cudaFuncGetAttributes(&f, prefill_attn_kernel));
    int regs = f.numRegs;
#ifdef LVLM_TEST_HOOKS
    if (g_attn_regs) regs = g_attn_regs;
#endif
    return 3 * regs >= kARegsFew + 2 * kARegsMany ? LVLM_OK : LVLM_ERR_CUDA;
}

size_t prefill_attn_workspace(const lvlm_dims* d) {
    ScoreLayout L;
    return score_layout(d, &L) ? L.total : 0;
}

}  // namespace lvlm

#ifdef LVLM_TEST_HOOKS
extern "C" void lvlm_debug_set_attn_regs(int n) { lvlm::g_attn_regs = n; }
#endif

extern "C" lvlm_status lvlm_prefill_attn(const void* Q, const void* K, const void* V, const lvlm_dims* d,
                                          float scale, void* out, float* lse, float* score, float* score_head,
                                          void* ws, size_t ws_bytes, int32_t* dev_status, void* stream_) {
    using namespace lvlm;
    cudaStream_t stream = (cudaStream_t)stream_;
    if (!Q || !K || !V || !out || !lse || !d || d->B <= 0 || d->H <= 0 || d->Hkv <= 0 || d->H % d->Hkv || d->N <= 0 ||
        d->cap < d->N || !(scale > 0.f))
        return LVLM_ERR_INVALID_ARG;
    if (score_head && !score) return LVLM_ERR_INVALID_ARG;
    if (d->D != kHeadDim) return LVLM_ERR_UNSUPPORTED;
    ScoreLayout L;
    if (score && !score_layout(d, &L)) return LVLM_ERR_INVALID_ARG;
    if (score && d->head_stride != 0 && d->head_stride < d->n) return LVLM_ERR_INVALID_ARG;
    ScoreStrides st;
    st.q_sh = d->q_stride_h ? d->q_stride_h : d->D;
    st.q_sn = d->q_stride_n ? d->q_stride_n : (int64_t)d->H * d->D;
    st.q_sb = d->q_stride_b ? d->q_stride_b : (int64_t)d->N * st.q_sn;
    st.kv_sh = d->kv_stride_h ? d->kv_stride_h : (int64_t)d->cap * d->D;
    st.kv_sb = d->kv_stride_b ? d->kv_stride_b : (int64_t)d->Hkv * st.kv_sh;
    if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(out) || st.q_sh % 8 || st.q_sn % 8 || st.q_sb % 8 ||
        st.kv_sh % 8 || st.kv_sb % 8)
        return LVLM_ERR_ALIGNMENT;
    char* wsb = static_cast<char*>(ws);
    if (score && (!ws || !aligned256(ws) || ws_bytes < L.total)) return LVLM_ERR_WORKSPACE;

    CUtensorMap qmap, kmap, vmap;
    {
        const uint64_t dims[4] = {(uint64_t)kHeadDim, (uint64_t)d->H, (uint64_t)d->N, (uint64_t)d->B};
        const uint64_t strides[3] = {(uint64_t)st.q_sh * 2, (uint64_t)st.q_sn * 2, (uint64_t)st.q_sb * 2};
        const uint32_t box[4] = {64, 1, (uint32_t)kAT, 1};
        if (!make_tmap_bf16(&qmap, Q, 4, dims, strides, box)) return LVLM_ERR_CUDA;
    }
    {
        const uint64_t dims[4] = {(uint64_t)kHeadDim, (uint64_t)d->N, (uint64_t)d->Hkv, (uint64_t)d->B};
        const uint64_t strides[3] = {(uint64_t)kHeadDim * 2, (uint64_t)st.kv_sh * 2, (uint64_t)st.kv_sb * 2};
        const uint32_t box[4] = {64, (uint32_t)kAT, 1, 1};
        if (!make_tmap_bf16(&kmap, K, 4, dims, strides, box) || !make_tmap_bf16(&vmap, V, 4, dims, strides, box))
            return LVLM_ERR_CUDA;
    }
    AttnArgs a;
    a.B = d->B; a.H = d->H; a.G = d->H / d->Hkv; a.Hkv = d->Hkv; a.N = d->N; a.causal = d->causal;
    a.q_lo = score ? d->q_lo : 0; a.q_hi = score ? d->q_hi : 0;
    a.scale_log2 = scale * kLog2eA;
    a.out = static_cast<__nv_bfloat16*>(out);
    a.out_sh = d->D; a.out_sn = (int64_t)d->H * d->D; a.out_sb = (int64_t)d->N * a.out_sn;
    a.lse = lse;
    a.lse_win = score ? reinterpret_cast<float*>(wsb + L.off_lse) : nullptr;
    a.dev_status = dev_status;
    const size_t smem = 1024 + (size_t)kATile * (2 + 2 * kAStages) + sizeof(AttnSmem);
    LVLM_RETURN_IF_CUDA(cudaFuncSetAttribute(prefill_attn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const lvlm_status fits = attn_registers_fit();
    if (fits != LVLM_OK) return fits;
    const int nqt = (d->N + kAT - 1) / kAT;
    const int64_t groups = (int64_t)d->B * d->Hkv, tiles = (int64_t)d->B * d->H * nqt;
    a.nqt = nqt;
    const int hp = a.G / 2, odd = a.G & 1;
    const int64_t pairs = groups * ((int64_t)(nqt / 2) * (2 * hp + odd) + (nqt % 2) * (hp + odd));
    a.split = attn_split(tiles, pairs, (double)d->B * d->H, nqt, d->causal) ? 1 : 0;
    const int64_t ctas = a.split ? tiles : pairs;
    if (ctas > 0x7FFFFFFFll) return LVLM_ERR_UNSUPPORTED;
    lvlm_status s0 = launch_kernel(prefill_attn_kernel, dim3((unsigned)ctas), dim3(kAThreads), smem, stream, 1, qmap, kmap, vmap, a);
    if (s0 != LVLM_OK || !score) return s0;
    // the column sums of the window: the second pass of lvlm_score_tokens, fed by the normalisers written above
    const __nv_bfloat16* Qwin = static_cast<const __nv_bfloat16*>(Q) + (int64_t)d->q_lo * st.q_sn;
    return launch_score_tc(Qwin, K, nullptr, d, st, scale, L, wsb, score, score_head, dev_status, stream,
                           /*normalisers_ready=*/true);
}
