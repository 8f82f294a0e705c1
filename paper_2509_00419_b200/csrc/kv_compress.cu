// lvlm_kv_compress: per (sequence, KV head) eviction of low-score cache entries
// (Section 3.2.2, paragraph 2: sort the scores in descending order, keep the entries whose
// accumulated score reaches the threshold beta, discard the other image entries; Appendix A.2:
// beta = 0.995).  A plan kernel finds the entry at which the threshold (and the budget) is met,
// builds the survivor map and compacts the small per-entry arrays; the shared in-place compaction kernel
// then moves the K and V rows.
#include "common.cuh"
#include "compact.cuh"

namespace lvlm {

struct KvLayout { size_t off_src, off_meta, off_nout, off_acc, off_pos, total; };

static bool kv_layout(const lvlm_dims* d, KvLayout* L) {
    if (!d || d->B <= 0 || d->Hkv <= 0 || d->cap <= 0 || d->recent < 0) return false;
    size_t off = 0;
    const size_t heads = (size_t)d->B * d->Hkv;
    L->off_src = off;  off = align_up(off + heads * d->cap * 4, 256);
    L->off_meta = off; off = align_up(off + heads * 4, 256);
    L->off_nout = off; off = align_up(off + heads * 4, 256);
    L->off_acc = off;  off = align_up(off + heads * d->cap * 4, 256);     // compacted acc_score and pos, copied back
    L->off_pos = off;  off = align_up(off + heads * d->cap * 4, 256);     // by the kernel that moves the rows
    L->total = off;
    return true;
}

size_t kv_compress_workspace(const lvlm_dims* d) {
    KvLayout L;
    return kv_layout(d, &L) ? L.total : 0;
}

// Score in integer units of 1 / per_unit, a power of two (negative and non-finite scores count as zero).
constexpr float kScoreUnits = 16777216.0f;               // units of 2^-24
__device__ __forceinline__ long long score_units(float s, float per_unit) {
    if (!(s > 0.f) || (__float_as_uint(s) & 0x7F800000u) == 0x7F800000u) return 0;
    return __float2ll_rn(s * per_unit);                  // (saturates at 2^63 - 1)
}

// ceil(beta_ppm * total / 10^6) for beta_ppm < 10^6, total < 2^63: with total = 10^6 q + r it is beta_ppm q + ceil(beta_ppm r / 10^6).
// (Divisions by a constant; a 128-bit long division took 7 us.)
__device__ __forceinline__ unsigned long long beta_of_total(unsigned long long beta_ppm, unsigned long long total) {
    const unsigned long long q = total / 1000000ull, r = total - q * 1000000ull;
    return beta_ppm * q + (beta_ppm * r + 999999ull) / 1000000ull;
}

__device__ __forceinline__ unsigned long long redux_add_u64(unsigned long long v) {
    // three limbs of 22 bits: 32 of them still fit a word (v < 2^63)
    const uint32_t l0 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)v & 0x3FFFFFu);
    const uint32_t l1 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> 22) & 0x3FFFFFu);
    const uint32_t l2 = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> 44));
    return (unsigned long long)l0 + ((unsigned long long)l1 << 22) + ((unsigned long long)l2 << 44);
}

// The score behind a key, and its units.
__device__ __forceinline__ float score_of_key(uint32_t dk) {
    const uint32_t asc = ~dk;
    return __uint_as_float((asc & 0x80000000u) ? (asc & 0x7FFFFFFFu) : ~asc);
}
__device__ __forceinline__ unsigned long long units_of_key(uint32_t dk, float per_unit) {
    return dk == 0xFFFFFFFFu ? 0ull : (unsigned long long)score_units(score_of_key(dk), per_unit);
}

// Scores so large that their sum may not fit 63 bits in units of 2^-24 (an entry of 2^49 units or more: 16384 smaller ones
// always fit).  A sum that wraps around would name a threshold that the entries do not reach, and survivors that
// are not there.  lo, hi: the sums of the low and of the high words of the units; if the whole sum does not fit, the unit
// is taken coarser, so that an entry has at most 2^48 of them.  best: the key of the largest finite score.
constexpr int kBigUnits = 49;
constexpr uint32_t kKeyOfInfinity = 0x007FFFFFu;         // the smallest key
__device__ __forceinline__ float units_that_fit(unsigned long long lo, unsigned long long hi, uint32_t best) {
    if (hi + (lo >> 32) < (1ull << 31)) return kScoreUnits;
    const uint32_t e = __float_as_uint(score_of_key(best)) >> 23;            // 127 + exponent, at least 25
    return __uint_as_float((127u + 47u - (e - 127u)) << 23);
}

// One CTA per (sequence, KV head).  A warp has 32 * KPT consecutive evictable entries, lane l of it l, l + 32, ..., as 32-bit
// keys (order-preserving image of the score: ascending key = descending score; among equal scores the lower index comes
// first).  Nothing is sorted: the score at which the accumulated score reaches the threshold, and the one that closes
// the budget, are found from the top, 11 bits a pass, at most three passes: a histogram in shared memory (of the count, or
// of the score in limbs of 18 bits, so that 16384 of them fit a word), a scan, and only the entries of the bucket that
// crosses the target go on.  88 heads of 3008 rows: 42 us a bit a time over 64-bit keys (a block-wide sum and a barrier
// each), 22 with two bits a time, now 16.  All sums are integers, so the result does not depend on the order of summation.
constexpr int kPlanDigit = 11, kPlanBuckets = 1 << kPlanDigit, kPlanLimb = 18, kPlanLimbs = 4;
constexpr int kPlanHist = kPlanBuckets + kPlanBuckets / 8;         // a word of padding every 8: a thread scans 8 buckets (or 2)
__device__ __forceinline__ uint32_t plan_bucket(uint32_t i) { return i + (i >> 3); }

template <int KPT, int MAXT>
__global__ void __launch_bounds__(MAXT)
kv_plan_kernel(float* acc_score, int32_t* pos, int32_t* len, const int32_t* __restrict__ e_lo,
               const int32_t* __restrict__ e_hi, int Hkv, int cap, int recent, int min_m,
               unsigned long long beta_ppm, int budget, int32_t* __restrict__ src_map,
               int32_t* __restrict__ meta, int32_t* __restrict__ nout, float* __restrict__ acc_new,
               int32_t* __restrict__ pos_new, int32_t* dev_status) {
    __shared__ __align__(16) uint32_t s_hist[kPlanLimbs][kPlanHist];
    __shared__ unsigned long long s_sum[32], s_before;
    __shared__ uint32_t s_and[32], s_or[32], s_big[32], s_digit;
    __shared__ int s_first_drop;

    pdl_enter();
    const int g = blockIdx.x, b = blockIdx.y;
    const int m_idx = b * Hkv + g;
    const int ln = len[m_idx];
    int32_t* src = src_map + (int64_t)m_idx * cap;
    float* acc = acc_score + (int64_t)m_idx * cap;
    if (ln < 0 || ln > cap) {
        if (threadIdx.x == 0) {
            if (dev_status) atomicOr(dev_status, LVLM_DEV_BOUNDS);
            meta[m_idx] = 0; nout[m_idx] = 0;           // nothing moves, length left as it is
        }
        return;
    }
    int lo = e_lo ? e_lo[b] : 0;
    int hi = e_hi ? e_hi[b] : ln;
    hi = min(hi, ln - recent);
    lo = min(max(lo, 0), ln);
    hi = max(hi, lo);
    const int m = hi - lo;
    if (m < min_m) return;                               // a head this small was planned by the warp kernel
    // only the warps that hold entries stay: every barrier below counts them alone
    const int nwarp = max(1, (m + 32 * KPT - 1) / (32 * KPT)), nthr = nwarp * 32;
    if ((int)threadIdx.x >= nthr) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto sync_active = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory"); };
    if (threadIdx.x == 0) s_first_drop = m;
    // compacted acc_score and pos go beside the map; the kernel that moves the K and V rows copies them back
    float* an = acc_new + (int64_t)m_idx * cap;
    const int32_t* ps = pos ? pos + (int64_t)m_idx * cap : nullptr;
    int32_t* pn = pos_new + (int64_t)m_idx * cap;

    // ---- my keys -------------------------------------------------------------------------------------
    const int j0 = warp * (32 * KPT) + lane;             // my entries: j0, j0 + 32, ...
    float sv[KPT];
    uint32_t key[KPT];
    unsigned long long un[KPT];                          // the scores in integer units
    bool nonfinite = false;
    uint32_t k_and = ~0u, k_or = 0u, big = 0u;
#pragma unroll
    for (int u = 0; u < KPT; ++u) sv[u] = j0 + 32 * u < m ? acc[lo + j0 + 32 * u] : 0.f;
#pragma unroll
    for (int u = 0; u < KPT; ++u) {
        key[u] = ~0u;                                    // past the end: the top value, no score
        un[u] = 0ull;
        if (j0 + 32 * u < m) {
            key[u] = desc_key(sv[u], &nonfinite);
            k_and &= key[u]; k_or |= key[u];
            un[u] = (unsigned long long)score_units(sv[u], kScoreUnits);
            big |= (uint32_t)(un[u] >> kBigUnits);
        }
    }
    if (nonfinite && dev_status) atomicOr(dev_status, LVLM_DEV_NONFINITE);
    k_and = __reduce_and_sync(0xFFFFFFFFu, k_and);       // bits in which the keys differ
    k_or = __reduce_or_sync(0xFFFFFFFFu, k_or);
    big = __reduce_or_sync(0xFFFFFFFFu, big);
    if (lane == 0) { s_and[warp] = k_and; s_or[warp] = k_or; s_big[warp] = big; }
    sync_active();
    k_and = __reduce_and_sync(0xFFFFFFFFu, lane < nwarp ? s_and[lane] : ~0u);
    k_or = __reduce_or_sync(0xFFFFFFFFu, lane < nwarp ? s_or[lane] : 0u);
    big = __reduce_or_sync(0xFFFFFFFFu, lane < nwarp ? s_big[lane] : 0u);
    const uint32_t diff = m > 0 ? (k_and ^ k_or) : 0u;

    // Exclusive prefix sum over the block's threads, in thread order, and the total.
    auto block_scan = [&](unsigned long long x, unsigned long long* total) -> unsigned long long {
        unsigned long long incl = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        sync_active();                                   // s_sum may still be read from a call before
        if (lane == 31) s_sum[warp] = incl;
        sync_active();
        const unsigned long long w = lane < nwarp ? s_sum[lane] : 0ull;
        *total = redux_add_u64(w);
        return redux_add_u64(lane < warp ? w : 0ull) + incl - x;
    };
    // Smallest score key T such that the entries with key <= T hold at least `target` (their count, or their score when
    // by_mass, in `limbs` limbs); *before: what the entries with a strictly better score hold.  The caller guarantees
    // that all entries together reach the target.
    auto search = [&](unsigned long long target, bool by_mass, int limbs, unsigned long long* before) -> uint32_t {
        unsigned long long below = 0ull;
        uint32_t prefix = k_and;                         // T, as far as it is known: the bits from `shift` up
        int shift = 32 - __clz((int)diff);               // (the bits from here up do not differ)
        const int per = (kPlanBuckets + nthr - 1) / nthr, b0 = min(kPlanBuckets, (int)threadIdx.x * per), b1 = min(kPlanBuckets, b0 + per);
        while (shift > 0) {
            const int hi_shift = shift;
            shift = max(0, shift - kPlanDigit);
            for (int i = threadIdx.x; i < limbs * (kPlanHist / 4); i += nthr)
                reinterpret_cast<uint4*>(s_hist)[i] = make_uint4(0u, 0u, 0u, 0u);
            sync_active();
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                // (shifts of 32 are not defined: two steps)
                if (j0 + 32 * u >= m || ((key[u] ^ prefix) >> (hi_shift - 1)) >> 1) continue;
                const uint32_t d = plan_bucket((key[u] >> shift) & (kPlanBuckets - 1));
                if (!by_mass) { atomicAdd(&s_hist[0][d], 1u); continue; }
#pragma unroll
                for (int l = 0; l < kPlanLimbs; ++l) {
                    const uint32_t x = (uint32_t)(un[u] >> (l * kPlanLimb)) & ((1u << kPlanLimb) - 1u);
                    if (x) atomicAdd(&s_hist[l][d], x);
                }
            }
            sync_active();
            unsigned long long mine = 0ull, total;
#pragma unroll
            for (int l = 0; l < kPlanLimbs; ++l) {       // (a limb summed over all entries fits a word)
                uint32_t x = 0u;
                if (l < limbs) {
#pragma unroll 8
                    for (int i = b0; i < b1; ++i) x += s_hist[l][plan_bucket(i)];
                }
                mine += (unsigned long long)x << (l * kPlanLimb);
            }
            unsigned long long run = below + block_scan(mine, &total);
            if (run < target && run + mine >= target) {  // the bucket that crosses the target is one of mine
                unsigned long long b = run;
                int d = b0;
#pragma unroll 4
                for (int i = b0; i < b1; ++i) {          // (no early exit: the loads overlap)
                    unsigned long long x = 0ull;
#pragma unroll
                    for (int l = 0; l < kPlanLimbs; ++l)
                        if (l < limbs) x += (unsigned long long)s_hist[l][plan_bucket(i)] << (l * kPlanLimb);
                    run += x;
                    if (run < target) { b = run; d = i + 1; }
                }
                s_digit = (uint32_t)d;
                s_before = b;
            }
            sync_active();
            below = s_before;
            // (the digit may reach above the bits that differ: those bits are the same in every key)
            prefix = (prefix & ~((kPlanBuckets - 1u) << shift)) | (s_digit << shift);
        }
        *before = below;
        return prefix;
    };

    // ---- how many entries of E reach the threshold, how many the budget allows ---------------------------
    int k_beta = m, need = 0;
    uint32_t T = ~0u;                                    // survivors: score key < T, and the first `need` entries of key T
    bool have_T = false;
    unsigned long long before = 0ull;
    if (beta_ppm < 1000000ull && m > 0) {
        unsigned long long mine = 0ull, total;
        float per_unit = kScoreUnits;
        if (big) {
            unsigned long long lo_w = 0ull, hi_w = 0ull;
            uint32_t best = ~0u;
#pragma unroll
            for (int u = 0; u < KPT; ++u) {
                lo_w += un[u] & 0xFFFFFFFFull;
                hi_w += un[u] >> 32;
                if (un[u]) best = min(best, key[u]);
            }
            block_scan(lo_w, &lo_w);
            block_scan(hi_w, &hi_w);
            best = __reduce_min_sync(0xFFFFFFFFu, best);
            if (lane == 0) s_big[warp] = best;           // (the flags were read before the scans)
            sync_active();
            per_unit = units_that_fit(lo_w, hi_w, __reduce_min_sync(0xFFFFFFFFu, lane < nwarp ? s_big[lane] : ~0u));
#pragma unroll
            for (int u = 0; u < KPT; ++u) un[u] = un[u] ? units_of_key(key[u], per_unit) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < KPT; ++u) mine += un[u];
        block_scan(mine, &total);
        const unsigned long long thr = beta_of_total(beta_ppm, total);
        if (thr == 0) k_beta = 1;
        else {
            const int limbs = min(kPlanLimbs, (63 - __clzll((long long)total)) / kPlanLimb + 1);     // (no entry holds more than all)
            T = search(thr, true, limbs, &before);
            const unsigned long long each = units_of_key(T, per_unit);   // > 0: the entries of key T are needed
            need = (int)((thr - before + each - 1ull) / each);
            have_T = true;
        }
    }
    // Entries better than T and of score T, in the warps before mine (16 bits each), and of all warps.
    auto count_T = [&](int* all) -> int {
        int better = 0, equal = 0;
#pragma unroll
        for (int u = 0; u < KPT; ++u) {
            better += __popc(__ballot_sync(0xFFFFFFFFu, j0 + 32 * u < m && key[u] < T));
            equal += __popc(__ballot_sync(0xFFFFFFFFu, j0 + 32 * u < m && key[u] == T));
        }
        sync_active();
        if (lane == 0) s_sum[warp] = (unsigned long long)(uint32_t)(better | (equal << 16));
        sync_active();
        const uint32_t w = lane < nwarp ? (uint32_t)s_sum[lane] : 0u;
        *all = (int)__reduce_add_sync(0xFFFFFFFFu, w);
        return (int)__reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u);
    };
    int all = 0, before_me = 0;
    if (have_T) { before_me = count_T(&all); k_beta = (all & 0xFFFF) + need; }
    int kc = k_beta;
    if (budget > 0) kc = min(kc, budget - (ln - m));
    kc = min(max(kc, 0), m);
    if (kc < m && kc > 0 && !(have_T && kc == k_beta)) {
        T = search((unsigned long long)kc, false, 1, &before);
        need = kc - (int)before;
        before_me = count_T(&all);
    }

    // ---- survivor map, in index order: a warp's entries 32 at a time, places by ballot --------------------------
    {
        int eq = before_me >> 16;                        // entries of score T in the warps before mine
        int off = kc >= m ? warp * (32 * KPT) : kc == 0 ? 0 : (before_me & 0xFFFF) + min(eq, need);
        const uint32_t lt = (1u << lane) - 1u;
        int first_drop = m;
#pragma unroll
        for (int u = 0; u < KPT; ++u) {
            const int j = j0 + 32 * u;
            const bool valid = j < m, is_eq = valid && key[u] == T;
            const uint32_t beq = __ballot_sync(0xFFFFFFFFu, is_eq);
            const bool kept = valid && (kc >= m || (kc > 0 && (key[u] < T || (is_eq && eq + __popc(beq & lt) < need))));
            const uint32_t bk = __ballot_sync(0xFFFFFFFFu, kept), bd = __ballot_sync(0xFFFFFFFFu, valid && !kept);
            if (kept) {
                const int o = lo + off + __popc(bk & lt);
                src[o] = lo + j;
                an[o] = KPT > 4 && MAXT > 256 ? acc[lo + j] : sv[u];     // (1024 threads: 8 or 16 scores more do not fit the registers)
                if (ps) pn[o] = ps[lo + j];
            }
            if (first_drop == m && bd) first_drop = j - lane + __ffs((int)bd) - 1;
            off += __popc(bk);
            eq += __popc(beq);
        }
        if (lane == 0 && first_drop < m) atomicMin(&s_first_drop, first_drop);
    }
    const int new_len = lo + kc + (ln - hi);
    for (int o = threadIdx.x; o < new_len; o += nthr) {
        if (o < lo) src[o] = o;
        else if (o >= lo + kc) {
            const int sidx = hi + (o - lo - kc);
            src[o] = sidx;
            an[o] = acc[sidx];
            if (ps) pn[o] = ps[sidx];
        }
    }
    sync_active();
    if (threadIdx.x == 0) {
        meta[m_idx] = kc < m ? lo + s_first_drop : new_len;
        nout[m_idx] = new_len;
        len[m_idx] = new_len;
    }
}

// The same for caches of up to 2048 rows: one WARP per (sequence, KV head); lane l holds entries l, l + 32, ...
// (coalesced), every sum is a handful of shuffles and no barrier is needed, so an SM works on dozens of heads at
// once.  Only the 32-bit image of the score is searched: among entries of equal score the lower index comes first,
// so once the threshold score T is known, "the first `need` entries of score T" is a running count in index order
// and the index never has to enter the key.  The searches are loops over registers; the pass that writes the map
// is a loop over the entries that reads the scores again (they are in L1), which keeps the kernel's code short:
// a warp runs through it once, and straight-line code is fetched slower than it executes.
// MASS: the threshold beta is in use (without it only the budget's count search is compiled in).
__device__ __forceinline__ void plan_cp_async4(void* smem, const void* gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem) : "memory");
}

template <int KPL, bool MASS>
__global__ void __launch_bounds__(128)
kv_plan_warp_kernel(float* acc_score, int32_t* pos, int32_t* len, const int32_t* __restrict__ e_lo,
                    const int32_t* __restrict__ e_hi, int heads, int Hkv, int cap, int recent, int only_small,
                    unsigned long long beta_ppm, int budget, int32_t* __restrict__ src_map,
                    int32_t* __restrict__ meta, int32_t* __restrict__ nout, float* __restrict__ acc_new,
                    int32_t* __restrict__ pos_new, int32_t* dev_status) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int m_idx = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (m_idx >= heads) return;
    const int b = m_idx / Hkv;
    const int ln = len[m_idx];
    int32_t* src = src_map + (int64_t)m_idx * cap;
    float* acc = acc_score + (int64_t)m_idx * cap;
    if (ln < 0 || ln > cap) {
        if (lane == 0) {
            if (dev_status) atomicOr(dev_status, LVLM_DEV_BOUNDS);
            meta[m_idx] = 0; nout[m_idx] = 0;           // nothing moves, length left as it is
        }
        return;
    }
    int lo = e_lo ? e_lo[b] : 0;
    int hi = e_hi ? e_hi[b] : ln;
    hi = min(hi, ln - recent);
    lo = min(max(lo, 0), ln);
    hi = max(hi, lo);
    const int m = hi - lo;
    if (only_small && m > 32 * KPL) return;              // too many entries for the registers: the CTA kernel plans it

    // The scores and the position ids of the evictable entries come to shared memory by asynchronous copies
    // (all of them in flight at once); the scores are turned into keys there, by a loop over the entries, and
    // then taken into registers.
    extern __shared__ __align__(16) uint32_t s_plan[];   // per warp: [KPL * 32] keys, [KPL * 32] position ids
    uint32_t* my_hk = s_plan + (threadIdx.x >> 5) * (2 * KPL * 32);
    uint32_t* my_pos = my_hk + KPL * 32;
    const int32_t* ps = pos ? pos + (int64_t)m_idx * cap : nullptr;
#pragma unroll 4
    for (int j = lane; j < m; j += 32) {
        plan_cp_async4(&my_hk[j], acc + lo + j);
        if (ps) plan_cp_async4(&my_pos[j], ps + lo + j);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncwarp();
    uint32_t k_and = ~0u, k_or = 0u;
    bool nonfinite = false;
#pragma unroll 4
    for (int j = lane; j < KPL * 32; j += 32) {
        uint32_t h = ~0u;                                // past the end: the top value
        if (j < m) { h = desc_key(__uint_as_float(my_hk[j]), &nonfinite); k_and &= h; k_or |= h; }
        my_hk[j] = h;
    }
    if (nonfinite && dev_status) atomicOr(dev_status, LVLM_DEV_NONFINITE);
    uint32_t hk[KPL];                                    // ascending = descending score
#pragma unroll
    for (int u = 0; u < KPL; ++u) hk[u] = my_hk[u * 32 + lane];       // (written by this very lane)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        k_and &= __shfl_xor_sync(0xFFFFFFFFu, k_and, o);
        k_or |= __shfl_xor_sync(0xFFFFFFFFu, k_or, o);
    }
    const uint32_t diff = m > 0 ? (k_and ^ k_or) : 0u;
    float per_unit = kScoreUnits;
    // Score units of the entries with key <= cand (or < cand), summed over the warp.
    auto mass_upto = [&](uint32_t cand, bool strict) -> unsigned long long {
        unsigned long long ms = 0;
#pragma unroll
        for (int u = 0; u < KPL; ++u) {
            uint32_t h = hk[u];
            if (KPL > 32) asm volatile("" : "+r"(h));    // worked out again at every use: 64 more registers would not fit
            if (strict ? h < cand : h <= cand) ms += units_of_key(h, per_unit);
        }
        return redux_add_u64(ms);
    };
    // Smallest score key T such that the entries with key <= T are at least `target` many (by_count) or hold at
    // least `target` units of score: built bit by bit from the top, over the bits in which the keys differ.
    // Entries past the end carry the top key and no score: they are counted only where every real entry is.
    auto search = [&](unsigned long long target, bool by_count) -> uint32_t {
        uint32_t ans = k_and, todo = diff;
#pragma unroll 1
        while (todo) {
            const int bit = 31 - __clz((int)todo);
            todo &= ~(1u << bit);
            const uint32_t cand = (ans & ~(1u << bit)) | ((1u << bit) - 1u);
            unsigned long long have;
            if (!MASS || by_count) {
                int cnt = 0;
#pragma unroll
                for (int u = 0; u < KPL; ++u) cnt += hk[u] <= cand;
                have = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)cnt);
            } else {
                have = mass_upto(cand, false);
            }
            if (have >= target) ans &= ~(1u << bit); else ans |= 1u << bit;
        }
        return ans;
    };
    auto count_below = [&](uint32_t T) -> int {          // entries with a strictly better score than T
        int c = 0;
#pragma unroll
        for (int u = 0; u < KPL; ++u) c += hk[u] < T;
        return (int)__reduce_add_sync(0xFFFFFFFFu, (uint32_t)c);
    };

    // ---- how many entries reach the threshold, how many the budget allows --------------------------------------
    int k_beta = m;
    uint32_t T = ~0u;                                    // survivors: score key < T, and the first `need` entries of key T
    int need = 0;
    bool have_T = false;
    if (MASS && m > 0) {
        uint32_t best = ~0u;                             // the largest finite score
#pragma unroll
        for (int u = 0; u < KPL; ++u) if (hk[u] > kKeyOfInfinity) best = min(best, hk[u]);
        best = __reduce_min_sync(0xFFFFFFFFu, best);
        if (units_of_key(best, kScoreUnits) >> kBigUnits) {
            unsigned long long lo_w = 0ull, hi_w = 0ull;
#pragma unroll 1
            for (int j = lane; j < KPL * 32; j += 32) {                      // (the keys are in shared memory still)
                const unsigned long long x = units_of_key(my_hk[j], kScoreUnits);
                lo_w += x & 0xFFFFFFFFull;
                hi_w += x >> 32;
            }
            per_unit = units_that_fit(redux_add_u64(lo_w), redux_add_u64(hi_w), best);
        }
        const unsigned long long total = mass_upto(~0u, false);
        const unsigned long long thr = beta_of_total(beta_ppm, total);
        if (thr == 0) k_beta = 1;
        else {
            T = search(thr, false);
            const int c = count_below(T);
            const unsigned long long below = mass_upto(T, true);
            const unsigned long long each = units_of_key(T, per_unit);       // > 0: the entries of key T are needed
            need = (int)((thr - below + each - 1ull) / each);
            k_beta = c + need;
            have_T = true;
        }
    }
    int kc = k_beta;
    if (budget > 0) kc = min(kc, budget - (ln - m));
    kc = min(max(kc, 0), m);
    if (kc < m && kc > 0 && !(have_T && kc == k_beta)) {
        T = search((unsigned long long)kc, true);
        need = kc - count_below(T);
    }

    // ---- the survivor map, in index order: 32 entries a round, places by ballot ---------------------------------
    float* an = acc_new + (int64_t)m_idx * cap;
    int32_t* pn = pos_new + (int64_t)m_idx * cap;
    const uint32_t lt_mask = (1u << lane) - 1u;
    int first_drop = m;
    if (kc < m) {
        int base = 0, eq_base = 0;
#pragma unroll 2
        for (int j0 = 0; j0 < m; j0 += 32) {
            const int j = j0 + lane;
            const bool valid = j < m;
            const float sv = valid ? acc[lo + j] : 0.f;
            bool nf = false;
            const uint32_t h = valid ? desc_key(sv, &nf) : ~0u;
            const bool is_eq = valid && h == T;
            const uint32_t beq = __ballot_sync(0xFFFFFFFFu, is_eq);
            const bool kept = valid && kc > 0 && (h < T || (is_eq && eq_base + __popc(beq & lt_mask) < need));
            const uint32_t bk = __ballot_sync(0xFFFFFFFFu, kept);
            if (kept) {
                const int o = lo + base + __popc(bk & lt_mask);
                src[o] = lo + j;
                an[o] = sv;
                if (ps) pn[o] = (int32_t)my_pos[j];
            }
            const uint32_t bd = __ballot_sync(0xFFFFFFFFu, valid && !kept);
            if (first_drop == m && bd) first_drop = j0 + __ffs((int)bd) - 1;
            base += __popc(bk);
            eq_base += __popc(beq);
        }
    }
    const int new_len = lo + kc + (ln - hi);
    // rows that do not move (everything when nothing is evicted) and the rows behind the evictable range
    for (int o = lane; o < new_len; o += 32) {
        if (o < lo || kc >= m) {
            src[o] = o;
            if (o >= lo) { an[o] = acc[o]; if (ps) pn[o] = ps[o]; }
        } else if (o >= lo + kc) {
            const int sidx = hi + (o - lo - kc);
            src[o] = sidx;
            an[o] = acc[sidx];
            if (ps) pn[o] = ps[sidx];
        }
    }
    if (lane == 0) {
        meta[m_idx] = kc < m ? lo + first_drop : new_len;
        nout[m_idx] = new_len;
        len[m_idx] = new_len;
    }
}

}  // namespace lvlm

extern "C" lvlm_status lvlm_kv_compress(void* Kc, void* Vc, float* acc_score, int32_t* pos,
                                         int32_t* len, const int32_t* e_lo, const int32_t* e_hi,
                                         const lvlm_dims* d, float beta, int budget, void* ws,
                                         size_t ws_bytes, int32_t* dev_status, void* stream_) {
    using namespace lvlm;
    cudaStream_t stream = (cudaStream_t)stream_;
    KvLayout L;
    if (!Kc || !Vc || !acc_score || !len || !kv_layout(d, &L)) return LVLM_ERR_INVALID_ARG;
    if ((e_lo == nullptr) != (e_hi == nullptr)) return LVLM_ERR_INVALID_ARG;
    if (!(beta > 0.f) || beta > 1.f) return LVLM_ERR_INVALID_ARG;
    if (d->D != kHeadDim || d->cap > kMaxSortN) return LVLM_ERR_UNSUPPORTED;
    const int64_t kv_sh = d->kv_stride_h ? d->kv_stride_h : (int64_t)d->cap * d->D;
    const int64_t kv_sb = d->kv_stride_b ? d->kv_stride_b : (int64_t)d->Hkv * kv_sh;
    if (!aligned16(Kc) || !aligned16(Vc) || kv_sh % 8 || kv_sb % 8) return LVLM_ERR_ALIGNMENT;
    if (!ws || !aligned256(ws) || ws_bytes < L.total) return LVLM_ERR_WORKSPACE;
    char* wsb = static_cast<char*>(ws);
    int32_t* src_map = reinterpret_cast<int32_t*>(wsb + L.off_src);
    int32_t* meta = reinterpret_cast<int32_t*>(wsb + L.off_meta);
    int32_t* nout = reinterpret_cast<int32_t*>(wsb + L.off_nout);
    float* acc_new = reinterpret_cast<float*>(wsb + L.off_acc);
    int32_t* pos_new = reinterpret_cast<int32_t*>(wsb + L.off_pos);

    const unsigned long long beta_ppm = (unsigned long long)llrint((double)beta * 1.0e6);
    const int heads = d->B * d->Hkv;
    lvlm_status st;
#define LVLM_PLAN_WARP_(KPL_, SMALL_, MASS_)                                                                     \
    (cudaFuncSetAttribute(kv_plan_warp_kernel<KPL_, MASS_>, cudaFuncAttributeMaxDynamicSharedMemorySize,              \
                          4 * 2 * KPL_ * 32 * 4) != cudaSuccess                                                       \
         ? LVLM_ERR_CUDA                                                                                             \
         : launch_kernel(kv_plan_warp_kernel<KPL_, MASS_>, dim3((heads + 3) / 4), dim3(128), 4 * 2 * KPL_ * 32 * 4,   \
                         stream, 1, acc_score, pos, len, e_lo, e_hi, heads, d->Hkv, d->cap, d->recent, SMALL_,        \
                         beta_ppm, budget, src_map, meta, nout, acc_new, pos_new, dev_status))
#define LVLM_PLAN_WARP(KPL_, SMALL_) \
    st = beta_ppm < 1000000ull ? LVLM_PLAN_WARP_(KPL_, SMALL_, true) : LVLM_PLAN_WARP_(KPL_, SMALL_, false)
    // With enough heads to fill the GPU with one warp each, a warp per head (no barrier in the searches); a CTA per
    // head otherwise, and for the heads whose entries do not fit a warp's registers.
    const bool many = heads >= 4 * 148;
    // Entries a thread: the plan is a chain of passes over them, so few while the heads leave SMs idle; with more heads than SMs warps
    // wait for one another anyhow, and long caches are better off with fewer of them.  us of a compression (beta 0.99) with 16 / 8 / 4
    // entries, heads x rows: 40 x 3000 31.2 / - / 27.8, 148 x 4096 56.1 / - / 54.0, 100 x 6000 67.2 / 61.2, 148 x 8000 90.9 / 88.0; 149 x 1100
    // 36.4 / 32.8 / 30.2, 320 x 1100 48.1 / 46.9 / 43.4, 200 x 2048 48.2 / 46.0 / 45.7, 320 x 2048 64.4 / 63.2 / 68.1, 448 x 3000 114.7 / 112.3 / 125.4,
    // 400 x 3500 116.3 / 114.7 / 122.8, 700 x 3000 172.5 / 162.3 / 175.8; 256 x 4096 78.0 / 79.4, 512 x 4096 145.0 / 146.9, 256 x 5000
    // 96.3 / 100.3, 560 x 5000 190.8 / 201.2, 300 x 6000 149.8 / 151.5.
    const int kpt = d->cap <= (heads <= 148 ? 4096 : 1024) ? 4 : d->cap <= (heads <= 148 ? 8192 : 3584) ? 8 : 16;
    int threads = ((d->cap + kpt - 1) / kpt + 31) / 32 * 32;
    int min_m = 0;                                       // heads the CTA kernel leaves to the warp kernel
    bool cta_kernel = true;
    if (many) {
        if (d->cap <= 512) LVLM_PLAN_WARP(16, 0);
        else if (d->cap <= 1024) LVLM_PLAN_WARP(32, 0);
        else if (d->cap <= 1536) LVLM_PLAN_WARP(48, 0);
        else if (d->cap <= 2048) LVLM_PLAN_WARP(64, 0);
        else LVLM_PLAN_WARP(32, 1);                      // long caches: the heads with up to 1024 evictable entries
        if (st != LVLM_OK) return st;
        cta_kernel = d->cap > 2048;                      // ... the others get a CTA each
        min_m = 32 * 32 + 1;
    }
    if (cta_kernel) {
        // a CTA per head; warps without entries leave at once
        auto kernel = kpt == 4 ? (threads <= 256 ? kv_plan_kernel<4, 256> : kv_plan_kernel<4, 1024>)
                               : kpt == 8 ? kv_plan_kernel<8, 1024> : threads <= 256 ? kv_plan_kernel<16, 256> : kv_plan_kernel<16, 1024>;
        st = launch_kernel(kernel, dim3(d->Hkv, d->B), dim3(threads), 0, stream, 1, acc_score, pos, len, e_lo, e_hi, d->Hkv, d->cap,
                           d->recent, min_m, beta_ppm, budget, src_map, meta, nout, acc_new, pos_new, dev_status);
    }
#undef LVLM_PLAN_WARP
#undef LVLM_PLAN_WARP_
    if (st != LVLM_OK) return st;
    CompactJob j;
    j.base0 = Kc; j.base1 = Vc; j.stride_b = kv_sb * 2; j.stride_g = kv_sh * 2; j.B = d->B; j.G = d->Hkv;
    j.V = kHeadDim / 8; j.src_map = src_map; j.maps_per_g = d->Hkv; j.map_stride = d->cap;
    j.meta = meta; j.meta_stride = 1; j.nout = nout; j.N = d->cap;
    j.side_dst[0] = acc_score; j.side_src[0] = acc_new;
    if (pos) { j.side_dst[1] = pos; j.side_src[1] = pos_new; }
    return launch_inplace_compact(j, stream);
}
