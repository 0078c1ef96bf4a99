// Strip plan: Step 2 as three products over strips of query rows.
//
// The sweeps (gc_quad.cu, gc_tc.cu) form every logit twice, once per gradient, because nothing of
// size B x N may leave the chip.  A strip of query rows may: the exponentials of `rows` queries
// against all N passages fit the L2 for ordinary batches, and a bounded workspace for the rest.
// Per strip:
//
//   logit kernel   S = Q P^T on tcgen05, 256 x 256 tiles; the epilogue leaves, per row and group of
//                  64 columns, the raw maximum m and sum of e = 2^((s - m) log2e / tau) as a slot and
//                  the e themselves, each in [0, 1], in 16 bits (see stash_pack_small: off by at most 2^-11 of a
//                  value down to 2^-14, by 2^-9 of it down to 2^-126)
//   row kernel     merges a row's slots into row_lse, its share of the loss, and turns the row, in
//                  place, into the bf16 weights W_ij = p_ij - [j = r_i] (0 at the masked pair)
//   grad kernel    dQ = W P and dP += W^T Q in one launch; tiles of both products are dealt out in
//                  equal runs of 64-deep contraction blocks
//
// Six B N d multiply-adds for the six that count, against eight in the sweeps.  fp32 inputs take the
// same route with every value as three bf16 terms (x = t1 + t2 + t3 exactly): six products for S,
// the logits kept as fp32, weights as two terms, five products per gradient.  gc_loss_fwd runs the
// logit kernel without its stores; gc_loss_bwd's logit kernel is given row_lse and writes W itself.
//
// All matrix work runs in CTA pairs (cta_group::2, M = 256): two producer warps, one issuing warp
// (the leader's), eight epilogue warps; tensor memory holds two accumulators (fp32 gradients: four of half the
// width), so the epilogue of a tile runs under the next tile's products.  Every wait is bounded.
#include <cuda_fp16.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "tc_common.cuh"

namespace gc {

namespace {

constexpr int ST_THREADS = 32 * (NPROD + 1 + NSOFT);
constexpr int KB = 64;                               // contraction depth of a ring stage
constexpr int MAX_ST = 6;
constexpr int MAX_ACC = 4;                           // accumulators in tensor memory: two of 256 columns, four of 128
constexpr uint32_t HALF_CHUNK = 8192;                // 64 rows x 128 bytes
constexpr float LOG2E = 1.4426950408889634f;
constexpr float LN2 = 0.6931471805599453f;

enum LogitMode { LOGIT_FWD = 0, LOGIT_STASH = 1, LOGIT_W = 2, LOGIT_W2 = 3 };

struct StripBars {
    uint64_t full[MAX_ST];
    uint64_t empty[MAX_ST];
    uint64_t acc_full[MAX_ACC];
    uint64_t acc_free[MAX_ACC];        // this CTA's epilogue warps have read the buffer
    uint64_t acc_free_peer[MAX_ACC];   // leader: the same, forwarded from the second CTA
};

__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap* map, int c0, int c1,
                                                 int c2, uint32_t bar_cluster) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar_cluster)
        : "memory");
}
__device__ __forceinline__ void tma_add_3d(const CUtensorMap* map, uint32_t src, int c0, int c1,
                                           int c2) {
    asm volatile(
        "cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.bulk_group [%0, {%2, %3, %4}], [%1];"
        ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_read0() {
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
__device__ __forceinline__ void bulk_wait_all() {
    asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint32_t pack_h2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint32_t pack_b2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Exponentials of a group in 16 bits, two to a word.  Relative to the group's largest they cover as many
// octaves as the logits span (a passage far below a hard negative of its group still has a row of dP), which
// fp16 alone does not: below 2^-14 it rounds to multiples of 2^-24.  So: from 2^-14 on fp16, ten bits of
// mantissa, with a sign bit of 0; below, a sign bit of 1 and the upper 15 bits of the fp32 number without
// its sign, eight bits of mantissa, down to 2^-126.  The logits of most groups span fewer octaves: the second
// form costs them a minimum over the logits here.  A block of 32 rows x 64 columns that uses it marks its slots
// with a negative sum, so that the row kernel decides once per round of 2048 columns.
// Measured, us, kernels with fp16 alone / as they are: logit kernel of a build 1531 x 3062 x 768 11.7 / 12.1, of
// gradients 4096 x 8192 x 1024 54.6 / 56.5 and 4096 x 1024 x 768 14.7 / 15.5, row pass 6.1 / 6.1 (with a test per
// 16 bytes in place of the mark 6.4).
constexpr float STASH_FP16 = 6.103515625e-5f;            // 2^-14
__device__ __forceinline__ uint32_t stash_pack_small(uint32_t h, float a, float b) {
    if (a < STASH_FP16) h = (h & 0xffff0000u) | 0x8000u | ((__float_as_uint(a) + 0x4000u) >> 15);
    if (b < STASH_FP16) h = (h & 0xffffu) | 0x80000000u | ((__float_as_uint(b) + 0x4000u) >> 15 << 16);
    return h;
}
// what such a code stands for
__device__ __forceinline__ float stash_round_small(float a) {
    return __uint_as_float((__float_as_uint(a) + 0x4000u) & 0xffff8000u);
}
// f times the two numbers
__device__ __forceinline__ float2 stash_times(uint32_t h, float f) {
    const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&h));
    return make_float2(v.x * f, v.y * f);
}
__device__ __forceinline__ float2 stash_times_small(uint32_t h, float f) {
    float2 v = stash_times(h, f);
    if (h & 0x8000u) v.x = __uint_as_float((h & 0x7fffu) << 15) * f;
    if (h & 0x80000000u) v.y = __uint_as_float((h >> 16 & 0x7fffu) << 15) * f;
    return v;
}

// p - 1 of a positive from its raw logit (roundings spelled out: two kernels form it, same bits).
__device__ __forceinline__ float positive_weight(float raw, float inv_tau, float lse) {
    return __fsub_rn(ex2(__fmul_rn(__fsub_rn(__fmul_rn(raw, inv_tau), lse), LOG2E)), 1.f);
}

// ---- what every matrix kernel of this file shares: setup, teardown, forwarding ---------------------
struct PairCtx {
    uint32_t tmem;
    uint32_t rank;
    uint32_t smem;           // 1024-byte aligned dynamic shared memory
    int warp, lane;
};

__device__ __forceinline__ PairCtx pair_setup(uint8_t* raw, StripBars& bars, uint32_t* tmem_s,
                                              int* abort_s) {
    PairCtx c;
    c.warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    c.lane = threadIdx.x & 31;
    c.rank = cluster_ctarank();
    c.smem = (smem_u32(raw) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        *abort_s = 0;
        for (int s = 0; s < MAX_ST; ++s) {
            mbar_init(smem_u32(&bars.full[s]), 2);        // the leader's two producer warps
            mbar_init(smem_u32(&bars.empty[s]), 1);
        }
        for (int b = 0; b < MAX_ACC; ++b) {
            mbar_init(smem_u32(&bars.acc_full[b]), 1);
            mbar_init(smem_u32(&bars.acc_free[b]), NSOFT);
            mbar_init(smem_u32(&bars.acc_free_peer[b]), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (c.warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_s)), "r"((uint32_t)TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    c.tmem = *tmem_s;
    return c;
}

__device__ __forceinline__ void pair_teardown(const PairCtx& c, volatile int* abort_flag,
                                              int* dev_status) {
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // let bulk copies still in flight land before the shared memory is released
        uint64_t t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
        if (threadIdx.x == 0 && dev_status) atomicOr(dev_status, GC_DEV_WAIT_LIMIT);
        __syncthreads();
    }
    // By here nothing remote is under way: the leader has waited for every load and every forwarded arrival, the
    // second CTA for every product (its last accumulator) and every commit (ring_drained).
    cluster_meet();
    if (c.warp == MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;"
                     ::"r"(c.tmem), "r"((uint32_t)TMEM_COLS) : "memory");
    }
}

// The second CTA's idle issuing warp passes "buffer read" on to the leader: one remote arrival per
// use instead of eight (a remote arrival stalls the arriving warp for more than a thousand cycles).  Only
// what the leader waits for (wait_acc_free, of use n + NB): an arrival that nobody waits for could reach the
// leader's shared memory after it has left.
template <int NB = 2>
__device__ __forceinline__ void forward_acc_free(StripBars& bars, int uses, volatile int* abort_flag) {
    for (int n = 0; n < uses - NB; ++n) {
        const int b = n % NB;
        if (!mbar_wait(smem_u32(&bars.acc_free[b]), (uint32_t)(n / NB) & 1u, abort_flag)) return;
        if (elect_one()) mbar_arrive_cluster(mapa_u32(smem_u32(&bars.acc_free_peer[b]), 0));
    }
}
template <int NB = 2>
__device__ __forceinline__ bool wait_acc_free(StripBars& bars, int n, volatile int* abort_flag) {
    const int b = n % NB;
    const uint32_t par = ((uint32_t)(n / NB) & 1u) ^ 1u;
    return mbar_wait(smem_u32(&bars.acc_free[b]), par, abort_flag) &&
           mbar_wait(smem_u32(&bars.acc_free_peer[b]), par, abort_flag);
}

// The last step of a CTA's first producer, from where its ring stands: all stages have been given back.  The commits that
// give them back come from the leader into both CTAs; the last of them nobody else waits for.
__device__ __forceinline__ void ring_drained(StripBars& bars, int stages, int stage, uint32_t phase,
                                             volatile int* abort_flag) {
    for (int n = 0; n < stages; ++n) {
        if (!mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag)) return;
        if (++stage == stages) { stage = 0; phase ^= 1u; }
    }
}

// ---------------------------------------------------------------------------------------------------
// Logit kernel
// ---------------------------------------------------------------------------------------------------
struct LogitParams {
    int rows, N;                 // rows of the strip, passages
    int kblocks;                 // ceil(d / 64)
    int tiles_m, tiles_n;
    float c1;                    // log2(e) / tau
    float inv_tau;
    int mask_on, mask_shift;     // masked column of strip row i: i + mask_shift
    const int32_t* pos_idx;      // of the strip's rows
    int pos_base, pos_n;         // counted from passage pos_base of the pos_n a positive may point at
    const float* row_lse;        // LOGIT_W, LOGIT_W2
    const float* col_neg;        // LOGIT_W2: per passage, log2 of its multiplicity as a positive minus
                                 // its own logsumexp over the queries (log2 units; -inf: none)
    const float* col_lse;        // LOGIT_W2, may be NULL: that logsumexp; the terms of the loss of both
    const float* pos_logit;      // directions are then formed here
    float zero_anchor_lse;       // log B
    float* terms;
    float2* slots;               // [rows][slot_pitch] (raw maximum, sum; LOGIT_STASH: sum negated where the
                                 // group's codes are of both forms)
    int slot_pitch;
    float* pos_ws;               // positive's raw logit
    float* res;                  // LOGIT_W: what the positive's weight lost to bf16
    int* zero;                   // counters of the kernels that follow, cleared here
    int zero_count;
    int* zero2;                  // LOGIT_FWD, may be NULL: likewise
    int zero2_count;
    int* dev_status;
};

// Tile order: groups of 8 row tiles, row tiles fastest, so that the tiles in flight share operands.
__device__ __forceinline__ void logit_tile(int t, int tiles_m, int tiles_n, int* m, int* n) {
    const int per = 8 * tiles_n;
    const int g = t / per, r = t - g * per;
    const int h = min(8, tiles_m - 8 * g);
    *n = r / h;
    *m = 8 * g + (r - *n * h);
}

// Counters for the kernels that follow, cleared by the epilogue warps of every block of the grid, however
// few there are (thread: 0 .. 32 NSOFT - 1; NULL: nothing to clear).
__device__ __forceinline__ void clear_words(int* words, int count, int thread) {
    if (!words) return;
    for (int e = (int)blockIdx.x * (32 * NSOFT) + thread; e < count; e += (int)gridDim.x * (32 * NSOFT)) words[e] = 0;
}

// BN: passages per tile (a CTA loads BN / 2 of them).  What bounds it: tcgen05 at 256 x 256 tiles (a
// stage of 64 is 512 cycles of products for 32 KB per CTA); the epilogue's two special-function
// operations per 32 lanes and clock stay below that from d = 256 on.
template <int MODE, int BN>
__global__ void __launch_bounds__(ST_THREADS, 1)
strip_logit_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapP,
                   const __grid_constant__ CUtensorMap mapW, const LogitParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) StripBars bars;
    __shared__ uint32_t tmem_s;
    __shared__ int abort_s;
    volatile int* abort_flag = &abort_s;
    const PairCtx c = pair_setup(smem_raw, bars, &tmem_s, &abort_s);
    constexpr uint32_t A_BYTES = CHUNK_BYTES, B_BYTES = BN / 2 * 128, STAGE = A_BYTES + B_BYTES;
    // (weights are formed in the epilogue with row_lse given: it is the longer part there, and a second
    // staging buffer gives more than a sixth stage: 4096 x 8192 x 1024, 246 against 249 us per pass)
    constexpr int SB = MODE >= LOGIT_W && BN == 256 ? 2 : 1, NST = SB == 2 ? 5 : 6;
    const int total = p.tiles_m * p.tiles_n;
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    dep_release();
    dep_wait();

    if (c.warp < NPROD) {
        // warp 0: query rows, warp 1: passage rows
        const bool is_a = c.warp == 0;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int t = pair; t < total && ok; t += pairs) {
            int m, n;
            logit_tile(t, p.tiles_m, p.tiles_n, &m, &n);
            const int row = is_a ? m * 256 + (int)c.rank * 128 : n * BN + (int)c.rank * (BN / 2);
            for (int kb = 0; kb < p.kblocks; ++kb) {
                ok = mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag);
                if (!ok) break;
                const uint32_t full = smem_u32(&bars.full[stage]);
                const uint32_t full_leader = mapa_u32(full, 0);
                const uint32_t dst = c.smem + stage * STAGE + (is_a ? 0u : A_BYTES);
                if (elect_one()) {
                    if (c.rank == 0) mbar_expect_tx(full, 2 * (is_a ? A_BYTES : B_BYTES));
                    tma_load_3d_pair(dst, is_a ? &mapQ : &mapP, kb * KB, row, 0, full_leader);
                }
                if (++stage == NST) { stage = 0; phase ^= 1u; }
            }
        }
        if (ok && is_a) ring_drained(bars, NST, stage, phase, abort_flag);
    } else if (c.warp == MMA_WARP) {
        if (c.rank == 0) {
            const uint32_t idesc = instr_desc(BN, false, 256, false);
            int stage = 0, use = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int t = pair; t < total && ok; t += pairs, ++use) {
                ok = wait_acc_free(bars, use, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t acc = c.tmem + (use & 1) * 256;
                for (int kb = 0; kb < p.kblocks; ++kb) {
                    ok = mbar_wait(smem_u32(&bars.full[stage]), phase, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = desc_lo(c.smem + stage * STAGE, 0);
                    const uint32_t b = desc_lo(c.smem + stage * STAGE + A_BYTES, 0);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (k == 0 && kb == 0) mma_ss<false, true>(acc, a, b, idesc);
                            else                   mma_ss<true, true>(acc, a + 2 * k, b + 2 * k, idesc);
                        }
                        tc_commit_pair(smem_u32(&bars.empty[stage]));
                        if (kb == p.kblocks - 1) tc_commit_pair(smem_u32(&bars.acc_full[use & 1]));
                    }
                    if (++stage == NST) { stage = 0; phase ^= 1u; }
                }
            }
        } else {
            int uses = 0;
            for (int t = pair; t < total; t += pairs) ++uses;
            forward_acc_free(bars, uses, abort_flag);
        }
    } else {
        const int ew = c.warp - (NPROD + 1);
        const int q = c.warp & 3, half = ew >> 2, lane = c.lane;
        constexpr int HC = BN / 2;                       // columns of this warp
        clear_words(p.zero, p.zero_count, ew * 32 + lane);
        if (MODE == LOGIT_FWD) clear_words(p.zero2, p.zero2_count, ew * 32 + lane);
        const uint32_t stage_buf = c.smem + NST * STAGE + (uint32_t)ew * (SB * 4096u);
        const uint64_t c1_2 = pack2(p.c1, p.c1);
        int use = 0;
        for (int t = pair; t < total; t += pairs, ++use) {
            int m, n;
            logit_tile(t, p.tiles_m, p.tiles_n, &m, &n);
            const int row0 = m * 256 + (int)c.rank * 128 + 32 * q;
            const int i = row0 + lane;
            const int col0 = n * BN + half * HC;
            // the row's special columns
            int pos = -1, masked = -1;
            float neg_lse = -INFINITY, lse_i = 0.f;
            if (i < p.rows) {
                pos = p.pos_idx ? p.pos_idx[i] : -1;
                int flag = pos < 0 || pos >= p.pos_n ? GC_DEV_POS_RANGE : 0;
                pos -= p.pos_base;
                if (p.mask_on) {
                    masked = i + p.mask_shift;
                    if (pos == masked && !flag) flag = GC_DEV_POS_MASKED;
                }
                if (flag || pos < 0 || pos >= p.N) pos = -1;
                if (MODE == LOGIT_W || MODE == LOGIT_W2) {
                    lse_i = p.row_lse[i];
                    neg_lse = -(lse_i * LOG2E);
                    if (n == 0 && half == 0) {
                        if (pos < 0) p.res[i] = 0.f;     // no usable positive: nothing is lost to rounding
                        if (flag && p.dev_status) atomicOr(p.dev_status, flag);
                        // (the column direction of an unusable positive: a zero anchor row)
                        if (MODE == LOGIT_W2 && p.terms) {
                            const float pl = p.pos_logit[i];
                            p.terms[i] = 0.5f * ((lse_i - pl) + (flag ? p.zero_anchor_lse : p.col_lse[pos] - pl));
                        }
                    }
                }
            }
            if (!mbar_wait(smem_u32(&bars.acc_full[use & 1]), (uint32_t)(use >> 1) & 1u, abort_flag))
                break;
            tc_fence_after();
            const uint32_t src = c.tmem + (use & 1) * 256 + ((uint32_t)(32 * q) << 16) + half * HC;
            float run_m = -INFINITY, run_l = 0.f;
#pragma unroll 1
            for (int g = 0; g < HC / 64; ++g) {
                const int jg = col0 + 64 * g;
                float s[64];
                {
                    uint32_t v0[32], v1[32];
                    tmem_ld32(src + 64 * g, v0);
                    tmem_ld32(src + 64 * g + 32, v1);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        s[e] = __uint_as_float(v0[e]);
                        s[32 + e] = __uint_as_float(v1[e]);
                    }
                }
                if (g == HC / 64 - 1) {                  // the buffer is free for the tile after next
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bars.acc_free[use & 1]));
                }
                const int dp = pos - jg, dm = masked - jg;
                const bool special = (unsigned)dp < 64u || (unsigned)dm < 64u;
                const bool any_special = __any_sync(0xffffffffu, special) || jg + 64 > p.N;
                float pos_raw = 0.f;
                uint32_t h[MODE == LOGIT_STASH ? 32 : 1];        // the group's codes
                if (MODE != LOGIT_W2) {
                    float least = INFINITY;              // of the raw logits, special columns among them
                    if (MODE != LOGIT_FWD) {
                        float mn[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
                        for (int e = 4; e < 64; ++e) mn[e & 3] = fminf(mn[e & 3], s[e]);
                        least = fminf(fminf(mn[0], mn[1]), fminf(mn[2], mn[3]));
                    }
                    if (any_special) {
#pragma unroll
                        for (int e = 0; e < 64; ++e) {
                            if (e == dp) {
                                if (MODE == LOGIT_W) pos_raw = s[e];
                                else p.pos_ws[i] = s[e];
                            }
                            // the stored exponentials and their group's maximum leave the positive out:
                            // where it dominates its row, its neighbours keep their precision
                            if (e == dm || jg + e >= p.N || (MODE != LOGIT_FWD && e == dp)) s[e] = -INFINITY;
                        }
                    }
                    float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
                    for (int e = 4; e < 64; ++e) mx[e & 3] = fmaxf(mx[e & 3], s[e]);
                    const float gm = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                    // (a little before 2^-14, so that every smaller exponential finds its code)
                    const bool small = MODE != LOGIT_FWD && __any_sync(0xffffffffu, (least - gm) * p.c1 < -13.9f);
                    const float ref = gm == -INFINITY ? 0.f : gm;
                    const float off = -ref * p.c1;
                    const uint64_t off2 = pack2(off, off);
                    uint64_t sum2 = pack2(0.f, 0.f), sum2b = sum2;
#pragma unroll
                    for (int e = 0; e < 64; e += 4) {
                        float a, b, x, y;
                        unpack2(fma2(pack2(s[e], s[e + 1]), c1_2, off2), a, b);
                        unpack2(fma2(pack2(s[e + 2], s[e + 3]), c1_2, off2), x, y);
                        s[e] = ex2(a); s[e + 1] = ex2(b); s[e + 2] = ex2(x); s[e + 3] = ex2(y);
                        sum2 = add2(sum2, pack2(s[e], s[e + 1]));
                        sum2b = add2(sum2b, pack2(s[e + 2], s[e + 3]));
                    }
                    float sa, sb;
                    unpack2(add2(sum2, sum2b), sa, sb);
                    const float sum = sa + sb;
                    if (MODE == LOGIT_STASH) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) h[e] = pack_h2(s[2 * e], s[2 * e + 1]);
                        if (small) {
#pragma unroll
                            for (int e = 0; e < 32; ++e) h[e] = stash_pack_small(h[e], s[2 * e], s[2 * e + 1]);
                        }
                    }
                    if (MODE == LOGIT_STASH) {
                        if (i < p.rows) p.slots[(int64_t)i * p.slot_pitch + (jg >> 6)] = make_float2(gm, small ? -sum : sum);
                    } else if (MODE == LOGIT_W) {
                        // what the row kernel makes of the stored exponentials, bit for bit
                        const float f = gm > -INFINITY ? ex2(fmaf(gm, p.c1, neg_lse)) : 0.f;
                        if (small) {
#pragma unroll
                            for (int e = 0; e < 64; e += 2) {
                                const float2 v = stash_times(pack_h2(s[e], s[e + 1]), f);
                                s[e] = s[e] < STASH_FP16 ? stash_round_small(s[e]) * f : v.x;
                                s[e + 1] = s[e + 1] < STASH_FP16 ? stash_round_small(s[e + 1]) * f : v.y;
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < 64; e += 2) {
                                const float2 v = stash_times(pack_h2(s[e], s[e + 1]), f);
                                s[e] = v.x;
                                s[e + 1] = v.y;
                            }
                        }
                        if ((unsigned)dp < 64u) {
                            const float pw = positive_weight(pos_raw, p.inv_tau, lse_i);
                            p.res[i] = pw - __bfloat162float(__float2bfloat16_rn(pw));
#pragma unroll
                            for (int e = 0; e < 64; ++e) if (e == dp) s[e] = pw;
                        }
                    } else {
                        const float mn = fmaxf(run_m, gm), r = mn == -INFINITY ? 0.f : mn;
                        run_l = run_l * ex2((run_m - r) * p.c1) + sum * ex2((gm - r) * p.c1);
                        run_m = mn;
                    }
                } else {
                    const float4* cn = reinterpret_cast<const float4*>(p.col_neg + jg);
#pragma unroll
                    for (int e = 0; e < 64; e += 4) {
                        const float4 n4 = jg + e < p.N ? cn[e >> 2] : make_float4(0.f, 0.f, 0.f, 0.f);
                        const float nn[4] = {n4.x, n4.y, n4.z, n4.w};
#pragma unroll
                        for (int x = 0; x < 4; ++x)
                            s[e + x] = ex2(fmaf(s[e + x], p.c1, neg_lse)) + ex2(fmaf(s[e + x], p.c1, nn[x]));
                    }
                    if (any_special) {
#pragma unroll
                        for (int e = 0; e < 64; ++e) {
                            if (e == dp) {
                                s[e] -= 2.f;
                                p.res[i] = s[e] - __bfloat162float(__float2bfloat16_rn(s[e]));
                            }
                        }
                    }
                }
                if (MODE != LOGIT_FWD) {
                    // 32 rows x 64 columns of 16 bits, 128-byte swizzle, one bulk tensor store
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(SB - 1) : "memory");
                    __syncwarp();
                    const uint32_t box = stage_buf + (uint32_t)(g & (SB - 1)) * 4096u, buf = box + lane * 128;
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            w[e] = MODE == LOGIT_STASH ? h[MODE == LOGIT_STASH ? 4 * j + e : 0]
                                                       : pack_b2(s[8 * j + 2 * e], s[8 * j + 2 * e + 1]);
                        sts_v4(buf + (uint32_t)((j ^ (lane & 7)) << 4), w[0], w[1], w[2], w[3]);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {                     // (an empty group when nothing is stored)
                        if (row0 < p.rows && jg < p.N)
                            tma_store_3d(&mapW, box, jg, row0, 0);
                        else
                            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    }
                }
            }
            if (MODE == LOGIT_FWD && i < p.rows)
                p.slots[(int64_t)i * p.slot_pitch + 2 * n + half] = make_float2(run_m, run_l);
        }
        if (MODE != LOGIT_FWD) {
            if (lane == 0) bulk_wait_all();
            __syncwarp();
        }
    }
    pair_teardown(c, abort_flag, p.dev_status);
}

// fp32 inputs as three bf16 terms each ([3][rows][d] planes): 256 x 128 tiles, six products per step.
// The tensor core's additions truncate, so the leading product alternates between two accumulators
// and the five small ones have a third; the epilogue adds the three in fp32 and writes the raw logits.
// Bound by the products: 24 per stage of 72 KB per CTA.
constexpr int F_BN = 128;
constexpr uint32_t F_STAGE = 3 * CHUNK_BYTES + 3 * HALF_CHUNK;
constexpr int F_NST = 2;

__global__ void __launch_bounds__(ST_THREADS, 1)
strip_logit_f32_kernel(const __grid_constant__ CUtensorMap mapQ,
                       const __grid_constant__ CUtensorMap mapP,
                       const __grid_constant__ CUtensorMap mapS, const LogitParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) StripBars bars;
    __shared__ uint32_t tmem_s;
    __shared__ int abort_s;
    volatile int* abort_flag = &abort_s;
    const PairCtx c = pair_setup(smem_raw, bars, &tmem_s, &abort_s);
    const int total = p.tiles_m * p.tiles_n;
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    dep_release();
    dep_wait();

    if (c.warp < NPROD) {
        const bool is_a = c.warp == 0;
        const uint32_t bytes = is_a ? CHUNK_BYTES : HALF_CHUNK;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int t = pair; t < total && ok; t += pairs) {
            int m, n;
            logit_tile(t, p.tiles_m, p.tiles_n, &m, &n);
            const int row = is_a ? m * 256 + (int)c.rank * 128 : n * F_BN + (int)c.rank * (F_BN / 2);
            for (int kb = 0; kb < p.kblocks; ++kb) {
                ok = mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag);
                if (!ok) break;
                const uint32_t full = smem_u32(&bars.full[stage]);
                const uint32_t full_leader = mapa_u32(full, 0);
                const uint32_t dst = c.smem + stage * F_STAGE + (is_a ? 0u : 3 * CHUNK_BYTES);
                if (elect_one()) {
                    if (c.rank == 0) mbar_expect_tx(full, 6 * bytes);
                    for (int term = 0; term < 3; ++term)
                        tma_load_3d_pair(dst + term * bytes, is_a ? &mapQ : &mapP, kb * KB, row, term,
                                         full_leader);
                }
                if (++stage == F_NST) { stage = 0; phase ^= 1u; }
            }
        }
        if (ok && is_a) ring_drained(bars, F_NST, stage, phase, abort_flag);
    } else if (c.warp == MMA_WARP) {
        if (c.rank == 0) {
            const uint32_t idesc = instr_desc(F_BN, false, 256, false);
            int stage = 0, use = 0;
            uint32_t phase = 0;
            bool ok = true;
            for (int t = pair; t < total && ok; t += pairs, ++use) {
                // one set of accumulators: every use waits for the one before it
                ok = mbar_wait(smem_u32(&bars.acc_free[0]), ((uint32_t)use & 1u) ^ 1u, abort_flag) &&
                     mbar_wait(smem_u32(&bars.acc_free_peer[0]), ((uint32_t)use & 1u) ^ 1u, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t rest = c.tmem + 256;
                for (int kb = 0; kb < p.kblocks; ++kb) {
                    ok = mbar_wait(smem_u32(&bars.full[stage]), phase, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    constexpr uint32_t TA = CHUNK_BYTES >> 4, TB = HALF_CHUNK >> 4;
                    const uint32_t a0 = desc_lo(c.smem + stage * F_STAGE, 0);
                    const uint32_t b0 = desc_lo(c.smem + stage * F_STAGE + 3 * CHUNK_BYTES, 0);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const uint32_t a = a0 + 2 * k, b = b0 + 2 * k;
                            const uint32_t lead = c.tmem + 128 * (k & 1);
                            if (kb == 0 && k < 2) mma_ss<false, true>(lead, a, b, idesc);
                            else                  mma_ss<true, true>(lead, a, b, idesc);
                            if (kb == 0 && k == 0) mma_ss<false, true>(rest, a, b + TB, idesc);
                            else                   mma_ss<true, true>(rest, a, b + TB, idesc);
                            mma_ss<true, true>(rest, a + TA, b, idesc);
                            mma_ss<true, true>(rest, a + TA, b + TB, idesc);
                            mma_ss<true, true>(rest, a, b + 2 * TB, idesc);
                            mma_ss<true, true>(rest, a + 2 * TA, b, idesc);
                        }
                        tc_commit_pair(smem_u32(&bars.empty[stage]));
                        if (kb == p.kblocks - 1) tc_commit_pair(smem_u32(&bars.acc_full[0]));
                    }
                    if (++stage == F_NST) { stage = 0; phase ^= 1u; }
                }
            }
        } else {
            // (the leader waits for every use but the last)
            int n = 0;
            for (int t = pair; t + pairs < total; t += pairs, ++n) {
                if (!mbar_wait(smem_u32(&bars.acc_free[0]), (uint32_t)n & 1u, abort_flag)) break;
                if (elect_one()) mbar_arrive_cluster(mapa_u32(smem_u32(&bars.acc_free_peer[0]), 0));
            }
        }
    } else {
        const int ew = c.warp - (NPROD + 1);
        const int q = c.warp & 3, half = ew >> 2, lane = c.lane;
        clear_words(p.zero, p.zero_count, ew * 32 + lane);
        const uint32_t slot = c.smem + F_NST * F_STAGE + (uint32_t)ew * 8192u;
        int use = 0;
        for (int t = pair; t < total; t += pairs, ++use) {
            int m, n;
            logit_tile(t, p.tiles_m, p.tiles_n, &m, &n);
            const int row0 = m * 256 + (int)c.rank * 128 + 32 * q;
            const int col0 = n * F_BN + 64 * half;
            if (!mbar_wait(smem_u32(&bars.acc_full[0]), (uint32_t)use & 1u, abort_flag)) break;
            tc_fence_after();
            const uint32_t src = c.tmem + ((uint32_t)(32 * q) << 16) + 64 * half;
            uint32_t s[2][32];
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                uint32_t v[32], u[32];
                tmem_ld32(src + 32 * g, s[g]);
                tmem_ld32(src + 128 + 32 * g, v);
                tmem_ld32(src + 256 + 32 * g, u);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    s[g][e] = __float_as_uint((__uint_as_float(s[g][e]) + __uint_as_float(v[e])) +
                                              __uint_as_float(u[e]));
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(smem_u32(&bars.acc_free[0]));
                bulk_wait_read0();
            }
            __syncwarp();
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                stage_block(slot + g * 4096, s[g], 1.f, lane);
                __syncwarp();
                if (lane == 0 && row0 < p.rows && col0 + 32 * g < p.N)
                    tma_store_3d(&mapS, slot + g * 4096, col0 + 32 * g, row0, 0);
            }
        }
        if (lane == 0) bulk_wait_all();
        __syncwarp();
    }
    pair_teardown(c, abort_flag, p.dev_status);
}

// x = t1 + t2 + t3, each term the upper 16 bits of what the earlier ones left: planes [3][rows][ldt].
__device__ __forceinline__ void split3(float x, uint32_t& t1, uint32_t& t2, uint32_t& t3) {
    t1 = __float_as_uint(x) & 0xffff0000u;
    const float r = x - __uint_as_float(t1);
    t2 = __float_as_uint(r) & 0xffff0000u;
    t3 = __float_as_uint(r - __uint_as_float(t2));
}
__global__ void __launch_bounds__(256)
split_terms_kernel(const float* Q, int64_t ldq, int64_t B, uint2* __restrict__ tq,
                   const float* P, int64_t ldp, int64_t N, uint2* __restrict__ tp,
                   int d4) {
    dep_release();
    dep_wait();
    const int64_t nq = B * d4, total = nq + N * d4;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const bool is_q = e < nq;
        const int64_t f = is_q ? e : e - nq;
        const int64_t r = f / d4;
        const int c = 4 * (int)(f - r * d4);
        const float4 x = *reinterpret_cast<const float4*>(is_q ? Q + r * ldq + c : P + r * ldp + c);
        const int64_t plane = is_q ? nq : N * d4;
        uint2* dst = (is_q ? tq : tp) + f;
        uint32_t a[4], b[4], t[4];
        split3(x.x, a[0], b[0], t[0]); split3(x.y, a[1], b[1], t[1]);
        split3(x.z, a[2], b[2], t[2]); split3(x.w, a[3], b[3], t[3]);
        dst[0] = make_uint2(__byte_perm(a[0], a[1], 0x7632), __byte_perm(a[2], a[3], 0x7632));
        dst[plane] = make_uint2(__byte_perm(b[0], b[1], 0x7632), __byte_perm(b[2], b[3], 0x7632));
        dst[2 * plane] = make_uint2(__byte_perm(t[0], t[1], 0x7632), __byte_perm(t[2], t[3], 0x7632));
    }
}

// ---------------------------------------------------------------------------------------------------
// Row kernel
// ---------------------------------------------------------------------------------------------------
struct RowParams {
    int rows, N;
    int row0;                     // first row of the strip within the call
    float c1, inv_tau;
    int mask_on, mask_shift;      // masked column of strip row i: i + mask_shift
    const int32_t* pos_idx;       // of the strip's rows
    int pos_base, pos_n;          // as in LogitParams
    const float2* slots;
    int slot_pitch, nslots;
    const float* pos_ws;
    float* res;
    float* row_lse;               // of the strip's rows: written, or read when lse_given
    float* pos_logit;             // may be NULL
    float* loss;
    float* red;                   // with weights: one loss term per row of the call, summed by the
                                  // gradient kernel; otherwise one share per block of the call
    int* ticket;
    int block0, blocks_total;     // this launch's first block and the blocks of all strips
    float inv_mean;
    int64_t ldw;                  // elements
    int split;                    // strip_row_kernel<true>: 2^split warps share a row's rounds
    int seg_rounds;               // strip_row_kernel<true>: rounds of 2048 columns per segment
    int* dev_status;
    // fp32 inputs
    const float* S;
    int64_t lds;
    int lse_given, want_w;
    // two-direction loss
    int* count;                   // queries per passage, counted here
    const int* mult;              // rows are passages: their counts, and
    float* col_neg;               // where LOGIT_W2's column factors go
};

// Shares of the loss, EACH per block (of its first threads), are added in a fixed order: a share's rows in row
// order, then the shares in a fixed pattern by the block that draws the last ticket.
template <int EACH = 1>
__device__ __forceinline__ void loss_share(const RowParams& p, float mine) {
    __shared__ int last_s;
    __shared__ float warp_s[8];
    if (threadIdx.x < EACH) {
        p.red[(p.block0 + blockIdx.x) * EACH + threadIdx.x] = mine;
        __threadfence();
    }
    if (EACH > 1) __syncthreads();
    if (threadIdx.x == 0) {
        last_s = atomicAdd(p.ticket, 1) == p.blocks_total - 1;
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    float v = 0.f;
#pragma unroll 4
    for (int b = threadIdx.x; b < p.blocks_total * EACH; b += blockDim.x) v += __ldcg(p.red + b);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) warp_s[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.f;
        for (int w = 0; w < (int)blockDim.x / 32; ++w) s += warp_s[w];
        *p.loss = s * p.inv_mean;
    }
}

// The positive of strip row i as a column of the strip (-1: none there), and what is wrong with it.
__device__ __forceinline__ int row_pos(const RowParams& p, int i, int* flags) {
    const int raw = p.pos_idx ? p.pos_idx[i] : -1, pos = raw - p.pos_base;
    *flags = raw < 0 || raw >= p.pos_n ? GC_DEV_POS_RANGE
             : p.mask_on && pos == i + p.mask_shift ? GC_DEV_POS_MASKED : 0;
    return *flags || pos < 0 || pos >= p.N ? -1 : pos;
}

// bf16 inputs: a warp per row, or (WRITE) 2^split warps, each taking every 2^split-th round of 2048
// columns of the block's segment.  They merge the row's (max, sum) slots, form row_lse, the positive's
// weight and the loss term, then turn the row's 16-bit exponentials into bf16 weights in place: eight
// 16-byte pieces in flight per lane, each one's successor requested as soon as it has been used, the
// slots of the next round with them; one special-function operation per group of 64 columns, its result
// passed around by shuffles.  Rows go last to first: the logits written last are still in the L2.
// Bound by the latency and bandwidth of the memory (4 bytes moved per pair).  Measured, us, one warp per
// row, rows in order, each round's slots read when it begins -> as it is now:
//   1531 x 3062  5.9 -> 4.7   4096 x 8192  23.8 -> 20.3   6000 x 12000   76 -> 48
//   2048 x 32768  62 -> 52    8192 x 16384  120 -> 91     4096 x 131072 480 -> 387 (5.5 TB/s)
// RESIDENT, the blocks an SM is to hold: seven (72 registers a thread), six where the grid then fits in
// one go (1531 x 3062: 5.1 us with seven, 4.7 with six; 4096 x 8192: 20.3 and 22.0).
constexpr int row_warps(bool write) { return write ? 4 : 8; }      // rows per block
constexpr int MOST_THREAD_SLOTS = 8;                // strip_lse_kernel
constexpr int ROW_PIECES = 8;                       // of 8 columns, per lane and round
constexpr int ROW_ROUND = 32 * ROW_PIECES;          // pieces per warp and round: 32 groups of 64 columns
template <bool WRITE, int RESIDENT>
__global__ void __launch_bounds__(WRITE ? 128 : 256, RESIDENT)
strip_row_kernel(uint4* __restrict__ W, const RowParams p) {
    constexpr int ROW_WARPS = WRITE ? 4 : 8;
    __shared__ float terms[ROW_WARPS];
    __shared__ float2 shares[ROW_WARPS];
    dep_release();
    dep_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int split = WRITE ? p.split : 0, sub = warp & ((1 << split) - 1);
    // the rows written last come first: they are still in the L2
    const int block = WRITE ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x;
    const int i = (block * ROW_WARPS + warp) >> split;
    const bool live = i < p.rows;
    const int n8 = (p.N + 7) / 8, stride = ROW_ROUND << split;
    const int s0 = WRITE ? (int)blockIdx.y * p.seg_rounds * ROW_ROUND : 0;
    const int k0 = s0 + sub * ROW_ROUND;
    const int k1 = WRITE ? min(n8, s0 + p.seg_rounds * ROW_ROUND) : 0;
    const float2* sl = p.slots + (int64_t)(live ? i : 0) * p.slot_pitch;
    uint4* row = W + (int64_t)(live ? i : 0) * (p.ldw / 8);
    // (max, sum) of the row: from the slots, shared out over the row's warps where there are many, and,
    // with weights, from the positive, which is not in the slots then.  All but the first two of a lane
    // come before the row's own pieces take their registers.
    const int shared = p.nslots > 64 ? split : 0;
    const int step = 32 << shared, first_slot = (shared ? sub * 32 : 0) + lane;
    float m = -INFINITY, l = 0.f, pos_raw = -INFINITY;
    int flags = 0, pos = -1;
    auto slot = [&](int s) { return s < p.nslots ? __ldcg(sl + s) : make_float2(-INFINITY, 0.f); };
    auto join = [&](float2 v, float ref) { l = fmaf(WRITE ? fabsf(v.y) : v.y, ex2((v.x - ref) * p.c1), l); };
    if (live) {
        for (int s = first_slot + 2 * step; s < p.nslots; s += 8 * step) {
            float2 v[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) v[x] = slot(s + step * x);
            float top = m;
#pragma unroll
            for (int x = 0; x < 8; ++x) top = fmaxf(top, v[x].x);
            const float ref = top == -INFINITY ? 0.f : top;
            l *= ex2((m - ref) * p.c1);
#pragma unroll
            for (int x = 0; x < 8; ++x) join(v[x], ref);
            m = top;
        }
    }
    uint4 raw[ROW_PIECES];
    if (WRITE && live) {
#pragma unroll
        for (int x = 0; x < ROW_PIECES; ++x) {
            const int k = k0 + lane + 32 * x;
            if (k < k1) raw[x] = __ldcg(row + k);
        }
    }
    if (live) {
        const float2 v0 = slot(first_slot), v1 = slot(first_slot + step);
        pos_raw = __ldcg(p.pos_ws + i);
        pos = row_pos(p, i, &flags);
        if (pos < 0) pos_raw = -INFINITY;
        float top = fmaxf(m, fmaxf(v0.x, v1.x));
        if (WRITE) top = fmaxf(top, pos_raw);
        for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
        const float ref = top == -INFINITY ? 0.f : top;
        l *= ex2((m - ref) * p.c1);
        join(v0, ref);
        join(v1, ref);
        m = top;
        if (WRITE && lane == 0 && (!shared || sub == 0)) l += ex2((pos_raw - ref) * p.c1);
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    }
    if (WRITE && shared) {
        if (lane == 0) shares[warp] = make_float2(m, l);
        __syncthreads();
        const int first = warp - sub;
        for (int w = 0; w < 1 << split; ++w) m = fmaxf(m, shares[first + w].x);
        const float ref = m == -INFINITY ? 0.f : m;
        l = 0.f;
        for (int w = 0; w < 1 << split; ++w) l = fmaf(shares[first + w].y, ex2((shares[first + w].x - ref) * p.c1), l);
    }
    if (live) {
        const float lse = m * p.inv_tau + log2f(l) * LN2;
        const float pl = pos < 0 ? 0.f : pos_raw * p.inv_tau;
        const float pw = positive_weight(pos_raw, p.inv_tau, lse);
        if (lane == 0) {
            terms[warp] = lse - pl;
            if (!WRITE || (blockIdx.y == 0 && sub == 0)) {
                p.row_lse[i] = lse;
                if (p.pos_logit) p.pos_logit[i] = pl;
                if (flags && p.dev_status) atomicOr(p.dev_status, flags);
                if (!WRITE && p.count && pos >= 0) atomicAdd(p.count + pos, 1);
                if (!WRITE && p.col_neg) {
                    const int n = p.mult[i];
                    p.col_neg[i] = n > 0 ? log2f((float)n) - lse * LOG2E : -INFINITY;
                }
                if (WRITE) {
                    p.red[p.row0 + i] = lse - pl;
                    p.res[i] = pos < 0 ? 0.f : pw - __bfloat162float(__float2bfloat16_rn(pw));
                }
            }
        }
        if (WRITE) {
            const float neg = -(lse * LOG2E);
            const int wk = pos < 0 ? -1 : pos >> 3;
            // round after round: lane g of a round holds the factor of its group of 64 columns
            auto slot_of = [&](int kr) {
                const int g = (kr >> 3) + lane;
                return g < p.nslots ? __ldcg(sl + g) : make_float2(-INFINITY, 0.f);
            };
            float2 next = slot_of(k0);
            for (int kr = k0; kr < k1; kr += stride) {
                // (a group with no allowed column holds zeros)
                const float2 now = next;
                if (kr + stride < k1) next = slot_of(kr + stride);
                const float fg = now.x > -INFINITY ? ex2(fmaf(now.x, p.c1, neg)) : 0.f;
                auto weights = [&](int k, const float2 (&v)[4]) {
                    float w[8];
#pragma unroll
                    for (int e = 0; e < 4; ++e) { w[2 * e] = v[e].x; w[2 * e + 1] = v[e].y; }
                    if (wk == k) {
#pragma unroll
                        for (int e = 0; e < 8; ++e) if (e == (pos & 7)) w[e] = pw;
                    }
                    row[k] = make_uint4(pack_b2(w[0], w[1]), pack_b2(w[2], w[3]),
                                        pack_b2(w[4], w[5]), pack_b2(w[6], w[7]));
                };
                if (!__any_sync(0xffffffffu, now.y < 0.f)) {
#pragma unroll
                    for (int x = 0; x < ROW_PIECES; ++x) {
                        const float f = __shfl_sync(0xffffffffu, fg, 4 * x + (lane >> 3));
                        const int k = kr + lane + 32 * x;
                        if (k >= k1) continue;
                        const float2 v[4] = {stash_times(raw[x].x, f), stash_times(raw[x].y, f),
                                             stash_times(raw[x].z, f), stash_times(raw[x].w, f)};
                        weights(k, v);
                        if (k + stride < k1) raw[x] = __ldcg(row + k + stride);
                    }
                } else {
                    // both forms: one piece after the other, read again (code kept short: unrolled like the other it
                    // cost every launch, 872 x 872 x 768 22.2 us a build against 21.7)
#pragma unroll 1
                    for (int x = 0; x < ROW_PIECES; ++x) {
                        const float f = __shfl_sync(0xffffffffu, fg, 4 * x + (lane >> 3));
                        const int k = kr + lane + 32 * x;
                        if (k >= k1) continue;
                        const uint4 h = __ldcg(row + k);
                        const float2 v[4] = {stash_times_small(h.x, f), stash_times_small(h.y, f),
                                             stash_times_small(h.z, f), stash_times_small(h.w, f)};
                        weights(k, v);
                    }
#pragma unroll
                    for (int x = 0; x < ROW_PIECES; ++x) {
                        const int k = kr + lane + 32 * x + stride;
                        if (k < k1) raw[x] = __ldcg(row + k);
                    }
                }
            }
        }
    }
    if (!WRITE) {
        __syncthreads();
        float share = 0.f;
        if (threadIdx.x == 0)
            for (int w = 0; w < ROW_WARPS && blockIdx.x * ROW_WARPS + w < p.rows; ++w) share += terms[w];
        loss_share(p, share);
    }
}

// The loss alone where a row has few slots and there are many rows: a thread per row (strip_row_kernel<false>
// gives a warp to the two slots of 256 passages: 64000 x 128, 32.7 us a launch, 6.3 here; 8000 rows are even).
__global__ void __launch_bounds__(256)
strip_lse_kernel(const RowParams p) {
    __shared__ float sums[8];
    dep_release();
    dep_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 256 + (int)threadIdx.x;
    float term = 0.f;
    if (i < p.rows) {
        const float2* sl = p.slots + (int64_t)i * p.slot_pitch;
        float2 v[MOST_THREAD_SLOTS];
        float m = -INFINITY, l = 0.f;
#pragma unroll
        for (int s = 0; s < MOST_THREAD_SLOTS; ++s) {
            v[s] = s < p.nslots ? __ldcg(sl + s) : make_float2(-INFINITY, 0.f);
            m = fmaxf(m, v[s].x);
        }
        int flags;
        const int pos = row_pos(p, i, &flags);
        const float ref = m == -INFINITY ? 0.f : m;
#pragma unroll
        for (int s = 0; s < MOST_THREAD_SLOTS; ++s) l = fmaf(v[s].y, ex2((v[s].x - ref) * p.c1), l);
        const float lse = m * p.inv_tau + log2f(l) * LN2;
        const float pl = pos < 0 ? 0.f : __ldcg(p.pos_ws + i) * p.inv_tau;
        p.row_lse[i] = lse;
        if (p.pos_logit) p.pos_logit[i] = pl;
        if (flags && p.dev_status) atomicOr(p.dev_status, flags);
        if (p.count && pos >= 0) atomicAdd(p.count + pos, 1);
        if (p.col_neg) {
            const int n = p.mult[i];
            p.col_neg[i] = n > 0 ? log2f((float)n) - lse * LOG2E : -INFINITY;
        }
        term = lse - pl;
    }
    for (int o = 16; o > 0; o >>= 1) term += __shfl_xor_sync(0xffffffffu, term, o);
    if (lane == 0) sums[warp] = term;
    __syncthreads();
    float share = 0.f;
    if (threadIdx.x == 0)
        for (int w = 0; w < 8; ++w) share += sums[w];
    loss_share(p, share);
}

// fp32 inputs: one block (BLOCK = true), or a warp of it, per row of raw logits.  Maximum, sum and weights
// are three passes over the row (from the first level cache after the first; a warp from 101776 rows of 34: 49 us,
// a block 269); the weights leave as two
// bf16 terms, planes [2][rows][ldw].  With lse_given (gc_loss_bwd) only the last pass runs.
template <bool BLOCK>
__global__ void __launch_bounds__(256)
strip_row_f32_kernel(uint2* __restrict__ W, const RowParams p) {
    __shared__ float sm[8];
    dep_release();
    dep_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int T = BLOCK ? 256 : 32;                  // threads of a row
    const int t = BLOCK ? (int)threadIdx.x : lane;
    const int n4 = (p.N + 3) / 4;
    float share = 0.f;
    for (int i = BLOCK ? blockIdx.x : blockIdx.x * 8 + warp; i < p.rows; i += (int)gridDim.x * (BLOCK ? 1 : 8)) {
        const float4* row = reinterpret_cast<const float4*>(p.S + (int64_t)i * p.lds);
        const int masked = p.mask_on ? i + p.mask_shift : -1;
        int flags;
        const int pos = row_pos(p, i, &flags);
        if (t == 0 && flags && p.dev_status) atomicOr(p.dev_status, flags);
        auto load = [&](int k, float (&s)[4]) {
            const float4 v = row[k];
            s[0] = v.x; s[1] = v.y; s[2] = v.z; s[3] = v.w;
#pragma unroll
            for (int e = 0; e < 4; ++e) if (4 * k + e == masked || 4 * k + e >= p.N) s[e] = -INFINITY;
        };
        auto row_max = [&](float v) {
            for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
            if (!BLOCK) return v;
            if (lane == 0) sm[warp] = v;
            __syncthreads();
            v = sm[0];
            for (int w = 1; w < 8; ++w) v = fmaxf(v, sm[w]);
            __syncthreads();
            return v;
        };
        auto row_sum = [&](float v) {
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (!BLOCK) return v;
            if (lane == 0) sm[warp] = v;
            __syncthreads();
            v = sm[0];
            for (int w = 1; w < 8; ++w) v += sm[w];
            __syncthreads();
            return v;
        };
        float lse;
        const float raw_pos = pos < 0 ? 0.f : p.S[(int64_t)i * p.lds + pos];
        if (p.lse_given) {
            lse = p.row_lse[i];
        } else {
            float m = -INFINITY;
#pragma unroll 4
            for (int k = t; k < n4; k += T) {
                float s[4];
                load(k, s);
                m = fmaxf(m, fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3])));
            }
            m = row_max(m);
            const float ref = m == -INFINITY ? 0.f : m;
            float l = 0.f;
#pragma unroll 4
            for (int k = t; k < n4; k += T) {
                float s[4];
                load(k, s);
#pragma unroll
                for (int e = 0; e < 4; ++e) l += ex2((s[e] - ref) * p.c1);
            }
            l = row_sum(l);
            // the row's logsumexp and its positive logit come out of the same product with 1/tau: their
            // difference is exactly 0 when the positive is the only column
            lse = m * p.inv_tau + log2f(l) * LN2;
            const float pl = raw_pos * p.inv_tau;
            if (t == 0) {
                p.row_lse[i] = lse;
                if (p.pos_logit) p.pos_logit[i] = pl;
            }
            share += lse - pl;
            if (p.want_w && t == 0) p.red[p.row0 + i] = lse - pl;
        }
        if (p.want_w) {
            const float lse2 = lse * LOG2E;
            uint2* w1 = W + (int64_t)i * (p.ldw / 4);
            uint2* w2 = w1 + (int64_t)p.rows * (p.ldw / 4);
            const int wpos = pos;
#pragma unroll 4
            for (int k = t; k < n4; k += T) {
                float s[4];
                load(k, s);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    s[e] = ex2(fmaf(s[e], p.c1, -lse2));
                    if (4 * k + e == wpos) s[e] -= 1.f;
                }
                const uint32_t h0 = pack_b2(s[0], s[1]), h1 = pack_b2(s[2], s[3]);
                w1[k] = make_uint2(h0, h1);
                w2[k] = make_uint2(pack_b2(s[0] - __uint_as_float(h0 << 16), s[1] - __uint_as_float(h0 & 0xffff0000u)),
                                   pack_b2(s[2] - __uint_as_float(h1 << 16), s[3] - __uint_as_float(h1 & 0xffff0000u)));
            }
        }
    }
    if (!p.lse_given && !p.want_w) {
        // (a build adds the terms row by row in the same pattern: up to 8 rows per SM and warp, the same bits)
        if (!BLOCK) {
            if (lane == 0) sm[warp] = share;
            __syncthreads();
            loss_share<8>(p, threadIdx.x < 8 ? sm[threadIdx.x] : 0.f);
        } else {
            loss_share(p, share);
        }
    }
}

// ---------------------------------------------------------------------------------------------------
// Gradient kernel
// ---------------------------------------------------------------------------------------------------
struct GradSide {
    int tiles;                    // output tiles: 256 rows x `width` columns, columns fastest
    int tiles_n;
    int kblocks;                  // contraction blocks of 64
    int rows, cols;               // of the output
    int add;                      // 1: add to the output (strips after the first)
};

struct GradParams {
    GradSide side[2];             // 0: dQ = W P, 1: dP = W^T Q
    // How the tiles are dealt out to the CTA pairs.  whole >= 0: as whole tiles, dQ's to the first
    // `whole` pairs in turn, dP's to the others.  whole < 0: tiles_n neighbouring pairs form a group
    // (one pair per column tile, in step, so that they share the rows of W they read); the row tiles
    // of dQ, then of dP, are laid end to end and cut into `groups` equal runs of contraction blocks.
    int whole;
    int pairs;
    int units;                    // contraction blocks of all row tiles
    int groups;
    float scale;                  // 1 / (B tau)
    const float* res;             // dQ: what the positives' weights lost to bf16 (NULL: nothing)
    const int32_t* pos_idx;
    const __nv_bfloat16* P;       // passages, for the res terms
    int64_t ldp;
    const float* terms;           // loss terms of all rows of the call (NULL: no loss to form here)
    int n_terms;
    float inv_mean;
    float* loss;
    float* out[2];                // dQ, dP, and their pitches
    int64_t ldo[2];
    float* part;                  // [pairs][2 slots][2 CTAs][8 warps][32 x hw] partial tiles
    int* count;                   // [tiles of both sides][2 CTAs][8 warps]: shares in memory, and pieces of
                                  // their sum drawn << 16
    int* started;                 // pairs that have started, over the strips of the call, and how many of them when
    int all_started;              // all of this launch have (cut runs only)
    int* dev_status;
};

// A run of contraction blocks of one output tile.
struct Segment {
    int side, tile_m, tile_n, kb, n;
    int t0;                       // whole < 0: first unit of the row tile
};

// units * groups stays below 2^32: rows x passages of a strip are at most 768 M, or 256 x 2^24
__device__ __forceinline__ int unit_start(const GradParams& p, int g) {
    return (int)((unsigned)p.units * (unsigned)g / (unsigned)p.groups);
}
// Iterates over a pair's segments.  In a cut run the two cut tiles come first (their partial sums meet
// under the products of the tiles that follow), the whole ones after them.
struct SegmentWalk {
    int u, end, group, tile_n;    // whole >= 0: u counts tiles
    int phase;
    __device__ __forceinline__ SegmentWalk(const GradParams& p, int pair) {
        phase = 0;
        if (p.whole >= 0) {
            const bool q = pair < p.whole;
            u = q ? pair : pair - p.whole;
            end = p.side[q ? 0 : 1].tiles;
            group = q ? p.whole : p.pairs - p.whole;        // stride
            tile_n = q ? 0 : 1;                             // side
        } else {
            group = pair / p.side[0].tiles_n;
            tile_n = pair - group * p.side[0].tiles_n;
            u = unit_start(p, group);
            end = unit_start(p, group + 1);
        }
    }
    // the tile that unit v lies in, and the part of it in [u, end)
    __device__ __forceinline__ void locate(const GradParams& p, int v, Segment& s) const {
        const int first_p = p.side[0].tiles / p.side[0].tiles_n * p.side[0].kblocks;
        s.side = v >= first_p;
        const int k = s.side ? p.side[1].kblocks : p.side[0].kblocks;
        const int local = v - (s.side ? first_p : 0);
        s.tile_m = local / k;
        s.tile_n = tile_n;
        s.t0 = v - (local - s.tile_m * k);
        s.kb = max(u - s.t0, 0);
        s.n = min(k, end - s.t0) - s.kb;
    }
    __device__ __forceinline__ bool next(const GradParams& p, Segment& s) {
        if (u >= end) return false;
        if (p.whole >= 0) {
            s.side = tile_n;
            s.tile_m = u / p.side[0].tiles_n;
            s.tile_n = u - s.tile_m * p.side[0].tiles_n;
            s.kb = 0;
            s.n = s.side ? p.side[1].kblocks : p.side[0].kblocks;
            s.t0 = 0;
            u += group;
            return true;
        }
        if (phase == 0) {
            phase = 1;
            locate(p, u, s);
            if (s.kb > 0) { u += s.n; return true; }
        }
        if (phase == 1) {
            phase = 2;
            locate(p, end - 1, s);
            if (s.n < (s.side ? p.side[1].kblocks : p.side[0].kblocks)) { end -= s.n; return true; }
        }
        locate(p, u, s);
        u += s.n;
        return true;
    }
};

// A warp that has nothing left to do waits so long for the other shares of its last tile, if every pair of the launch
// has started.  Measured on an idle device, over 19 shapes: nearly all waits end within 3 us, the longest after 6.
constexpr uint64_t SUM_WAIT_NS = 10000;
constexpr int SUM_TAKEN = 0x8000;             // the last warp sums from tensor memory

// A tile cut between groups is summed from partial tiles in contraction order (the order of the sum, not of the
// arrivals, decides the bits).  The last warp to finish a share sees that all are in memory and sums them; warps
// that finished theirs before, and have no other work, are still there as a rule and draw pieces of the sum as well.
// Nobody depends on them: they leave after SUM_WAIT_NS, and at once while pairs of this launch have yet to start, which
// may need the room they hold; what has not been drawn is left to the last.
// (One rank's dQ of 512 x 8192 x 768, 10 shares to a tile: the last warp alone spent up to 15 K cycles on its 32 x 64
// sums, the warps together 6-8 K; one rank of eight of 4096 x 8192 x 768 71.7 -> 67.5 us.  dQ of 256 x 16384 x 768 with
// 20 SMs held by another stream: 76 us with waits of up to 20 us for pairs that could not start, 56 without them; 28
// on a free device; two streams of it at once 53 and 50 a pair of calls.)
//
// F32: weights as two terms, rows of the other side as three; products w1 (t1 + t2 + t3) +
// w2 (t1 + t2), 256 x 128 tiles.  The tensor core's additions truncate: every 128 of the contraction
// the accumulator is read out and added in fp32 registers, the next of the four taking over meanwhile.
template <bool F32, int WIDTH>
__global__ void __launch_bounds__(ST_THREADS, 1)
strip_grad_kernel(const __grid_constant__ CUtensorMap mapWk, const __grid_constant__ CUtensorMap mapWm,
                  const __grid_constant__ CUtensorMap mapP, const __grid_constant__ CUtensorMap mapQ,
                  const __grid_constant__ CUtensorMap mapDQ, const __grid_constant__ CUtensorMap mapDP,
                  const __grid_constant__ GradParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) StripBars bars;
    __shared__ uint32_t tmem_s;
    __shared__ int abort_s;
    volatile int* abort_flag = &abort_s;
    const PairCtx c = pair_setup(smem_raw, bars, &tmem_s, &abort_s);
    constexpr int TA = F32 ? 2 : 1, TB = F32 ? 3 : 1;     // operand terms
    constexpr uint32_t B_TERM = WIDTH / 2 * 128;          // 64 contraction rows x WIDTH / 2 columns
    constexpr uint32_t A_BYTES = TA * CHUNK_BYTES, STAGE = A_BYTES + TB * B_TERM;
    constexpr int NST = F32 ? 3 : 6;
    constexpr int CHUNK_KB = 2;                           // F32: blocks per accumulator read-out
    constexpr int HW = WIDTH / 2;                         // columns of an epilogue warp
    constexpr int NACC = F32 ? 4 : 2;                     // accumulators in tensor memory
    static_assert(NSOFT * (HW / 32) * (F32 ? 4096 : 6144) <= NST * STAGE, "the last tile is staged in the ring");
    const int pair = blockIdx.x >> 1;
    dep_release();
    // columns of a tile that exist, in whole 128s: a last tile of at most 128 columns runs at half width
    auto tile_width = [&](const GradSide& sd, int n0) { return WIDTH == 256 && sd.cols - n0 <= 128 ? 128 : WIDTH; };

    if (c.warp < NPROD) {
        const bool is_a = c.warp == 0;
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        // (The divisions of the first segment run under the kernel before.  Every role has a walk of its own: one made
        // before the roles part takes the operands of loads and products out of the uniform registers, 4096 x 8192 x
        // 768 5 us a build.)
        SegmentWalk walk(p, pair);
        Segment sg;
        bool more = walk.next(p, sg);
        dep_wait();
        for (; ok && more; more = walk.next(p, sg)) {
            const GradSide& sd = p.side[sg.side];
            const int m0 = sg.tile_m * 256 + (int)c.rank * 128;
            const int n0t = sg.tile_n * WIDTH;
            const int bw = tile_width(sd, n0t) / 2;       // columns this CTA loads
            const int n0 = n0t + (int)c.rank * bw;
            const uint32_t bytes = is_a ? A_BYTES : (uint32_t)TB * bw * 128u;
            for (int k = 0; k < sg.n; ++k) {
                ok = mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag);
                if (!ok) break;
                const uint32_t full = smem_u32(&bars.full[stage]);
                const uint32_t full_leader = mapa_u32(full, 0);
                const uint32_t dst = c.smem + stage * STAGE + (is_a ? 0u : A_BYTES);
                const int k0 = (sg.kb + k) * KB;
                if (elect_one()) {
                    if (c.rank == 0) mbar_expect_tx(full, 2 * bytes);
                    if (is_a) {
#pragma unroll
                        for (int term = 0; term < TA; ++term) {
                            const uint32_t d0 = dst + term * CHUNK_BYTES;
                            if (sg.side == 0) {           // rows of W: K-major
                                tma_load_3d_pair(d0, &mapWk, k0, m0, term, full_leader);
                            } else {                      // columns of W: MN-major, two atoms
                                tma_load_3d_pair(d0, &mapWm, m0, k0, term, full_leader);
                                tma_load_3d_pair(d0 + HALF_CHUNK, &mapWm, m0 + 64, k0, term, full_leader);
                            }
                        }
                    } else {
                        const CUtensorMap* map = sg.side == 0 ? &mapP : &mapQ;
#pragma unroll
                        for (int term = 0; term < TB; ++term) {
                            tma_load_3d_pair(dst + term * B_TERM, map, n0, k0, term, full_leader);
                            if (WIDTH == 256 && bw == 128)
                                tma_load_3d_pair(dst + HALF_CHUNK, map, n0 + 64, k0, term, full_leader);
                        }
                    }
                }
                if (++stage == NST) { stage = 0; phase ^= 1u; }
            }
        }
        if (ok && is_a) ring_drained(bars, NST, stage, phase, abort_flag);
    } else if (c.warp == MMA_WARP) {
        if (c.rank == 0) {
            int stage = 0, use = 0;
            uint32_t phase = 0;
            bool ok = true;
            SegmentWalk walk(p, pair);
            Segment sg;
            while (ok && walk.next(p, sg)) {
                const GradSide& sd = p.side[sg.side];
                const int width = tile_width(sd, sg.tile_n * WIDTH);
                const uint32_t idesc = instr_desc(width, true, 256, sg.side == 1);
                const uint32_t a_lbo = sg.side ? HALF_CHUNK : 0, a_step = sg.side ? 128 : 2;
                uint32_t acc = 0;
                for (int k = 0; k < sg.n; ++k) {
                    const bool fresh = F32 ? k % CHUNK_KB == 0 : k == 0;
                    if (fresh) {
                        ok = wait_acc_free<NACC>(bars, use, abort_flag);
                        if (!ok) break;
                        tc_fence_after();
                        acc = c.tmem + (use % NACC) * (TMEM_COLS / NACC);
                    }
                    ok = mbar_wait(smem_u32(&bars.full[stage]), phase, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = desc_lo(c.smem + stage * STAGE, a_lbo);
                    const uint32_t b = desc_lo(c.smem + stage * STAGE + A_BYTES, HALF_CHUNK);
                    const bool last = F32 ? (k % CHUNK_KB == CHUNK_KB - 1 || k == sg.n - 1) : k == sg.n - 1;
                    if (elect_one()) {
                        if (fresh) mma_ss<false, true>(acc, a, b, idesc);
                        else       mma_ss<true, true>(acc, a, b, idesc);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk) {
                            const uint32_t ak = a + kk * a_step, bk = b + kk * 128;
                            if (kk) mma_ss<true, true>(acc, ak, bk, idesc);
                            if (F32) {
                                constexpr uint32_t A2 = CHUNK_BYTES >> 4, B1 = B_TERM >> 4;
                                mma_ss<true, true>(acc, ak, bk + B1, idesc);
                                mma_ss<true, true>(acc, ak, bk + 2 * B1, idesc);
                                mma_ss<true, true>(acc, ak + A2, bk, idesc);
                                mma_ss<true, true>(acc, ak + A2, bk + B1, idesc);
                            }
                        }
                        tc_commit_pair(smem_u32(&bars.empty[stage]));
                        if (last) tc_commit_pair(smem_u32(&bars.acc_full[use % NACC]));
                    }
                    if (last) ++use;
                    if (++stage == NST) { stage = 0; phase ^= 1u; }
                }
            }
        } else {
            int uses = 0;
            SegmentWalk walk(p, pair);
            Segment sg;
            while (walk.next(p, sg)) uses += F32 ? (sg.n + CHUNK_KB - 1) / CHUNK_KB : 1;
            forward_acc_free<NACC>(bars, uses, abort_flag);
        }
    } else {
        const int ew = c.warp - (NPROD + 1);
        const int q = c.warp & 3, half = ew >> 2, lane = c.lane;
        constexpr int SB = F32 || WIDTH == 256 ? 1 : 2;   // staging buffers of 4 KB
        const uint32_t stage_buf = c.smem + NST * STAGE + (uint32_t)ew * (SB * 4096u);
        const int cw = (int)c.rank * 8 + ew;              // this warp among the 16 of a tile
        constexpr size_t PART_FLOATS = 32 * HW;
        int use = 0, nstore = 0;
        bool ok = true;
        SegmentWalk walk(p, pair);
        Segment sg, nx;
        bool more = walk.next(p, nx);
        dep_wait();
        if (p.whole < 0 && ew == 0 && c.rank == 0 && lane == 0) atomicAdd(p.started, 1);
        if (p.terms && blockIdx.x == 0) {
            // the loss: a fixed order of sums, under the first products
            __shared__ float sums[NSOFT];
            float v = 0.f;
#pragma unroll 4
            for (int e = ew * 32 + lane; e < p.n_terms; e += 32 * NSOFT) v += __ldcg(p.terms + e);
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) sums[ew] = v;
            asm volatile("bar.sync 1, %0;" ::"n"(32 * NSOFT) : "memory");
            if (ew == 0 && lane == 0) {
                v = 0.f;
                for (int w = 0; w < NSOFT; ++w) v += sums[w];
                *p.loss = v * p.inv_mean;
            }
        }
        for (bool any = more; ok && any; any = more) {
            sg = nx;
            more = walk.next(p, nx);                      // false: sg is the pair's last
            const GradSide& sd = p.side[sg.side];
            const int row0 = sg.tile_m * 256 + (int)c.rank * 128 + 32 * q;
            const int n0 = sg.tile_n * WIDTH;
            const int hw = tile_width(sd, n0) / 2;        // columns of this warp
            const int col0 = n0 + half * hw;
            const bool whole = sg.n == sd.kblocks;
            const uint32_t lanes = (uint32_t)(32 * q) << 16;
            // What the positives' weights lost is r_i times the positive's passage.  A lane reads 8 columns of row
            // 8 k + lane / 4 of those (a lane per row, 32 cache lines to a load, held up a tile's epilogue by
            // 7 K cycles), two blocks ahead of their use and the first two before the products are waited for.
            float r_i = 0.f;
            int pos_i = -1;
            if (!F32 && sg.side == 0 && p.res && row0 + lane < sd.rows) {
                r_i = p.res[row0 + lane];
                if (r_i != 0.f) pos_i = p.pos_idx[row0 + lane];
            }
            const bool fix = !F32 && __any_sync(0xffffffffu, pos_i >= 0);
            uint4 px[F32 ? 1 : 8];
            auto fetch_p = [&](int cb) {
                if (F32 || !fix) return;
                const int col = col0 + 32 * cb + 8 * (lane & 3);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int pos = __shfl_sync(0xffffffffu, pos_i, 8 * k + (lane >> 2));
                    px[F32 ? 0 : 4 * (cb & 1) + k] = pos >= 0 && col < sd.cols
                        ? *reinterpret_cast<const uint4*>(p.P + (int64_t)pos * p.ldp + col) : make_uint4(0, 0, 0, 0);
                }
            };
            // first and last group with a share of this tile, and the tile's counter
            const int group = walk.group, tn = sd.tiles_n;
            int gf = group, gl = group;
            int* counter = p.count + ((sg.side ? p.side[0].tiles : 0) + sg.tile_m * tn + sg.tile_n) * 16 + cw;
            if (!whole) {
                const int t1 = sg.t0 + sd.kblocks;
                while (unit_start(p, gf) > sg.t0) --gf;
                while (unit_start(p, gl + 1) < t1) ++gl;
            } else {
                fetch_p(0);
                fetch_p(1);                               // (a tile has at least two blocks of 32 columns per warp)
            }
            float acc[F32 ? HW : 1];
            if (F32) {
                const int chunks = (sg.n + CHUNK_KB - 1) / CHUNK_KB;
#pragma unroll
                for (int e = 0; e < (F32 ? HW : 1); ++e) acc[e] = -0.f;       // adds nothing, not even a sign
#pragma unroll 1
                for (int ch = 0; ch < chunks && ok; ++ch, ++use) {
                    ok = mbar_wait(smem_u32(&bars.acc_full[use % NACC]), (uint32_t)(use / NACC) & 1u, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t src = c.tmem + (use % NACC) * (TMEM_COLS / NACC) + lanes + half * HW;
#pragma unroll
                    for (int g = 0; g < HW / 32; ++g) {
                        uint32_t v[32];
                        tmem_ld32(src + 32 * g, v);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 32; ++e) {
                            const float x = __uint_as_float(v[e]);
                            acc[32 * g + e] += x;
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bars.acc_free[use % NACC]));
                }
                if (!ok) break;
            } else {
                ok = mbar_wait(smem_u32(&bars.acc_full[use % NACC]), (uint32_t)(use / NACC) & 1u, abort_flag);
                if (!ok) break;
                tc_fence_after();
            }
            const uint32_t src = c.tmem + (use % NACC) * (TMEM_COLS / NACC) + lanes + half * hw;
            auto own_block = [&](int cb, uint32_t (&v)[32]) {
                if (F32) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(acc[F32 ? 32 * cb + e : 0]);
                } else {
                    tmem_ld32(src + 32 * cb, v);
                    tmem_ld_wait();
                }
            };
            auto release_acc = [&]() {
                if (F32) return;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.acc_free[use % NACC]));
            };
            // The passages from there to lane = row, through 2 KB of shared memory: 64 bytes to a row, 16-byte chunks
            // swizzled against conflicts.
            auto spread_p = [&](uint32_t box, int cb) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int r = 8 * k + (lane >> 2);
                    const uint4 x = px[F32 ? 0 : 4 * (cb & 1) + k];
                    sts_v4(box + r * 64 + (((lane & 3) ^ (r >> 1 & 3)) << 4), x.x, x.y, x.z, x.w);
                }
            };
            auto add_p = [&](uint32_t box, uint32_t (&v)[32]) {
                if (pos_i < 0) return;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t w[4];
                    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                                 : "r"(box + lane * 64 + ((j ^ (lane >> 1 & 3)) << 4)) : "memory");
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        v[8 * j + 2 * e] = __float_as_uint(fmaf(
                            r_i, __uint_as_float(w[e] << 16), __uint_as_float(v[8 * j + 2 * e])));
                        v[8 * j + 2 * e + 1] = __float_as_uint(fmaf(
                            r_i, __uint_as_float(w[e] & 0xffff0000u), __uint_as_float(v[8 * j + 2 * e + 1])));
                    }
                }
            };
            auto store = [&](uint32_t buf, int cb) {     // (an empty group when nothing is stored)
                const int col = col0 + 32 * cb;
                const CUtensorMap* map = sg.side == 0 ? &mapDQ : &mapDP;
                if (row0 >= sd.rows || col >= sd.cols)
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                else if (sd.add) tma_add_3d(map, buf, col, row0, 0);
                else             tma_store_3d(map, buf, col, row0, 0);
            };
            // one block of 32 columns to the output: the positives' remainder, scale, staging, store
            auto finish = [&](uint32_t (&v)[32], int cb) {
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(SB - 1) : "memory");
                __syncwarp();
                const uint32_t buf = stage_buf + (uint32_t)(nstore & (SB - 1)) * 4096u;
                ++nstore;
                if (!F32 && fix) {
                    spread_p(buf, cb);
                    __syncwarp();
                    add_p(buf, v);
                    __syncwarp();
                }
                stage_block(buf, v, p.scale, lane);
                __syncwarp();
                if (lane == 0) store(buf, cb);
            };
            // group g's share of the tile: slot 0 when its run starts inside the tile, else 1
            auto part_of = [&](int g, int slot) {
                return reinterpret_cast<float4*>(
                    p.part + (((size_t)(g * tn + sg.tile_n) * 2 + slot) * 16 + cw) * PART_FLOATS);
            };
            if (whole && !more) {
                // The pair's last tile: nothing uses the ring any more, so that every block has a buffer of its own there.
                // (4096 x 4096 x 512, both gradients, one tile to a pair: from the last product to the last store 7.8 K
                // cycles for dQ, 6.5 K for dP, as long as 16 MB take into the L2; block after block through one buffer,
                // with a lane per row of the passages, 12 K and 5-7 K.)
                const uint32_t buf = c.smem + (uint32_t)ew * (HW / 32 * 4096u);
                const uint32_t box = c.smem + NSOFT * (HW / 32 * 4096u) + (uint32_t)ew * (HW / 32 * 2048u);
                if (!F32 && fix) {
#pragma unroll
                    for (int cb = 0; cb < HW / 32; ++cb) {
                        if (32 * cb >= hw) break;
                        spread_p(box + cb * 2048u, cb);
                        if (cb + 2 < HW / 32 && 32 * (cb + 2) < hw) fetch_p(cb + 2);
                    }
                    __syncwarp();
                }
#pragma unroll
                for (int cb = 0; cb < HW / 32; ++cb) {
                    if (32 * cb >= hw) break;
                    uint32_t v[32];
                    own_block(cb, v);
                    if (!F32 && fix) add_p(box + cb * 2048u, v);
                    stage_block_unfenced(buf + cb * 4096u, v, p.scale, lane);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    for (int cb = 0; 32 * cb < hw; ++cb) store(buf + cb * 4096u, cb);
            } else if (whole) {
#pragma unroll
                for (int cb = 0; cb < HW / 32; ++cb) {
                    if (32 * cb >= hw) break;
                    uint32_t v[32];
                    own_block(cb, v);
                    if (32 * (cb + 1) >= hw) release_acc();
                    finish(v, cb);
                    if (cb + 2 < HW / 32 && 32 * (cb + 2) < hw) fetch_p(cb + 2);
                }
            } else {
                // Where all other shares (of a few) are in memory already (as a rule: a group meets the front part
                // of its first tile long before the neighbour meets the back part of its last), this
                // share goes into the sum straight from tensor memory, and whoever waits need not.  (Not from the
                // registers of the fp32 sums: the two sums at once do not fit, and with the running one in local memory a
                // read-out took 4 K cycles where its products take 2.6 K: 2048 x 4096 x 768, 239 us a build against 199.)
                bool direct = false;
                int published = 0;
                if (!F32 && gl - gf < 3) {
                    if (lane == 0) {
                        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(published) : "l"(counter) : "memory");
                        if (published == gl - gf) atomicAdd(counter, SUM_TAKEN);
                    }
                    direct = __shfl_sync(0xffffffffu, published, 0) == gl - gf;
                }
                if (direct) {
                    __threadfence();
#pragma unroll
                    for (int cb = 0; cb < HW / 32; ++cb) {
                        if (32 * cb >= hw) break;
                        float s[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) s[e] = -0.f;
                        for (int g = gf; g <= gl; ++g) {
                            if (g == group) {             // (read here: held beside the sums, 300 bytes a thread spilled)
                                uint32_t v[32];
                                own_block(cb, v);
#pragma unroll
                                for (int e = 0; e < 32; ++e) s[e] += __uint_as_float(v[e]);
                                continue;
                            }
                            const float4* o = part_of(g, g == gf ? 1 : 0);
#pragma unroll
                            for (int j0 = 0; j0 < 8; j0 += 4) {
                                float4 x[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) x[j] = __ldcg(o + (cb * 8 + j0 + j) * 32 + lane);
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                    float* t = s + 4 * (j0 + j);
                                    t[0] += x[j].x; t[1] += x[j].y; t[2] += x[j].z; t[3] += x[j].w;
                                }
                            }
                        }
                        uint32_t v[32];
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(s[e]);
                        fetch_p(cb);
                        finish(v, cb);
                    }
                    release_acc();
                } else {
                    float4* mine = part_of(group, sg.kb == 0 ? 1 : 0);
#pragma unroll
                    for (int cb = 0; cb < HW / 32; ++cb) {
                        if (32 * cb >= hw) break;
                        uint32_t v[32];
                        own_block(cb, v);
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            __stcg(mine + (cb * 8 + j) * 32 + lane,
                                   make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                               __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3])));
                    }
                    release_acc();
                    __threadfence();
                    __syncwarp();
                    // A share is in memory: one more in the counter's lower half.  A warp with nothing left to do waits
                    // for the others if they are all at work, so that they sum the tile together (see SUM_WAIT_NS).
                    int complete = 0, published = 0;
                    if (lane == 0) {
                        complete = (atomicAdd(counter, 1) & 0xffff) == gl - gf;
                        if (!complete && !more && *reinterpret_cast<volatile int*>(p.started) == p.all_started) {
                            const uint64_t t0 = global_ns();
                            do {
                                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(published) : "l"(counter) : "memory");
                                complete = (published & 0xffff) == gl - gf + 1;
                            } while (!complete && !(published & SUM_TAKEN) && global_ns() - t0 < SUM_WAIT_NS);
                        }
                    }
                    if (__shfl_sync(0xffffffffu, complete, 0)) {
                        __threadfence();
                        // pieces of 4 NJ columns, drawn from the counter's upper half; PB shares' loads in flight
                        auto sum_pieces = [&](auto nj) {
                            constexpr int NJ = decltype(nj)::value, PB = (F32 ? 8 : 12) / NJ;
                            auto draw = [&]() { return lane == 0 ? atomicAdd(counter, 0x10000) >> 16 : 0; };
                            const int pieces = hw / (4 * NJ);
                            int drawn = draw();
                            for (;;) {
                                const int piece = __shfl_sync(0xffffffffu, drawn, 0);
                                if (piece >= pieces) break;
                                float4 s[NJ];
                                uint2 pw[NJ];            // the positive's passage
#pragma unroll
                                for (int j = 0; j < NJ; ++j) {
                                    const int col = col0 + 4 * (piece * NJ + j);
                                    if (!F32 && pos_i >= 0 && col < sd.cols)
                                        pw[j] = *reinterpret_cast<const uint2*>(p.P + (int64_t)pos_i * p.ldp + col);
                                    s[j] = make_float4(-0.f, -0.f, -0.f, -0.f);
                                }
#pragma unroll 1
                                for (int g0 = gf; g0 <= gl; g0 += PB) {
                                    float4 x[PB][NJ];
#pragma unroll
                                    for (int b = 0; b < PB; ++b) {
                                        const int g = min(g0 + b, gl);
                                        const float4* o = part_of(g, g == gf ? 1 : 0) + piece * NJ * 32 + lane;
#pragma unroll
                                        for (int j = 0; j < NJ; ++j) x[b][j] = __ldcg(o + j * 32);
                                    }
                                    if (g0 == gf) drawn = draw();
#pragma unroll
                                    for (int b = 0; b < PB; ++b) {
                                        if (g0 + b <= gl) {
#pragma unroll
                                            for (int j = 0; j < NJ; ++j) {
                                                s[j].x += x[b][j].x; s[j].y += x[b][j].y;
                                                s[j].z += x[b][j].z; s[j].w += x[b][j].w;
                                            }
                                        }
                                    }
                                }
#pragma unroll
                                for (int j = 0; j < NJ; ++j) {
                                    const int col = col0 + 4 * (piece * NJ + j);
                                    if (row0 + lane >= sd.rows || col >= sd.cols) continue;
                                    if (!F32 && pos_i >= 0) {
                                        s[j].x = fmaf(r_i, __uint_as_float(pw[j].x << 16), s[j].x);
                                        s[j].y = fmaf(r_i, __uint_as_float(pw[j].x & 0xffff0000u), s[j].y);
                                        s[j].z = fmaf(r_i, __uint_as_float(pw[j].y << 16), s[j].z);
                                        s[j].w = fmaf(r_i, __uint_as_float(pw[j].y & 0xffff0000u), s[j].w);
                                    }
                                    float4 r = make_float4(s[j].x * p.scale, s[j].y * p.scale, s[j].z * p.scale, s[j].w * p.scale);
                                    float4* dst = reinterpret_cast<float4*>(
                                        p.out[sg.side] + (int64_t)(row0 + lane) * p.ldo[sg.side] + col);
                                    if (sd.add) {         // rounds as bulk reductions do: neither flushes subnormals
                                        const float4 o = *dst;
                                        r = make_float4(__fadd_rn(o.x, r.x), __fadd_rn(o.y, r.y), __fadd_rn(o.z, r.z),
                                                        __fadd_rn(o.w, r.w));
                                    }
                                    *dst = r;
                                }
                            }
                        };
                        if (gl - gf < 7) sum_pieces(std::integral_constant<int, 4>{});
                        else             sum_pieces(std::integral_constant<int, 2>{});
                    }
                }
            }
            if (!F32) ++use;
        }
        if (lane == 0) bulk_wait_all();
        __syncwarp();
    }
    pair_teardown(c, abort_flag, p.dev_status);
}

// ---------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------
// A row-major matrix of 16-bit or fp32 values as [planes][rows][cols]; boxes of 128 bytes x box_rows,
// 128-byte swizzle, out-of-range elements read as zero and are not written.
bool map3(CUtensorMap* map, bool f32, const void* base, int64_t rows, int64_t cols, int64_t pitch,
          int64_t planes, int64_t plane_pitch, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t es = f32 ? 4 : 2;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)planes};
    cuuint64_t strides[2] = {(cuuint64_t)pitch * es, (cuuint64_t)plane_pitch * es};
    cuuint32_t box[3] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
              const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }
int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }
int pairs_of_device() { return sm_count() / 2; }

constexpr size_t SMEM_L256 = 1024 + 6 * (CHUNK_BYTES + 16384) + NSOFT * 4096;    // or 5 stages, NSOFT * 8192
constexpr size_t SMEM_L128 = 1024 + 6 * (CHUNK_BYTES + 8192) + NSOFT * 4096;
constexpr size_t SMEM_LF32 = 1024 + F_NST * F_STAGE + NSOFT * 8192;
constexpr size_t SMEM_G = 1024 + 6 * (CHUNK_BYTES + 16384) + NSOFT * 4096;
constexpr size_t SMEM_G128 = 1024 + 6 * (CHUNK_BYTES + 8192) + NSOFT * 8192;
constexpr size_t SMEM_GF32 = 1024 + 3 * (2 * CHUNK_BYTES + 3 * 8192) + NSOFT * 4096;
static_assert(SMEM_L256 <= SMEM_LIMIT - 1024 && SMEM_LF32 <= SMEM_LIMIT - 1024 &&
              SMEM_GF32 <= SMEM_LIMIT - 1024, "shared memory budget");

// The shared-memory limit belongs to the (kernel, device) pair; set once for all kernels here.
cudaError_t configure_kernels() {
    static bool done[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (done[dev]) return cudaSuccess;
    const struct { const void* f; size_t bytes; } all[] = {
        {(const void*)strip_logit_kernel<LOGIT_FWD, 256>, SMEM_L256},
        {(const void*)strip_logit_kernel<LOGIT_FWD, 128>, SMEM_L128},
        {(const void*)strip_logit_kernel<LOGIT_STASH, 256>, SMEM_L256},
        {(const void*)strip_logit_kernel<LOGIT_STASH, 128>, SMEM_L128},
        {(const void*)strip_logit_kernel<LOGIT_W, 256>, SMEM_L256},
        {(const void*)strip_logit_kernel<LOGIT_W, 128>, SMEM_L128},
        {(const void*)strip_logit_kernel<LOGIT_W2, 256>, SMEM_L256},
        {(const void*)strip_logit_kernel<LOGIT_W2, 128>, SMEM_L128},
        {(const void*)strip_logit_f32_kernel, SMEM_LF32},
        {(const void*)strip_grad_kernel<false, 256>, SMEM_G},
        {(const void*)strip_grad_kernel<false, 128>, SMEM_G128},
        {(const void*)strip_grad_kernel<true, 128>, SMEM_GF32},
    };
    for (const auto& k : all) {
        const cudaError_t e = cudaFuncSetAttribute(k.f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)k.bytes);
        if (e != cudaSuccess) return e;
    }
    done[dev] = true;
    return cudaSuccess;
}

// How the gradient tiles of a strip are dealt out (see GradParams): the cheapest by a count of cycles.
struct GradDeal { int width, whole, pairs; };
GradDeal deal_grads(int64_t rows, int64_t N, int d, bool f32, bool dq, bool dp) {
    const int pairs = pairs_of_device();
    GradDeal best{};
    double best_cost = 0;
    for (int width = f32 ? 128 : 256; width >= 128; width -= 128) {
        const int tn = (int)ceil_div(d, width);
        // Cycles per contraction block; what cutting tiles costs by itself; and per part of a tile, whose
        // sums are added up one after the other.  Fitted to 443 bf16 shapes (20 to 24000 queries, 64 to 2048 columns,
        // one gradient or both) and 129 fp32 shapes (34 to 4096 queries, 64 to 768 columns), with 4 to 25 choices
        // forced at each.  How much slower the choice this makes is than the best, on average / at worst: ordinary bf16
        // shapes 0.3 / 6 %, those beyond 4096 x 8192 x 768 0.9 / 14 %, one rank's share of a batch 0.8 / 10 %, one side of
        // at most 260 rows 3 / 31 %, fp32 0.3 / 6 %.  (us, tiles cut / whole: both gradients of 2952 x 2214 x 512 47.6 /
        // 35.6, of 4160 x 4160 x 768 87.9 / 77.8, of 12525 x 37575 x 1024 1980 / 2500; dQ of 2048 x 16384 x 768 90 / 109,
        // of 779 x 3118 x 384 23.8 / 27.2; fp32, 1024 x 2048 x 768 62.0 / 54.9)
        const bool both = dq && dp;
        const double unit = f32 ? 1400 : width == 256 ? 560 : 400;
        const double cut = f32 ? (both ? 14500 : 8500) : width == 256 ? 19000 : both ? 15500 : 11000;
        const double part = f32 ? 450 : width == 256 ? 2500 : 160;
        // A block of a cut run takes 5 % more, on average over 92 shapes beyond 4096 x 8192 x 768 in short runs and 55 under
        // the power cap (both gradients, cut / whole: 6532 x 19596 x 640 413 / 394 us with 4 % more blocks on the longest
        // pair of whole tiles; under the power cap 20969 x 62907 x 640 5043 / 4879 with 17 % more.  Not everywhere:
        // 20450 x 20450 x 896 1695 / 1952 with 9 % more).  fp32: none seen.
        const double along = f32 ? 0 : 0.05;
        // A pair's next tile takes at least the epilogue of this one (dQ's adds what the positives' weights lost):
        // tiles of few contraction blocks are bound by it.  4671 x 30 x 128, both gradients: 18 dQ tiles of one
        // block to a pair 71 us, 19 pairs for them 14; 7 x 9470 x 128: 26 dP tiles of one block to a pair 44 us.
        const double epi_q = width == 256 ? 12000 : 6000, epi_p = width == 256 ? 11000 : 3200;
        const int64_t kq = ceil_div(N, KB), kp = ceil_div(rows, KB);
        const int64_t tq = dq ? ceil_div(rows, 256) * tn : 0, tp = dp ? ceil_div(N, 256) * tn : 0;
        auto offer = [&](double cost, int whole, int used) {
            if (best.pairs == 0 || cost < best_cost) { best = {width, whole, used}; best_cost = cost; }
        };
        auto tiles_cost = [&](int64_t n, int64_t k, double epilogue) {
            return (double)(n - 1) * (k * unit > epilogue ? k * unit : epilogue) + k * unit;
        };
        // whole tiles, every split of the pairs between the two products
        if (tq + tp <= pairs) {
            offer((double)(tq && kq > kp ? kq : tp ? (tq && kq > kp ? kq : kp) : kq) * unit, tq ? (int)tq : 0, (int)(tq + tp));
        } else {
            for (int w = tq ? 1 : 0; w <= (tp ? pairs - 1 : pairs); ++w) {
                if (!tq && w) break;
                const double a = tq ? tiles_cost(ceil_div(tq, w), kq, epi_q) : 0;
                const double b = tp ? tiles_cost(ceil_div(tp, pairs - w), kp, epi_p) : 0;
                offer(a > b ? a : b, w, pairs);
            }
        }
        // equal runs of contraction blocks, at least four to a pair: as many as cost least
        if (tn > pairs) continue;
        const double units = (double)((tq * kq + tp * kp) / tn), longest = (double)(tq && (kq > kp || !tp) ? kq : kp);
        int groups = (int)(units * sqrt(unit / (part * longest)));
        if (groups > pairs / tn) groups = pairs / tn;
        if (groups > units / 4) groups = (int)(units / 4);
        if (groups < 1) groups = 1;
        const double run = units / groups;
        double cost = run * unit;
        if (tq && run > kq && run / kq * epi_q > cost) cost = run / kq * epi_q;
        if (tp && run > kp && run / kp * epi_p > cost) cost = run / kp * epi_p;
        offer(cost + cut + along * run * unit + part * longest * groups / units, -1, groups * tn);
    }
    return best;
}

// Columns of a logit tile: 128 while there are at most one and a half 256-wide tiles to a CTA pair (more
// pairs busy, or a shorter last wave, and epilogues that overlap products).  us per build of d = 768 with
// 256 / 128: 500 x 1000 22.9 / 20.5, 1531 x 3062 35.1 / 33.7 (72 tiles, 74 pairs), 1300 x 3900 43.6 / 40.6 (96),
// 1700 x 3400 46.3 / 44.1 (98); from there on nothing or a loss: 1800 x 3600 49.8 / 49.7 (120), 2048 x 4096
// 51.5 / 51.6 (128), 3000 x 6000 78.9 / 81.7 (288).  d = 256 and 512, and the loss alone: the same sides.
int logit_width(int64_t rows, int64_t N) {
    return 2 * ceil_div(rows, 256) * ceil_div(N, 256) <= 3 * (int64_t)pairs_of_device() ? 128 : 256;
}

struct StripLayout {
    int64_t rows;                 // of a strip (the last may be shorter)
    int strips;
    int64_t ldw;
    int slot_pitch;
    size_t zero, slots, pos, res, red, w, part, s, tq, tp, total;
};

StripLayout strip_layout(int64_t B, int64_t N, int d, int dtype, bool fwd_only = false) {
    StripLayout l{};
    const bool f32 = dtype == GC_F32;
    // Few strips: each costs a read and a write of dP and the fill and drain of three kernels.  Whether
    // a strip's weights stay in the L2 matters less (8192 x 16384 x 768: 586 us in one strip of 268 MB,
    // 666 in four of 67 MB).  bf16: 768 M pairs, 1.5 GB of weights (ms in strips of 0.5 GB, or 1 GB beyond
    // 65536 passages, and of 1.5-2 GB: 16384 x 32768 x 768 2.38 / 2.33, 40000 x 80000 x 512 11.1 / 10.7,
    // 65536 x 131072 x 768 38.3 / 37.0, loss and gradients of 40000 x 120000 x 256 11.5 / 11.0; 4 GB would
    // give 10.5, 37.8 and 10.5); fp32 holds 8 bytes a pair and does four times the arithmetic: 64 M pairs.
    l.ldw = ceil_div(N, 64) * 64;
    int64_t r = ((int64_t)(f32 ? 64 : 768) << 20) / l.ldw / 256 * 256;
    if (r < 256) r = 256;
    const int64_t n = ceil_div(B, r);
    r = ceil_div(ceil_div(B, n), 256) * 256;
    l.strips = (int)ceil_div(B, r);
    l.rows = B < r ? B : r;
    l.slot_pitch = (int)(ceil_div(N, 256) * 4);
    const int64_t tiles = ceil_div(l.rows, 256) * ceil_div(d, 128) + ceil_div(N, 256) * ceil_div(d, 128);
    size_t off = 0;
    const size_t counters = fwd_only ? 0 : (size_t)tiles * 16;
    l.zero = off;  off += up256(sizeof(int) * (64 + counters));     // word 0: ticket of the loss, 32: pairs started
    l.pos = off;   off += up256(sizeof(float) * (size_t)l.rows);
    l.red = off;   off += up256(sizeof(float) * (size_t)(B + 8 * sm_count()));
    if (!f32) {
        const int64_t pitch = fwd_only ? 2 * ceil_div(N, 128) : l.slot_pitch;
        l.slots = off;  off += up256(sizeof(float2) * (size_t)l.rows * (size_t)pitch);
    } else {
        const size_t dp = (size_t)((d + 7) / 8 * 8);
        l.s = off;   off += up256(4 * (size_t)l.rows * (size_t)l.ldw);
        l.tq = off;  off += up256(6 * (size_t)B * dp);
        l.tp = off;  off += up256(6 * (size_t)N * dp);
    }
    if (!fwd_only) {
        l.res = off;   off += up256(sizeof(float) * (size_t)l.rows);
        l.w = off;     off += up256((f32 ? 4 : 2) * (size_t)l.rows * (size_t)l.ldw);
        l.part = off;  off += (size_t)pairs_of_device() * 2 * 16 * 32 * (f32 ? 64 : 128) * 4;
    }
    l.total = off;
    return l;
}

struct StripRun {
    const Problem& p;
    StripLayout l;
    char* ws;
    cudaStream_t st;
    int* dev_status;
    bool f32, shared;
    const float* col_neg = nullptr;
    const TwoDirection* two = nullptr;
    float grad_scale = 1.f;
    int started = 0;              // CTA pairs of the gradient launches with cut runs so far

    StripRun(const Problem& pr, void* w, int* status, cudaStream_t s, bool fwd_only = false)
        : p(pr), l(strip_layout(pr.B, pr.N, pr.d, pr.dtype, fwd_only)), ws(static_cast<char*>(w)), st(s),
          dev_status(status), f32(pr.dtype == GC_F32),
          shared(pr.Q == pr.P && pr.ldq == pr.ldp && pr.B == pr.N) {}

    template <typename T> T* at(size_t off) { return reinterpret_cast<T*>(ws + off); }
    int64_t rows_of(int s) const { return s == l.strips - 1 ? p.B - (int64_t)s * l.rows : l.rows; }
    float c1() const { return LOG2E / p.tau; }
    int shift(int s) const { return (int)(p.mask_shift + (int64_t)s * l.rows); }
    void* terms_p() { return ws + (shared ? l.tq : l.tp); }

    // planes of 16-bit rows: the inputs themselves, or the terms of fp32 inputs
    bool rows_map(CUtensorMap* m, bool q, int64_t first, int64_t count, int box) {
        if (!f32) {
            const char* base = static_cast<const char*>(q ? p.Q : p.P);
            const int64_t ld = q ? p.ldq : p.ldp;
            return map3(m, false, base + first * ld * 2, count, p.d, ld, 1, count * ld, box);
        }
        const int64_t all = q ? p.B : p.N;
        const char* base = static_cast<const char*>(q ? (void*)(ws + l.tq) : terms_p());
        return map3(m, false, base + first * p.d * 2, count, p.d, p.d, 3, all * p.d, box);
    }

    cudaError_t split() {
        const int64_t items = (p.B + (shared ? 0 : p.N)) * (p.d / 4);
        int64_t blocks = ceil_div(items, 256);
        if (blocks > 8 * sm_count()) blocks = 8 * sm_count();
        return launch_chained(split_terms_kernel, (unsigned)blocks, 256, 0, 1, st,
                      static_cast<const float*>(p.Q), p.ldq, p.B, at<uint2>(l.tq),
                      static_cast<const float*>(p.P), p.ldp, shared ? (int64_t)0 : p.N, at<uint2>(l.tp),
                      p.d / 4);
    }

    cudaError_t logits(int s, int mode, const float* row_lse, bool zero_ticket) {
        const int64_t row0 = (int64_t)s * l.rows, rows = rows_of(s);
        const int pairs = pairs_of_device();
        const int tiles_m = (int)ceil_div(rows, 256);
        const int bn = f32 ? 128 : logit_width(rows, p.N);
        LogitParams lp{};
        lp.rows = (int)rows; lp.N = (int)p.N;
        lp.kblocks = (int)ceil_div(p.d, KB);
        lp.tiles_m = tiles_m;
        lp.tiles_n = (int)ceil_div(p.N, bn);
        lp.c1 = c1(); lp.inv_tau = 1.f / p.tau;
        lp.mask_on = p.mask_mode == GC_MASK_SELF; lp.mask_shift = shift(s);
        lp.pos_idx = p.pos_idx ? p.pos_idx + row0 : nullptr;
        lp.pos_base = (int)p.pos_base; lp.pos_n = (int)(p.n_total > 0 ? p.n_total : p.N);
        lp.col_neg = col_neg;
        if (two) {
            lp.col_lse = two->col_lse; lp.pos_logit = two->pos_logit;
            lp.terms = mode == LOGIT_W2 ? at<float>(l.red) + row0 : nullptr;
            if (mode == LOGIT_FWD && zero_ticket && !two->columns) { lp.zero2 = two->mult; lp.zero2_count = (int)p.N; }
            if (mode == LOGIT_W2) lp.pos_logit += row0;
            lp.zero_anchor_lse = logf((float)p.B);
        }
        lp.row_lse = row_lse ? row_lse + row0 : nullptr;
        lp.slots = at<float2>(l.slots);
        lp.slot_pitch = mode == LOGIT_FWD ? 2 * lp.tiles_n : l.slot_pitch;
        lp.pos_ws = at<float>(l.pos);
        lp.res = at<float>(l.res);
        const int skip = zero_ticket ? 0 : 64;
        lp.zero = at<int>(l.zero) + skip;
        lp.zero_count = (int)((l.pos - l.zero) / sizeof(int)) - skip;
        lp.dev_status = dev_status;
        CUtensorMap mq, mp, mw;
        if (!rows_map(&mq, true, row0, rows, 128) || !rows_map(&mp, false, 0, p.N, bn / 2)) return cudaErrorInvalidValue;
        if (!(f32 ? map3(&mw, true, ws + l.s, rows, p.N, l.ldw, 1, rows * l.ldw, 32)
                  : map3(&mw, false, ws + l.w, rows, p.N, l.ldw, 1, rows * l.ldw, 32)))
            return cudaErrorInvalidValue;
        const int total = lp.tiles_m * lp.tiles_n;
        const unsigned grid = 2u * (unsigned)(total < pairs ? total : pairs);
        if (f32) return launch_chained(strip_logit_f32_kernel, grid, ST_THREADS, SMEM_LF32, 2, st, mq, mp, mw, lp);
        auto go = [&](auto k256, auto k128) {
            return bn == 256 ? launch_chained(k256, grid, ST_THREADS, SMEM_L256, 2, st, mq, mp, mw, lp)
                             : launch_chained(k128, grid, ST_THREADS, SMEM_L128, 2, st, mq, mp, mw, lp);
        };
        if (mode == LOGIT_FWD) return go(strip_logit_kernel<LOGIT_FWD, 256>, strip_logit_kernel<LOGIT_FWD, 128>);
        if (mode == LOGIT_STASH) return go(strip_logit_kernel<LOGIT_STASH, 256>, strip_logit_kernel<LOGIT_STASH, 128>);
        if (mode == LOGIT_W2) return go(strip_logit_kernel<LOGIT_W2, 256>, strip_logit_kernel<LOGIT_W2, 128>);
        return go(strip_logit_kernel<LOGIT_W, 256>, strip_logit_kernel<LOGIT_W, 128>);
    }

    // fp32: a warp to a row of logits
    bool short_rows() const { return p.N <= 512; }
    // the loss alone: a thread to a row
    int forward_slots(int s) const { return (int)(2 * ceil_div(p.N, logit_width(rows_of(s), p.N))); }
    bool row_threads(int s) const { return forward_slots(s) <= MOST_THREAD_SLOTS && rows_of(s) >= 8192; }
    int row_blocks(int s, bool write) const {
        if (!f32) return (int)ceil_div(rows_of(s), write ? row_warps(true) : row_threads(s) ? 256 : row_warps(false));
        if (short_rows()) return (int)std::min<int64_t>(ceil_div(rows_of(s), 8), 8 * (int64_t)sm_count());
        const int64_t n = rows_of(s), most = 8 * (int64_t)sm_count();
        return (int)(n < most ? n : most);
    }

    cudaError_t rows_kernel(int s, bool write, bool lse_given, float* row_lse, float* pos_logit,
                            float* loss) {
        const int64_t row0 = (int64_t)s * l.rows, rows = rows_of(s);
        RowParams rp{};
        rp.rows = (int)rows; rp.N = (int)p.N; rp.row0 = (int)row0;
        rp.c1 = c1(); rp.inv_tau = 1.f / p.tau;
        rp.mask_on = p.mask_mode == GC_MASK_SELF; rp.mask_shift = shift(s);
        rp.pos_idx = p.pos_idx ? p.pos_idx + row0 : nullptr;
        rp.pos_base = (int)p.pos_base; rp.pos_n = (int)(p.n_total > 0 ? p.n_total : p.N);
        rp.slots = at<float2>(l.slots);
        if (write) {
            rp.slot_pitch = l.slot_pitch;
            rp.nslots = (int)ceil_div(p.N, 64);
        } else {
            rp.nslots = rp.slot_pitch = forward_slots(s);
        }
        rp.pos_ws = at<float>(l.pos);
        rp.res = at<float>(l.res);
        rp.row_lse = row_lse + row0;
        rp.pos_logit = pos_logit ? pos_logit + row0 : nullptr;
        rp.loss = loss;
        rp.red = at<float>(l.red);
        rp.ticket = at<int>(l.zero);
        rp.block0 = 0;
        for (int k = 0; k < s; ++k) rp.block0 += row_blocks(k, write);
        rp.blocks_total = 0;
        for (int k = 0; k < l.strips; ++k) rp.blocks_total += row_blocks(k, write);
        rp.inv_mean = 1.f / (float)(p.b_total > 0 ? p.b_total : p.B);
        rp.ldw = l.ldw;
        rp.dev_status = dev_status;
        rp.S = f32 ? at<float>(l.s) : nullptr;
        rp.lds = l.ldw;
        rp.lse_given = lse_given; rp.want_w = write;
        if (two && !write) {
            if (two->columns) { rp.mult = two->mult + row0; rp.col_neg = two->col_neg + row0; }
            else              rp.count = two->mult;
        }
        const unsigned grid = (unsigned)row_blocks(s, write);
        if (f32)
            return short_rows() ? launch_chained(strip_row_f32_kernel<false>, grid, 256, 0, 1, st, at<uint2>(l.w), rp)
                                : launch_chained(strip_row_f32_kernel<true>, grid, 256, 0, 1, st, at<uint2>(l.w), rp);
        if (!write && row_threads(s)) return launch_chained(strip_lse_kernel, grid, 256, 0, 1, st, rp);
        const int64_t rounds = ceil_div(p.N, 8 * ROW_ROUND);
        // four warps to a row from three rounds on; a second segment where they would have more than two
        // rounds each (6144 x 24000: 132 us with it, 134 without; 4096 x 131072: 472 and 481), more
        // while there are few rows (512 x 32768: 11.7 with two, 17.8 with one)
        rp.split = !write ? 0 : rounds >= 3 ? 2 : rounds == 2 ? 1 : 0;
        const int64_t each = ceil_div(rounds, 1 << rp.split), room = 8 * (int64_t)sm_count() / rows;
        const int64_t least = each > 2 ? 2 : 1, segs = room > least ? (room < each ? room : each) : least;
        rp.seg_rounds = (int)ceil_div(each, segs) << rp.split;
        auto go = [&](auto k, dim3 g) { return launch_chained(k, g, 32 * row_warps(write), 0, 1, st, at<uint4>(l.w), rp); };
        if (!write) return go(strip_row_kernel<false, 1>, dim3(grid));
        const dim3 g((unsigned)ceil_div(rows, row_warps(true) >> rp.split), (unsigned)ceil_div(rounds, rp.seg_rounds));
        return (int64_t)g.x * g.y <= 6 * sm_count() ? go(strip_row_kernel<true, 6>, g)
                                                    : go(strip_row_kernel<true, 7>, g);
    }

    cudaError_t grads(int s, float* dQ, int64_t lddq, float* dP, int64_t lddp, float* loss) {
        const int64_t row0 = (int64_t)s * l.rows, rows = rows_of(s);
        const int planes = f32 ? 2 : 1;
        const GradDeal deal = deal_grads(rows, p.N, p.d, f32, dQ != nullptr, dP != nullptr);
        const int width = deal.width, tn = (int)ceil_div(p.d, width);
        GradParams gp{};
        gp.side[0] = {dQ ? (int)ceil_div(rows, 256) * tn : 0, tn, (int)ceil_div(p.N, KB), (int)rows, p.d, 0};
        gp.side[1] = {dP ? (int)ceil_div(p.N, 256) * tn : 0, tn, (int)ceil_div(rows, KB), (int)p.N, p.d, s > 0};
        gp.whole = deal.whole;
        gp.pairs = deal.pairs;
        gp.groups = deal.pairs / tn;
        gp.units = (gp.side[0].tiles * gp.side[0].kblocks + gp.side[1].tiles * gp.side[1].kblocks) / tn;
        gp.scale = grad_scale / ((float)(p.b_total > 0 ? p.b_total : p.B) * p.tau);
        gp.res = f32 ? nullptr : at<float>(l.res);
        gp.pos_idx = p.pos_idx + row0;
        gp.P = f32 ? nullptr : static_cast<const __nv_bfloat16*>(p.P);
        gp.ldp = p.ldp;
        if (loss && s == l.strips - 1) {
            gp.terms = at<float>(l.red);
            gp.n_terms = (int)p.B;
            gp.loss = loss;
            gp.inv_mean = 1.f / (float)(p.b_total > 0 ? p.b_total : p.B);
        }
        gp.out[0] = dQ ? dQ + row0 * lddq : nullptr; gp.ldo[0] = lddq;
        gp.out[1] = dP; gp.ldo[1] = lddp;
        gp.part = at<float>(l.part);
        gp.count = at<int>(l.zero) + 64;
        if (gp.whole < 0) started += gp.pairs;
        gp.started = at<int>(l.zero) + 32;
        gp.all_started = started;
        gp.dev_status = dev_status;
        CUtensorMap wk, wm, mp, mq, mdq, mdp;
        if (!map3(&wk, false, ws + l.w, rows, p.N, l.ldw, planes, rows * l.ldw, 128) ||
            !map3(&wm, false, ws + l.w, rows, p.N, l.ldw, planes, rows * l.ldw, 64) ||
            !rows_map(&mp, false, 0, p.N, 64) || !rows_map(&mq, true, row0, rows, 64))
            return cudaErrorInvalidValue;
        mdq = mq; mdp = mq;           // a missing output gets a map that is never used
        if (dQ && !make_out_map(&mdq, dQ + row0 * lddq, rows, p.d, lddq, 1)) return cudaErrorInvalidValue;
        if (dP && !make_out_map(&mdp, dP, p.N, p.d, lddp, 1)) return cudaErrorInvalidValue;
        const unsigned grid = 2u * (unsigned)gp.pairs;
        auto go = [&](auto k, size_t smem) {
            return launch_chained(k, grid, ST_THREADS, smem, 2, st, wk, wm, mp, mq, mdq, mdp, gp);
        };
        return f32 ? go(strip_grad_kernel<true, 128>, SMEM_GF32)
               : width == 128 ? go(strip_grad_kernel<false, 128>, SMEM_G128)
                              : go(strip_grad_kernel<false, 256>, SMEM_G);
    }
};

}  // namespace

// Calls with rows of at most 384 values that the sweeps (gc_narrow.cu, gc_tc.cu) serve better: they keep the
// weights on the chip and form the logits again, where strips write and read (in a build, also convert) the
// weights in memory.  They gain with the pairs; and where one side is far longer than the other, since the
// strip plan has few long gradient tiles there and few CTA pairs to take them.  us, sweeps / strips:
//   build     d =  64  2900 x 5800 57 / 56     4500 x 4500 58 / 63    d = 128  4000 x 4000 58 / 53   4500 x 4500 61 / 63
//             d = 256  6000 x 6000 101 / 101, 8192 x 8192 to the sweeps by the older sweep of sizes
//             d <= 128 6500 x 128 40 / 39      10000 x 128 42 / 53    12500 x 384 46 / 44
//                      64 x 6500 43 / 38       64 x 10000 47 / 53     100 x 12500 51 / 44
//             d = 256  64 x 10000 56 / 54      64 x 12500 60 / 63     64 x 16000 65 / 76    64 x 64000 10 : 8
//   backward  d =  64  2000 x 2000 28 / 24     2048 x 4096 31 / 34    d = 128  3000 x 1500 33 / 27   2048 x 4096 32 / 35
//             d <= 128 4000 x 64 about even    5000 x 64 27 / 30      5000 x 256 33 / 30     6500 x 256 35 / 36
//                      64 x 4000 about even    64 x 5000 25 / 29      100 x 32000 52 / 54    180 x 16000 even
//             d = 256  64 x 5000 31 / 30       64 x 6500 33 / 35      64 x 32000 79 / 89     64 x 64000 9 : 10
//   dQ alone  d <= 128 600 x 600 16 / 15       1000 x 1000 15 / 17    64 x 4000 10 : 13      16 x 16000 10 : 12
//             d = 256  1000 x 1000 18 / 18     1500 x 1500 20 / 21    64 x 12500 33 / 31     16000 x 256 10 : 17
//             d = 384  2000 x 2000 26 / 26     2000 x 4000 32 / 36    1024 x 16384 60 / 47   16000 x 180 10 : 13
//   dP alone  d <= 128 1000 x 1000 16 / 15     2000 x 1000 16 / 19    4000 x 64 10 : 15
//             d = 256  1500 x 1500 20 / 19     2000 x 2000 20 / 24    4000 x 256 10 : 9      128 x 16000 10 : 13
//             d = 384  2000 x 2000 27 / 25     4000 x 2000 32 / 36    6000 x 12000 159 / 123
//   dQ, loss  d <= 128 3500 x 3500 43 / 43     4000 x 4000 40 / 50    1000 x 12000 48 / 48   64000 x 128 10 : 14
//             d = 256  4000 x 4000 53 / 54     4000 x 8000 even
//             d = 384  4000 x 4000 54 / 54     4000 x 8000 77 / 87    1024 x 32768 122 / 93
//   dP of a rank (of eight; the sweeps launch two kernels more)   d = 128  3000 x 750 23 / 23   4096 x 1024 23 / 27
//             d = 256  6000 x 1500 37 / 34     8192 x 2048 44 / 44, 16384 x 2048 65 / 71
//   both directions  d = 128  12000 x 12000 431 / 366   16384 x 16384 585 / 646   7 x 9470 60 / 76
static bool sweeps_serve(StripUse use, int64_t B, int64_t N, int d) {
    constexpr int64_t M = 1 << 20;
    const int64_t pairs = B * N;
    const bool narrow = d <= 128, middle = !narrow && d <= 256;       // else up to 384
    if (use == STRIP_FWD) return false;
    if (use == STRIP_BUILD) {
        if (narrow && ((B >= 7168 && N <= 256) || (N >= 7168 && B <= 64))) return true;
        if (middle && B <= 64 && N >= 11264 && N < 49152) return true;
        return pairs > (d <= 64 ? 17 * M : narrow ? 18 * M : middle ? 56 * M : pairs);
    }
    if (use == STRIP_BWD) {
        if (narrow && ((B >= 4608 && N <= 128) || (B >= 6144 && N <= 384))) return true;
        if (narrow && N >= 4608 && (B <= 64 || (B <= 128 && N < 24576))) return true;
        if (middle && N >= 6144 && N < 49152 && B <= 64) return true;
        return narrow && pairs > (d <= 64 ? 6 * M : 7 * M);
    }
    if (use == STRIP_BUILD_DQ) {
        if (narrow) return B >= 32768 || pairs > (B <= 1024 ? 20 * M : 12 * M);
        return pairs > (middle ? 28 * M : B <= 1500 ? 44 * M : 15 * M);
    }
    if (use == STRIP_BWD_DQ) {
        if (narrow) return pairs > 3 * M / 4 || B > 2560 || N > 2560;
        if (middle) return B <= 256 ? N > 1280 && N < 8192 : pairs > M || B >= 8192;
        return B > 1024 && (pairs > 4 * M || B >= 8192);
    }
    if (use == STRIP_BWD_DP) {
        if (narrow) return pairs > 3 * M / 4 || B > 2560 || N > 8192;
        if (middle) return N > 256 && (pairs > 9 * M / 4 || N >= 8192);
        return N > 512 && pairs > 4 * M && (N < B + B / 2 || N > 8 * B);
    }
    if (use == STRIP_SHARD_DP) return pairs > (narrow ? 2 * M : middle ? 14 * M : pairs);
    if (!narrow && !middle) return false;
    return (narrow && pairs > 160 * M) || (B <= 64 && N >= 4096);       // STRIP_TWO_DIR
}

// Which calls take the strip plan.  fp32 and bf16 widths that are no multiple of 64: the problems of
// small_tiled_applicable.  (Both its bounds come from an earlier plan, which kept planes of partial sums per tile
// pair; strips would not need them.)  bf16 rows in whole 64s: all calls but those of sweeps_serve, and but more
// than 2^18 passages with more than 256 M pairs.  That limit dates from strips of as many pairs and is not where
// the routes cross now (us, sweeps / strips, 1024 x 300000 x 768: loss 514 / 322, backward 2394 / 1154, build 2572 /
// 1451, dQ with the loss 853 / 1084; 2048 x 524288 x 768: 1595 / 1098, 6409 / 4078, 6539 / 6681, 2911 / 3705).
// GRADCACHE_PLAN=sweeps: as in gc_small.cu.
bool strip_applicable(StripUse use, int64_t B, int64_t N, int d, int dtype) {
    const char* e = getenv("GRADCACHE_PLAN");
    if (e && strcmp(e, "sweeps") == 0) return false;
    if (d % 8 != 0 || d > MAX_D || small_applicable(B, N, d, dtype)) return false;
    if (N > (1 << 24) || B > (1 << 24)) return false;
    if (dtype == GC_F32 || d % 64 != 0) return small_tiled_applicable(B, N, d, dtype);
    if (N > 1 << 18 && B * N > (int64_t)256 << 20) return false;
    return d > 384 || !sweeps_serve(use, B, N, d);
}

// A build that forms the logits twice, for the logsumexp and then for the weights, and has no row pass:
// rows for which a product costs less than reading, converting and writing the weights out of the memory
// (384: 12000 x 24000 871 us with the row pass, 812 without, 16384 x 32768 1661 and 1593; 8192 x 16384
// 375 and 395.  512: 16384 x 16384 808 and 815).
static bool logits_twice(int64_t B, int64_t N, int d, int dtype) {
    return dtype != GC_F32 && d <= 384 && B * N > (int64_t)192 << 20;
}

size_t strip_workspace_bytes(int64_t B, int64_t N, int d, int dtype) {
    return strip_layout(B, N, d, dtype).total;
}
size_t strip_forward_bytes(int64_t B, int64_t N, int d, int dtype) {
    return strip_layout(B, N, d, dtype, true).total;
}

int strip_launches(int op, int64_t B, int64_t N, int d, int dtype) {
    const int strips = strip_layout(B, N, d, dtype).strips, pre = dtype == GC_F32 ? 1 : 0;
    if (op == GC_OP_FWD) return pre + 2 * strips;
    if (op == GC_OP_BWD) return pre + (dtype == GC_F32 ? 3 : 2) * strips;
    if (logits_twice(B, N, d, dtype)) return 4 * strips;
    return pre + 3 * strips;
}

cudaError_t strip_forward(const Problem& p, void* ws, float* loss, float* row_lse, float* pos_logit,
                          int* dev_status, cudaStream_t st, const TwoDirection* two) {
    cudaError_t e = configure_kernels();
    StripRun r(p, ws, dev_status, st, true);
    r.two = two;
    if (e == cudaSuccess && r.f32) e = r.split();
    for (int s = 0; s < r.l.strips && e == cudaSuccess; ++s) {
        e = r.logits(s, LOGIT_FWD, nullptr, s == 0);
        if (e == cudaSuccess) e = r.rows_kernel(s, false, false, row_lse, pos_logit, loss);
    }
    return e;
}

cudaError_t strip_build(const Problem& p, void* ws, float* loss, float* row_lse, float* pos_logit,
                        float* dQ, int64_t lddq, float* dP, int64_t lddp, int* dev_status,
                        cudaStream_t st) {
    if (dP && logits_twice(p.B, p.N, p.d, p.dtype)) {
        const cudaError_t f = strip_forward(p, ws, loss, row_lse, pos_logit, dev_status, st);
        return f == cudaSuccess ? strip_backward(p, ws, row_lse, dQ, lddq, dP, lddp, dev_status, st) : f;
    }
    cudaError_t e = configure_kernels();
    StripRun r(p, ws, dev_status, st);
    if (e == cudaSuccess && r.f32) e = r.split();
    for (int s = 0; s < r.l.strips && e == cudaSuccess; ++s) {
        e = r.logits(s, LOGIT_STASH, nullptr, s == 0);
        if (e == cudaSuccess) e = r.rows_kernel(s, true, false, row_lse, pos_logit, loss);
        if (e == cudaSuccess) e = r.grads(s, dQ, lddq, dP, lddp, loss);
    }
    return e;
}

cudaError_t strip_backward(const Problem& p, void* ws, const float* row_lse, float* dQ, int64_t lddq,
                           float* dP, int64_t lddp, int* dev_status, cudaStream_t st,
                           const float* col_neg, float grad_scale, const TwoDirection* two, float* loss) {
    cudaError_t e = configure_kernels();
    StripRun r(p, ws, dev_status, st);
    r.col_neg = col_neg;
    r.grad_scale = grad_scale;
    r.two = two;
    if (e == cudaSuccess && r.f32) e = r.split();
    for (int s = 0; s < r.l.strips && e == cudaSuccess; ++s) {
        e = r.logits(s, col_neg ? LOGIT_W2 : LOGIT_W, row_lse, s == 0);
        if (e == cudaSuccess && r.f32)
            e = r.rows_kernel(s, true, true, const_cast<float*>(row_lse), nullptr, nullptr);
        if (e == cudaSuccess) e = r.grads(s, dQ, lddq, dP, lddp, loss);
    }
    return e;
}

}  // namespace gc
