// One-launch plan for fp32 batches of a single tile: B <= 128 queries, N <= 128 passages, d a multiple
// of 8 up to 1024 (bf16: gc_small.cu).  CTA c owns columns [64 c, 64 c + 64) of dQ and dP.
//
// The logits of such a batch take six bf16 products per step (see below), so the CTAs of a cluster of
// up to four share them: each forms S over its part of the contraction, its own slice last, and sends
// the other CTAs' rows of the partial tile to their shared memory.  A CTA then has 128 / C rows of S
// whole; it takes their softmax and sends the weights W_ij = p_ij - [j = r_i] (0 at masked pairs, rows
// past B and columns past N) to every CTA of the cluster as two bf16 terms, operands of the products
//     dQ[:, slice] = W P[:, slice] / (B tau),     dP[:, slice] = W^T Q[:, slice] / (B tau)
// whose other operand is the slice's terms where the logit loop left them.  CTAs of different clusters
// do not talk to one another.  Cluster 0 also writes loss, row_lse, pos_logit and the pos_idx flags.
//
// Converter warps split every value into three bf16 terms x = t1 + t2 + t3 (each the upper 16 bits of
// what the previous ones left, so the sum is exact) as it arrives; S takes t1 t1', t1 t2', t1 t3',
// t2 t1', t2 t2', t3 t1' in fp32 accumulation (spread over three accumulators, see the MMA warp), the
// gradient products take w1 (t1 + t2 + t3) + w2 (t1 + t2).
//
// What bounds it (64 x 128 x 768, 16.7 us): a chain of latencies.  A step of 32 columns is 12 MMAs of a single
// CTA, 0.7 us; with every CTA taking all 24 steps the call was 28.7 us.
#include "tc_common.cuh"

namespace gc {

namespace {

constexpr int SF_WORKERS = 8;                    // converter / softmax / epilogue warps
constexpr int SF_PROD_WARP = 0;
constexpr int SF_MMA_WARP = 1;
constexpr int SF_FIRST_WORKER = 2;
constexpr int SF_THREADS = 32 * (SF_FIRST_WORKER + SF_WORKERS);
constexpr uint32_t TILE = 16384;                 // 128 rows x 128 bytes
constexpr int SF_STAGES = 2;
constexpr uint32_t SF_STAGE = 2 * TILE;          // 32 fp32 columns of Q and of P
constexpr uint32_t SF_TERM_OFF = SF_STAGES * SF_STAGE;       // q1 q2 q3 p1 p2 p3
constexpr uint32_t SF_RECV_OFF = SF_TERM_OFF + 6 * TILE;     // partial logits of this CTA's rows
constexpr uint32_t SF_GROUP = 32 * 128 * 4;                  // 32 rows of them
constexpr size_t SF_SMEM = 1024 + SF_RECV_OFF + 4 * SF_GROUP;
constexpr uint32_t COL_S = 0, COL_DQ = 256, COL_DP = 320, COL_S2 = 384;   // tensor-memory columns

static_assert(SF_SMEM <= SMEM_LIMIT - 1536, "shared memory budget");
static_assert(4 * TILE <= SF_TERM_OFF, "the weights fit over the drained ring");

struct SmallF32Params {
    int B, N, d;
    int op;                   // GC_OP_FWD, GC_OP_BWD, GC_OP_BUILD
    int mask_mode;
    int mask_shift;           // masked pair: j == i + mask_shift
    float scale2;             // log2(e) / tau
    float inv_tau;
    float out_scale;          // 1 / (B tau)
    float inv_mean;           // 1 / B
    const int32_t* pos_idx;
    const float* row_lse_in;  // GC_OP_BWD
    // Forward of several tiles (grid y = query tiles, grid z = passage tiles): one (max, sum) slot per
    // passage tile and row, slot t at [t * B + i] (natural-log units), and the positive's logit, for the
    // combine kernel that follows
    int tiled;
    float* part_m;
    float* part_l;
    float* pos_ws;
    int* zero_me;             // block ticket of the loss reduction that follows: cleared here
    float* loss;
    float* row_lse;
    float* pos_logit;         // may be NULL
    int have_q, have_p;       // gradients wanted
    int* dev_status;
};

struct SmallF32Bars {
    uint64_t full[SF_STAGES];
    uint64_t empty[SF_STAGES];
    uint64_t term_full[2];
    uint64_t term_empty[2];
    uint64_t s_full;
    uint64_t acc_full;
};

__device__ __forceinline__ float4 lds128f(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts128u(uint32_t addr, const uint32_t (&w)[4]) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(addr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
}
// to any CTA of the cluster
__device__ __forceinline__ void stc128u(uint32_t cluster_addr, const uint32_t (&w)[4]) {
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(cluster_addr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void workers_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(32 * SF_WORKERS) : "memory");
}

// C: CTAs of a cluster, 1, 2 or 4.
template <int C>
__global__ void __launch_bounds__(SF_THREADS, 1)
small_f32_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapP,
                 const __grid_constant__ CUtensorMap mapDQ, const __grid_constant__ CUtensorMap mapDP,
                 const SmallF32Params p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) SmallF32Bars bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ float x_row[SF_WORKERS][32], x_pos[32];     // exchange between the workers' columns
    __shared__ float loss_part[4];
    volatile int* abort_flag = &abort_s;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // warp-uniform
    const int lane = threadIdx.x & 31;
    const int slice = blockIdx.x;
    const int rank = C > 1 ? (int)cluster_ctarank() : 0;      // == slice % C
    const bool do_grad = p.op != GC_OP_FWD;
    // this CTA's tile pair: rows x0 .. of Q, rows y0 .. of P; B_ and N_ are the rows it holds
    const int x0 = 128 * (int)blockIdx.y, y0 = 128 * (int)blockIdx.z;
    const int B_ = min(128, p.B - x0), N_ = min(128, p.N - y0);
    const int blocks = (p.d + 63) / 64;                       // 64-column blocks of the contraction
    const bool own = do_grad && slice < blocks;
    // this CTA's blocks: rank, rank + C, ..., the own slice moved to the end
    const int mine = (blocks - rank + C - 1) / C;
    auto block_at = [&](int b) {
        if (!own) return rank + C * b;
        const int at = (slice - rank) / C;
        return rank + C * (b == mine - 1 ? at : b < at ? b : b + 1);
    };
    const int steps = 2 * mine;                               // of 32 columns
    const int n_pad = (N_ + 15) & ~15;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t w_smem = base;                             // over the drained ring
    const uint32_t term_smem = base + SF_TERM_OFF, recv_smem = base + SF_RECV_OFF;
    // the same place in CTA r of the cluster
    auto in_cta = [&](uint32_t addr, int r) { return C > 1 ? mapa_u32(addr, (uint32_t)r) : addr; };

    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < SF_STAGES; ++s) {
            mbar_init(smem_u32(&bars.full[s]), 1);
            mbar_init(smem_u32(&bars.empty[s]), SF_WORKERS);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&bars.term_full[s]), SF_WORKERS);
            mbar_init(smem_u32(&bars.term_empty[s]), 1);
        }
        mbar_init(smem_u32(&bars.s_full), 1);
        mbar_init(smem_u32(&bars.acc_full), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == SF_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_s)), "r"((uint32_t)TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (warp >= SF_FIRST_WORKER) {
        // rows past B (N) are never converted: the term tiles start out as zeros
        const uint32_t z[4] = {0u, 0u, 0u, 0u};
        for (int e = (int)threadIdx.x - 32 * SF_FIRST_WORKER; e < (int)(6 * TILE / 16); e += 32 * SF_WORKERS)
            sts128u(term_smem + 16 * e, z);
    }
    tc_fence_before();
    __syncthreads();
    if (C > 1) cluster_sync_all();     // the cluster's CTAs run: their shared memory may be written
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    dep_release();
    dep_wait();

    const int wt = (int)threadIdx.x - 32 * SF_FIRST_WORKER;     // worker thread 0 .. 255
    const int ww = warp - SF_FIRST_WORKER;                       // worker warp 0 .. 7
    const int q = warp & 3;                                      // tensor-memory lane quarter
    const int half = ww >> 2;                                    // column half of S / of a slice
    const uint32_t lane_addr = (uint32_t)(32 * q) << 16;
    bool ok = true;

    // ------------------------------ partial logits ------------------------------------------------
    if (warp == SF_PROD_WARP) {
        int stage = 0;
        uint32_t phase = 0;
        for (int t = 0; t < steps; ++t) {
            ok = mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag);
            if (!ok) break;
            const uint32_t full = smem_u32(&bars.full[stage]);
            const uint32_t dst = base + stage * SF_STAGE;
            const int col = 64 * block_at(t >> 1) + 32 * (t & 1);
            if (elect_one()) {
                mbar_expect_tx(full, 2 * TILE);
                tma_load_2d(dst, &mapQ, col, x0, full);
                tma_load_2d(dst + TILE, &mapP, col, y0, full);
            }
            if (++stage == SF_STAGES) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == SF_MMA_WARP) {
        const uint32_t idesc_s = instr_desc(n_pad, false, XROWS, false);
        for (int t = 0; t < steps; ++t) {
            const int h = t & 1;
            ok = mbar_wait(smem_u32(&bars.term_full[h]), (uint32_t)(t >> 1) & 1u, abort_flag);
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
                    const uint32_t k = (uint32_t)(2 * (2 * h + kk));     // 32 bytes per K = 16
                    const uint32_t q1 = desc_lo(term_smem, 0) + k;
                    const uint32_t p1 = desc_lo(term_smem + 3 * TILE, 0) + k;
                    constexpr uint32_t T = TILE >> 4;
                    // The accumulator adds with truncation: the leading product alternates between two
                    // accumulators and the five small ones have a third, so that each takes few
                    // additions of its own magnitude; the workers sum the three in fp32.
                    const uint32_t lead = tmem + COL_S + 128 * kk, rest = tmem + COL_S2;
                    if (t == 0) mma_ss<false, false>(lead, q1, p1, idesc_s);
                    else        mma_ss<true, false>(lead, q1, p1, idesc_s);
                    if (t == 0 && kk == 0) mma_ss<false, false>(rest, q1, p1 + T, idesc_s);
                    else                   mma_ss<true, false>(rest, q1, p1 + T, idesc_s);
                    mma_ss<true, false>(rest, q1 + T, p1, idesc_s);
                    mma_ss<true, false>(rest, q1 + T, p1 + T, idesc_s);
                    mma_ss<true, false>(rest, q1, p1 + 2 * T, idesc_s);
                    mma_ss<true, false>(rest, q1 + 2 * T, p1, idesc_s);
                }
                tc_commit(smem_u32(&bars.term_empty[h]));
                if (t == steps - 1) tc_commit(smem_u32(&bars.s_full));
            }
        }
    } else {
        // fp32 -> three bf16 terms by truncation (t1 = the upper 16 bits of x, t2 those of x - t1, t3
        // those of what is left: x = t1 + t2 + t3 exactly).  Item = 8 consecutive columns of one row
        // (two 16-byte pieces in, one piece per term out).  Eight neighbouring threads take four items
        // of row r and four of row r + 4, the second row fetching its two pieces in the opposite
        // order: loads and stores both fall on distinct banks.
        int stage = 0;
        uint32_t phase = 0;
        for (int t = 0; t < steps; ++t) {
            const int h = t & 1;
            ok = mbar_wait(smem_u32(&bars.full[stage]), phase, abort_flag) &&
                 mbar_wait(smem_u32(&bars.term_empty[h]), ((uint32_t)(t >> 1) & 1u) ^ 1u, abort_flag);
            if (!ok) break;
            const uint32_t src0 = base + stage * SF_STAGE;
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int id = wt + 256 * it;
                const int cp = id & 3, rr = (id >> 2) & 1, b = (id >> 3) & 3, a = (id >> 5) & 15;
                const int mat = id >> 9;
                const int r = 8 * a + b + 4 * rr, sw = r & 7;
                if (r >= (mat ? N_ : B_)) continue;
                const uint32_t src = src0 + mat * TILE + r * 128;
                const int first = (2 * cp) ^ rr;
                const float4 A = lds128f(src + (uint32_t)((first ^ sw) << 4));
                const float4 Bv = lds128f(src + (uint32_t)(((first ^ 1) ^ sw) << 4));
                const float4 f0 = rr ? Bv : A, f1 = rr ? A : Bv;
                const float x[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
                uint32_t t1[4], t2[4], t3[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t a0 = __float_as_uint(x[2 * e]), a1 = __float_as_uint(x[2 * e + 1]);
                    const float r0 = x[2 * e] - __uint_as_float(a0 & 0xffff0000u);
                    const float r1 = x[2 * e + 1] - __uint_as_float(a1 & 0xffff0000u);
                    const uint32_t b0 = __float_as_uint(r0), b1 = __float_as_uint(r1);
                    const float s0 = r0 - __uint_as_float(b0 & 0xffff0000u);
                    const float s1 = r1 - __uint_as_float(b1 & 0xffff0000u);
                    t1[e] = __byte_perm(a0, a1, 0x7632);      // the two upper halves
                    t2[e] = __byte_perm(b0, b1, 0x7632);
                    t3[e] = __byte_perm(__float_as_uint(s0), __float_as_uint(s1), 0x7632);
                }
                const uint32_t dst = term_smem + (uint32_t)(3 * mat) * TILE + r * 128 +
                                     (uint32_t)(((4 * h + cp) ^ sw) << 4);
                sts128u(dst, t1);
                sts128u(dst + TILE, t2);
                sts128u(dst + 2 * TILE, t3);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(smem_u32(&bars.term_full[h]));
                mbar_arrive(smem_u32(&bars.empty[stage]));
            }
            if (++stage == SF_STAGES) { stage = 0; phase ^= 1u; }
        }
        ok = ok && mbar_wait(smem_u32(&bars.s_full), 0, abort_flag);
        if (ok) {
            // this warp's 32 rows x 64 columns of the partial tile to the CTA that owns the rows: groups
            // of 32 rows, 16-byte pieces of a column group lane by lane
            tc_fence_after();
            constexpr int R = 4 / C;                            // groups of 32 rows per CTA
            const uint32_t dst = in_cta(recv_smem + (uint32_t)(rank * R + q % R) * SF_GROUP, q / R) +
                                 (uint32_t)(half * 16 * 32 + lane) * 16u;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const int jb = 64 * half + 32 * g;
                if (jb >= N_) break;
                uint32_t v[32], u[32], s[32];
                tmem_ld32(tmem + lane_addr + COL_S + jb, s);
                tmem_ld32(tmem + lane_addr + COL_S + 128 + jb, v);
                tmem_ld32(tmem + lane_addr + COL_S2 + jb, u);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    uint32_t w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        w[e] = __float_as_uint((__uint_as_float(s[4 * j + e]) + __uint_as_float(v[4 * j + e])) +
                                               __uint_as_float(u[4 * j + e]));
                    stc128u(dst + (uint32_t)((8 * g + j) * 32) * 16u, w);
                }
            }
        }
    }
    __syncwarp();
    if (C > 1) cluster_sync_all();
    else       __syncthreads();

    // ------------------------------ softmax of this CTA's rows --------------------------------------
    // Worker warp ww takes columns [16 ww, 16 ww + 16), a lane a row.
    if (warp >= SF_FIRST_WORKER) {
        constexpr int R = 4 / C;
        const int jb = 16 * ww;
        const uint32_t piece = (uint32_t)(((ww >> 2) * 16 + (ww & 3) * 4) * 32 + lane) * 16u;
#pragma unroll 1
        for (int g = 0; g < R; ++g) {
            const int quarter = rank * R + g;
            const int i = 32 * quarter + lane;
            float s[16];
#pragma unroll
            for (int c = 0; c < C; ++c) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 v = lds128f(recv_smem + (uint32_t)(c * R + g) * SF_GROUP + piece + (uint32_t)(j * 32) * 16u);
                    const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[4 * j + e] = c == 0 ? f[e] : s[4 * j + e] + f[e];
                }
            }
            // columns are counted within the tile: the positive and the masked pair of row i fall
            // into it or not
            const int32_t r_i = i < B_ ? p.pos_idx[x0 + i] : -1;
            int flags = 0;
            if (i < B_) {
                if (r_i < 0 || r_i >= p.N) flags = GC_DEV_POS_RANGE;
                else if (p.mask_mode == GC_MASK_SELF && r_i == x0 + i + p.mask_shift) flags = GC_DEV_POS_MASKED;
            }
            const int pos = (flags || r_i < y0 || r_i >= y0 + N_) ? -1 : r_i - y0;
            const int masked = p.mask_mode == GC_MASK_SELF ? x0 + i + p.mask_shift - y0 : -1;
            float lse2;
            if (p.op == GC_OP_BWD) {
                lse2 = p.row_lse_in[i < B_ ? x0 + i : 0] * 1.4426950408889634f;
            } else {
                // The maximum is kept in units of <q, p> (unscaled), so that the row's logsumexp and its
                // positive logit come out of the same product with 1/tau: lse_i - S_{i,r_i} is exactly 0
                // when the positive is the only column.
                float m = -INFINITY, sum = 0.f;
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    if (e == pos - jb) x_pos[lane] = s[e];
                    if (jb + e < N_ && e != masked - jb) m = fmaxf(m, s[e]);
                }
                x_row[ww][lane] = m;
                workers_sync();
                const float pos2 = pos >= 0 ? x_pos[lane] : 0.f;
#pragma unroll
                for (int w = 0; w < SF_WORKERS; ++w) m = fmaxf(m, x_row[w][lane]);
                workers_sync();
                const float ref = m == -INFINITY ? 0.f : m;     // all columns masked
#pragma unroll
                for (int e = 0; e < 16; ++e)                    // (s - max) first: the largest term is 2^0
                    if (jb + e < N_ && e != masked - jb) sum += ex2((s[e] - ref) * p.scale2);
                x_row[ww][lane] = sum;
                workers_sync();
                sum = 0.f;
#pragma unroll
                for (int w = 0; w < SF_WORKERS; ++w) sum += x_row[w][lane];
                const float lg = log2f(sum);                    // once per row: the accurate one
                lse2 = m * p.scale2 + lg;
                const float lnsum = lg * 0.6931471805599453f;
                if (p.tiled) {
                    if (ww == 0 && i < B_ && slice == rank) {
                        p.part_m[(int64_t)blockIdx.z * p.B + x0 + i] = m * p.inv_tau;
                        p.part_l[(int64_t)blockIdx.z * p.B + x0 + i] = sum;
                        if (pos >= 0) p.pos_ws[x0 + i] = pos2 * p.inv_tau;
                    }
                    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && wt == 0 && p.zero_me) *p.zero_me = 0;
                } else if (slice == rank && ww == 0) {          // cluster 0
                    float term = 0.f;
                    if (i < B_) {
                        p.row_lse[i] = m * p.inv_tau + lnsum;
                        if (p.pos_logit) p.pos_logit[i] = pos2 * p.inv_tau;
                        term = (m - pos2) * p.inv_tau + lnsum;  // no cancellation of two roundings
                    }
                    for (int o = 16; o > 0; o >>= 1) term += __shfl_xor_sync(0xffffffffu, term, o);
                    if (lane == 0)
                        asm volatile("st.shared::cluster.f32 [%0], %1;"
                                     ::"r"(in_cta(smem_u32(&loss_part[quarter]), 0)), "f"(term) : "memory");
                }
            }
            if (slice == rank && !p.tiled && ww == 0 && flags && p.dev_status) atomicOr(p.dev_status, flags);
            if (do_grad) {
                // Weights as MMA operands: chunk c = 64 columns, element (i, j) in 16-byte piece
                // ((j % 64) / 8) ^ (i % 8) of row i: a K-major A operand for dQ and, read by columns, an
                // MN-major one for dP.  The second term is two chunks further.
                float w[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    w[e] = ex2(fmaf(s[e], p.scale2, -lse2));
                    if (jb + e >= N_ || e == masked - jb) w[e] = 0.f;
                    if (e == pos - jb) w[e] -= 1.f;
                    if (i >= B_) w[e] = 0.f;
                }
                const uint32_t row = w_smem + (uint32_t)(jb >> 6) * TILE + i * 128;
#pragma unroll
                for (int pc = 0; pc < 2; ++pc) {
                    const uint32_t dst = row + (uint32_t)(((((jb & 63) >> 3) + pc) ^ (i & 7)) << 4);
                    uint32_t hi[4], lo[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float a = w[8 * pc + 2 * e], b = w[8 * pc + 2 * e + 1];
                        hi[e] = pack_bf16(a, b);
                        lo[e] = pack_bf16(a - __uint_as_float(hi[e] << 16), b - __uint_as_float(hi[e] & 0xffff0000u));
                    }
#pragma unroll
                    for (int c = 0; c < C; ++c) {
                        const uint32_t there = in_cta(dst, c);
                        stc128u(there, hi);
                        stc128u(there + 2 * TILE, lo);
                    }
                }
            }
            if (R > 1) workers_sync();                          // x_row and x_pos are free again
        }
        asm volatile("fence.proxy.async;" ::: "memory");
    }
    __syncwarp();
    if (C > 1) cluster_sync_all();
    else       __syncthreads();

    // ------------------------------ gradients of the own slice ---------------------------------------
    // (an abort anywhere in the cluster leaves undefined numbers and the status bit, nothing else)
    if (warp == SF_MMA_WARP) {
        if (own && !*abort_flag) {
            asm volatile("fence.proxy.async;" ::: "memory");
            tc_fence_after();
            const uint32_t idesc_dq = instr_desc(64, true, XROWS, false);    // A = W, K-major
            const uint32_t idesc_dp = instr_desc(64, true, XROWS, true);     // A = W^T: MN-major
            if (elect_one()) {
                // products (weight term, operand term): w1 t1, w1 t2, w1 t3, w2 t1, w2 t2 (the terms are
                // truncations: dropping t3 would leave a one-sided 2^-16)
                constexpr uint32_t T = TILE >> 4;
                const uint32_t w_term[5] = {0u, 0u, 0u, 2 * T, 2 * T};
                const uint32_t o_term[5] = {0u, T, 2 * T, 0u, T};
                const int kq = (N_ + 15) / 16, kp = (B_ + 15) / 16;          // the rest is zeros
                if (p.have_q)
                    for (int k = 0; k < kq; ++k) {
#pragma unroll
                        for (int pr = 0; pr < 5; ++pr) {
                            const uint32_t a = desc_lo(w_smem + (k >> 2) * TILE, 0) + w_term[pr] + 2 * (k & 3);
                            const uint32_t b = desc_lo(term_smem + 3 * TILE, 0) + o_term[pr] + 128 * k;
                            if (k == 0 && pr == 0) mma_ss<false, false>(tmem + COL_DQ, a, b, idesc_dq);
                            else                   mma_ss<true, false>(tmem + COL_DQ, a, b, idesc_dq);
                        }
                    }
                if (p.have_p)
                    for (int k = 0; k < kp; ++k) {
#pragma unroll
                        for (int pr = 0; pr < 5; ++pr) {
                            const uint32_t a = desc_lo(w_smem, TILE) + w_term[pr] + 128 * k;
                            const uint32_t b = desc_lo(term_smem, 0) + o_term[pr] + 128 * k;
                            if (k == 0 && pr == 0) mma_ss<false, false>(tmem + COL_DP, a, b, idesc_dp);
                            else                   mma_ss<true, false>(tmem + COL_DP, a, b, idesc_dp);
                        }
                    }
                tc_commit(smem_u32(&bars.acc_full));
            }
        }
    } else if (warp >= SF_FIRST_WORKER) {
        if (p.op != GC_OP_BWD && !p.tiled && slice == 0 && wt == 0)
            *p.loss = (((loss_part[0] + loss_part[1]) + loss_part[2]) + loss_part[3]) * p.inv_mean;
        // A warp's 32 x 32 block goes through a 4 KB buffer (over the received logits) and leaves with
        // one bulk tensor store, which clips it at the matrix's last row and column.
        if (own && mbar_wait(smem_u32(&bars.acc_full), 0, abort_flag)) {
            tc_fence_after();
            const int col = 64 * slice + 32 * half;
            const uint32_t slot = recv_smem + (uint32_t)ww * 8192u;
#pragma unroll
            for (int blk = 0; blk < 2; ++blk) {                 // dQ, dP
                const int rows = blk == 0 ? p.B : p.N;
                if (!(blk == 0 ? p.have_q : p.have_p) || 32 * q >= rows || col >= p.d) continue;
                uint32_t v[32];
                tmem_ld32(tmem + lane_addr + (blk == 0 ? COL_DQ : COL_DP) + 32 * half, v);
                tmem_ld_wait();
                stage_block(slot + (uint32_t)blk * 4096u, v, p.out_scale, lane);
                __syncwarp();
                if (lane == 0)
                    tma_store_3d(blk == 0 ? &mapDQ : &mapDP, slot + (uint32_t)blk * 4096u, col, 32 * q, 0);
            }
            if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
            __syncwarp();
        }
    }

    // ------------------------------ teardown ------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        // let bulk copies still in flight land before the shared memory is released
        uint64_t t0 = global_ns();
        while (global_ns() - t0 < 200000ull) __nanosleep(1000);
        if (threadIdx.x == 0 && p.dev_status) atomicOr(p.dev_status, GC_DEV_WAIT_LIMIT);
        __syncthreads();
    }
    if (warp == SF_MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     ::"r"(tmem), "r"((uint32_t)TMEM_COLS) : "memory");
    }
}

// CTAs that own columns, in whole clusters (a forward: one cluster forms the logits).
cudaError_t launch_f32(const Problem& pr, float* dQ, int64_t lddq, float* dP, int64_t lddp,
                       SmallF32Params p, unsigned tiles_x, unsigned tiles_y, cudaStream_t st) {
    CUtensorMap mq, mp;
    if (!make_map_f32(&mq, pr.Q, pr.B, pr.d, pr.ldq, 128) || !make_map_f32(&mp, pr.P, pr.N, pr.d, pr.ldp, 128))
        return cudaErrorInvalidValue;
    // gradient outputs as [1][rows][d] for the epilogue's bulk tensor stores; a missing one gets a map
    // that is never used
    CUtensorMap mdq = mq, mdp = mp;
    if (dQ && !make_out_map(&mdq, dQ, pr.B, pr.d, lddq, 1)) return cudaErrorInvalidValue;
    if (dP && !make_out_map(&mdp, dP, pr.N, pr.d, lddp, 1)) return cudaErrorInvalidValue;
    p.B = (int)pr.B; p.N = (int)pr.N; p.d = pr.d;
    p.mask_mode = pr.mask_mode;
    p.mask_shift = (int)pr.mask_shift;
    p.scale2 = 1.4426950408889634f / pr.tau;
    p.inv_tau = 1.f / pr.tau;
    const float batch = (float)(pr.b_total > 0 ? pr.b_total : pr.B);
    p.out_scale = 1.f / (batch * pr.tau);
    p.inv_mean = 1.f / batch;
    p.pos_idx = pr.pos_idx;
    p.have_q = dQ != nullptr;
    p.have_p = dP != nullptr;

    static bool configured_on[64] = {false};      // the attribute belongs to (kernel, device)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured_on[dev]) {
        const void* all[] = {(const void*)small_f32_kernel<1>, (const void*)small_f32_kernel<2>,
                             (const void*)small_f32_kernel<4>};
        for (const void* f : all) {
            const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SF_SMEM);
            if (e != cudaSuccess) return e;
        }
        configured_on[dev] = true;
    }
    const unsigned slices = ((unsigned)pr.d + 63) / 64;
    const unsigned c = slices >= 4 ? 4 : slices >= 2 ? 2 : 1;      // every CTA has a block
    const unsigned x = p.op == GC_OP_FWD ? c : (slices + c - 1) / c * c;
    const dim3 grid(x, tiles_x, tiles_y);
    if (c == 4) return launch_chained(small_f32_kernel<4>, grid, SF_THREADS, SF_SMEM, 4, st, mq, mp, mdq, mdp, p);
    if (c == 2) return launch_chained(small_f32_kernel<2>, grid, SF_THREADS, SF_SMEM, 2, st, mq, mp, mdq, mdp, p);
    return launch_chained(small_f32_kernel<1>, grid, SF_THREADS, SF_SMEM, 1, st, mq, mp, mdq, mdp, p);
}

}  // namespace

// op: GC_OP_FWD (loss, row_lse, pos_logit), GC_OP_BWD (dQ, dP from row_lse_in) or GC_OP_BUILD.
cudaError_t launch_small_f32(int op, const Problem& pr, const float* row_lse_in, float* loss, float* row_lse,
                             float* pos_logit, float* dQ, int64_t lddq, float* dP, int64_t lddp,
                             int* dev_status, cudaStream_t st) {
    SmallF32Params p{};
    p.op = op;
    p.row_lse_in = row_lse_in;
    p.loss = loss; p.row_lse = row_lse; p.pos_logit = pos_logit;
    p.dev_status = dev_status;
    return launch_f32(pr, dQ, lddq, dP, lddp, p, 1, 1, st);
}

// Forward of several tiles (gc_loss_fwd_static, whose array has no room for fp32 logits): slots part_m /
// part_l [passage tiles][B], pos_ws [B]; `red` is the scratch of the combine kernel that follows.
cudaError_t launch_small_tiled_fwd(const Problem& pr, float* part_m, float* part_l, float* pos_ws,
                                   float* red, int* dev_status, cudaStream_t st) {
    SmallF32Params p{};
    p.op = GC_OP_FWD;
    p.tiled = 1;
    p.part_m = part_m; p.part_l = part_l; p.pos_ws = pos_ws;
    p.zero_me = reinterpret_cast<int*>(red);
    p.dev_status = dev_status;
    return launch_f32(pr, nullptr, 0, nullptr, 0, p, (unsigned)((pr.B + 127) / 128), (unsigned)((pr.N + 127) / 128), st);
}

}  // namespace gc
