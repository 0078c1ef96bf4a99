// One-launch plan for bf16 batches of a single tile: B <= 128 queries, N <= 256 passages, d a multiple
// of 8 (fp32: gc_small_f32.cu).  Loss (Eq. 1) and the representation gradients (Eq. 5-7) of such a
// batch are a few hundred MFLOP: several dependent launches cost more than the work.
//
// CTA c owns columns [64 c, 64 c + 64) of dQ and dP; the CTAs do not talk to one another.  Every
// CTA forms the whole logit tile S = Q P^T (tcgen05, fp32 in tensor memory) from 64-column slices
// of Q and P that a producer warp streams through shared memory, the softmax warps turn it into
// the weights W_ij = p_ij - [j = r_i] (0 at masked pairs, rows past B and columns past N), kept
// in shared memory as bf16 MMA operands, and two more products give the CTA's columns,
//     dQ[:, slice] = W P[:, slice] / (B tau),     dP[:, slice] = W^T Q[:, slice] / (B tau),
// with the slice of P (of Q) read as the MN-major B operand where the bulk tensor load left it.
// CTA 0 also writes loss, row_lse, pos_logit and the pos_idx flags.
//
// Every mbarrier wait is bounded.  The launch may start under the kernel before it in the stream.
#include <stdlib.h>
#include <string.h>

#include "tc_common.cuh"

namespace gc {

namespace {

constexpr int SM_WORKERS = 8;                    // softmax / epilogue warps
constexpr int SM_PROD_WARP = 0;
constexpr int SM_MMA_WARP = 1;
constexpr int SM_FIRST_WORKER = 2;
constexpr int SM_THREADS = 32 * (SM_FIRST_WORKER + SM_WORKERS);
constexpr uint32_t TILE = 16384;                 // 128 rows x 128 bytes
constexpr int SM_STAGES = 3;
constexpr uint32_t BF_STAGE = 3 * TILE;          // Q slice + P slice (two row tiles)
constexpr uint32_t BF_W_OFF = SM_STAGES * BF_STAGE;          // four weight chunks behind the ring
constexpr size_t SM_DYN_SMEM = 1024 + (size_t)SM_STAGES * BF_STAGE + 4 * TILE;
constexpr uint32_t COL_S = 0, COL_DQ = 256, COL_DP = 320;    // tensor-memory columns

static_assert(SM_DYN_SMEM <= SMEM_LIMIT - SMEM_STATIC_RESERVE, "shared memory budget");

struct SmallParams {
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
    float* loss;
    float* row_lse;
    float* pos_logit;         // may be NULL
    float* dQ;
    int64_t lddq;
    float* dP;
    int64_t lddp;
    int* dev_status;
};

struct SmallBars {
    uint64_t full[SM_STAGES];
    uint64_t empty[SM_STAGES];
    uint64_t s_full;
    uint64_t w_full;
    uint64_t acc_full;
};

__device__ __forceinline__ void sts128u(uint32_t addr, const uint32_t (&w)[4]) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(addr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&h);
}
// All worker threads take a decision together (named barrier 1).
__device__ __forceinline__ bool workers_all(bool mine) {
    uint32_t all;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "barrier.cta.red.and.pred p, 1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(all) : "r"(mine ? 1u : 0u), "n"(32 * SM_WORKERS) : "memory");
    return all != 0;
}
// 32 columns of this thread's row of S
__device__ __forceinline__ void load_s(uint32_t trow, int jb, float (&s)[32]) {
    uint32_t v[32];
    tmem_ld32(trow + COL_S + jb, v);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 32; ++e) s[e] = __uint_as_float(v[e]);
}
__device__ __forceinline__ void workers_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(32 * SM_WORKERS) : "memory");
}

__global__ void __launch_bounds__(SM_THREADS, 1)
small_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapP,
             const __grid_constant__ CUtensorMap mapDQ, const __grid_constant__ CUtensorMap mapDP,
             const SmallParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) SmallBars bars;
    __shared__ uint32_t tmem_base_s;
    __shared__ int abort_s;
    __shared__ float x_max[2][128], x_sum[2][128], x_pos[2][128];   // exchange between the column halves
    __shared__ float loss_part[4];
    volatile int* abort_flag = &abort_s;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);   // warp-uniform
    const int lane = threadIdx.x & 31;
    const int slice = blockIdx.x;
    const bool do_grad = p.op != GC_OP_FWD;
    const int B_ = p.B, N_ = p.N;
    // steps of the S loop: 64 columns; then the CTA's own slice
    const int s_steps = (p.d + 63) / 64;
    const int g_steps = do_grad ? 1 : 0;
    const int n_pad = (N_ + 15) & ~15;
    const int ptiles = N_ > 128 ? 2 : 1;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    constexpr uint32_t STAGE = BF_STAGE;
    const uint32_t w_smem = base + BF_W_OFF;

    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < SM_STAGES; ++s) {
            mbar_init(smem_u32(&bars.full[s]), 1);
            mbar_init(smem_u32(&bars.empty[s]), 1);
        }
        mbar_init(smem_u32(&bars.s_full), 1);
        mbar_init(smem_u32(&bars.w_full), SM_WORKERS);
        mbar_init(smem_u32(&bars.acc_full), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == SM_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_s)), "r"((uint32_t)TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    dep_release();
    dep_wait();

    if (warp == SM_PROD_WARP) {
        // ------------------------------ loads -----------------------------------------------------
        // Rows past B (N) and columns past d read as zeros.
        int stage = 0;
        uint32_t phase = 0;
        for (int t = 0; t < s_steps + g_steps; ++t) {
            if (!mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag)) break;
            const uint32_t full = smem_u32(&bars.full[stage]);
            const uint32_t dst = base + stage * STAGE;
            const int col = t < s_steps ? 64 * t : 64 * slice;
            if (elect_one()) {
                mbar_expect_tx(full, (uint32_t)(1 + ptiles) * TILE);
                tma_load_2d(dst, &mapQ, col, 0, full);
                tma_load_2d(dst + TILE, &mapP, col, 0, full);
                if (ptiles == 2) tma_load_2d(dst + 2 * TILE, &mapP, col, 128, full);
            }
            if (++stage == SM_STAGES) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == SM_MMA_WARP) {
        // ------------------------------ MMA issuer ------------------------------------------------
        const uint32_t idesc_s = instr_desc(n_pad, false, XROWS, false);
        const uint32_t idesc_dq = instr_desc(64, true, XROWS, false);    // A = W, K-major
        const uint32_t idesc_dp = instr_desc(64, true, XROWS, true);     // A = W^T: MN-major
        const int nchunks = (N_ + 63) / 64;
        bool ok = true;
        uint32_t q_tile = 0, p_tile = 0;       // the CTA's own slices as MN-major B operands
        {
            int stage = 0;
            uint32_t phase = 0;
            for (int t = 0; t < s_steps && ok; ++t) {
                ok = mbar_wait(smem_u32(&bars.full[stage]), phase, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t a = desc_lo(base + stage * STAGE, 0);
                const uint32_t b = desc_lo(base + stage * STAGE + TILE, 0);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        if (t == 0 && kk == 0) mma_ss<false, false>(tmem + COL_S, a, b, idesc_s);
                        else mma_ss<true, false>(tmem + COL_S, a + 2 * kk, b + 2 * kk, idesc_s);
                    }
                    tc_commit(smem_u32(&bars.empty[stage]));
                }
                if (++stage == SM_STAGES) { stage = 0; phase ^= 1u; }
            }
            if (ok && elect_one()) tc_commit(smem_u32(&bars.s_full));
            if (ok && do_grad) {
                ok = mbar_wait(smem_u32(&bars.full[stage]), phase, abort_flag);
                q_tile = base + stage * STAGE;
                p_tile = q_tile + TILE;
            }
        }
        if (ok && do_grad) ok = mbar_wait(smem_u32(&bars.w_full), 0, abort_flag);
        if (ok && do_grad) {
            tc_fence_after();
            if (elect_one()) {
                // dQ slice: contraction over passages, 64 per weight chunk
                bool first = true;
                for (int c = 0; c < nchunks; ++c) {
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const uint32_t a = desc_lo(w_smem + c * TILE, 0) + 2 * kk;
                        const uint32_t b = desc_lo(p_tile + c * (TILE / 2), 0) + 128 * kk;
                        if (first) mma_ss<false, false>(tmem + COL_DQ, a, b, idesc_dq);
                        else       mma_ss<true, false>(tmem + COL_DQ, a, b, idesc_dq);
                        first = false;
                    }
                }
                // dP slice: contraction over the 128 query rows; 128 passages per block
                for (int blk = 0; blk < ptiles; ++blk) {
                    first = true;
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) {
                        const uint32_t a = desc_lo(w_smem + 2 * blk * TILE, TILE) + 128 * kk;
                        const uint32_t b = desc_lo(q_tile, 0) + 128 * kk;
                        if (first) mma_ss<false, false>(tmem + COL_DP + 64 * blk, a, b, idesc_dp);
                        else       mma_ss<true, false>(tmem + COL_DP + 64 * blk, a, b, idesc_dp);
                        first = false;
                    }
                }
                tc_commit(smem_u32(&bars.acc_full));
            }
        }
    } else {
        // ------------------------------ workers ---------------------------------------------------
        const int wt = threadIdx.x - 32 * SM_FIRST_WORKER;      // 0 .. 255
        const int q = warp & 3;                                  // tensor-memory lane quarter
        const int half = (warp - SM_FIRST_WORKER) >> 2;          // column half of S / of a slice
        const int i = 32 * q + lane;                             // row of S, of dQ, of a dP block
        const uint32_t lane_addr = (uint32_t)(32 * q) << 16;
        bool ok = true;
        ok = ok && mbar_wait(smem_u32(&bars.s_full), 0, abort_flag);
        if (workers_all(ok)) {
            tc_fence_after();
            // ------------------------------ softmax of row i over this half's columns -------------
            // One pass over the row keeps a running (max, sum); the special columns of a block of
            // 32 (past N, the masked pair, the positive) are patched after the plain arithmetic.
            const int j0 = half * 128;
            constexpr int nblk = 4;                               // blocks of 32 columns per half
            const int32_t r_i = i < B_ ? p.pos_idx[i] : -1;
            int flags = 0;
            if (i < B_) {
                if (r_i < 0 || r_i >= p.N) flags = GC_DEV_POS_RANGE;
                else if (p.mask_mode == GC_MASK_SELF && r_i == i + p.mask_shift) flags = GC_DEV_POS_MASKED;
            }
            const int pos = flags ? -1 : r_i;
            const int masked = p.mask_mode == GC_MASK_SELF ? i + p.mask_shift : -1;
            float lse2, pos2 = 0.f, lse_nat = 0.f, m_row = 0.f, lnsum_row = 0.f;
            if (p.op == GC_OP_BWD) {
                lse2 = p.row_lse_in[i < B_ ? i : 0] * 1.4426950408889634f;
            } else {
                // The running maximum is kept in units of <q, p> (unscaled), so that the row's
                // logsumexp and its positive logit come out of the same product with 1/tau:
                // lse_i - S_{i,r_i} is exactly 0 when the positive is the only column.
                float m = -INFINITY, sum = 0.f, lnsum = 0.f;
                for (int cb = 0; cb < nblk; ++cb) {
                    const int jb = j0 + 32 * cb;
                    if (jb >= N_) break;
                    float sr[32];
                    load_s(tmem + lane_addr, jb, sr);
                    if ((unsigned)(pos - jb) < 32u) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) if (e == pos - jb) pos2 = sr[e];
                    }
                    if ((unsigned)(masked - jb) < 32u) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) if (e == masked - jb) sr[e] = -INFINITY;
                    }
                    if (jb + 32 > N_) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) if (jb + e >= N_) sr[e] = -INFINITY;
                    }
                    float bm = sr[0];
#pragma unroll
                    for (int e = 1; e < 32; ++e) bm = fmaxf(bm, sr[e]);
                    const float mn = fmaxf(m, bm);
                    const float ref = mn == -INFINITY ? 0.f : mn;
                    float part = 0.f;      // (s - max) first: the largest term is exactly 2^0
#pragma unroll
                    for (int e = 0; e < 32; ++e) part += ex2((sr[e] - ref) * p.scale2);
                    sum = sum * ex2((m - ref) * p.scale2) + part;
                    m = mn;
                }
                x_max[half][i] = m;
                x_sum[half][i] = sum;
                x_pos[half][i] = pos2;
                workers_sync();
                const float m0 = x_max[0][i], m1 = x_max[1][i];
                m = fmaxf(m0, m1);
                const float mref = m == -INFINITY ? 0.f : m;                // all columns masked
                sum = x_sum[0][i] * ex2((m0 - mref) * p.scale2) +
                      x_sum[1][i] * ex2((m1 - mref) * p.scale2);
                pos2 = x_pos[0][i] + x_pos[1][i];                 // the other half holds 0
                const float lg = log2f(sum);          // once per row: the accurate one
                lse2 = m * p.scale2 + lg;
                lnsum = lg * 0.6931471805599453f;
                lse_nat = m * p.inv_tau + lnsum;
                m_row = m;
                lnsum_row = lnsum;
            }
            // ------------------------------ outputs of the forward (CTA 0) ------------------------
            if (slice == 0) {
                float term = 0.f;
                if (half == 0 && i < B_) {
                    if (p.op != GC_OP_BWD) {
                        const float pl = pos2 * p.inv_tau;
                        p.row_lse[i] = lse_nat;
                        if (p.pos_logit) p.pos_logit[i] = pl;
                        term = (m_row - pos2) * p.inv_tau + lnsum_row;   // no cancellation of two roundings
                    }
                    if (flags && p.dev_status) atomicOr(p.dev_status, flags);
                }
                if (p.op != GC_OP_BWD) {
                    for (int o = 16; o > 0; o >>= 1) term += __shfl_xor_sync(0xffffffffu, term, o);
                    if (half == 0 && lane == 0) loss_part[q] = term;
                    workers_sync();
                    if (wt == 0)
                        *p.loss = (((loss_part[0] + loss_part[1]) + loss_part[2]) + loss_part[3]) *
                                  p.inv_mean;
                }
            }
            if (do_grad) {
                // ------------------------------ weights as MMA operands ---------------------------
                // chunk c = 64 columns; element (i, j) in 16-byte piece ((j % 64) / 8) ^ (i % 8) of
                // row i: a K-major A operand for dQ and, read by columns, an MN-major one for dP.
                // Rows past B get lse = +inf: all their weights are 0.
                const float neg_lse = i < B_ ? -lse2 : -INFINITY;
                const int pos_w = i < B_ ? pos : -1;
                for (int cb = 0; cb < nblk; ++cb) {
                    const int jb = j0 + 32 * cb;                  // 4 pieces of 8 columns
                    float w[32];
                    if (jb < N_) {
                        load_s(tmem + lane_addr, jb, w);
#pragma unroll
                        for (int e = 0; e < 32; ++e) w[e] = ex2(fmaf(w[e], p.scale2, neg_lse));
                        if ((unsigned)(masked - jb) < 32u) {
#pragma unroll
                            for (int e = 0; e < 32; ++e) if (e == masked - jb) w[e] = 0.f;
                        }
                        if ((unsigned)(pos_w - jb) < 32u) {
#pragma unroll
                            for (int e = 0; e < 32; ++e) if (e == pos_w - jb) w[e] -= 1.f;
                        }
                        if (jb + 32 > N_) {
#pragma unroll
                            for (int e = 0; e < 32; ++e) if (jb + e >= N_) w[e] = 0.f;
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) w[e] = 0.f;
                    }
                    const uint32_t row = w_smem + (uint32_t)(jb >> 6) * TILE + i * 128;
#pragma unroll
                    for (int pc = 0; pc < 4; ++pc) {
                        const int piece = ((jb & 63) >> 3) + pc;
                        const uint32_t dst = row + (uint32_t)((piece ^ (i & 7)) << 4);
                        uint32_t hi[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) hi[e] = pack_bf16(w[8 * pc + 2 * e], w[8 * pc + 2 * e + 1]);
                        sts128u(dst, hi);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&bars.w_full));
                // ------------------------------ gradients out -------------------------------------
                // A warp's 32 x 32 block goes through a 4 KB buffer (two per warp, over the
                // drained pipeline buffers) and leaves with one bulk tensor store, which clips it
                // at the matrix's last row and column.
                if (mbar_wait(smem_u32(&bars.acc_full), 0, abort_flag)) {
                    tc_fence_after();
                    const int col = 64 * slice + 32 * half;
                    const uint32_t slot = base + (uint32_t)(warp - SM_FIRST_WORKER) * 8192u;
                    int n = 0;
                    for (int blk = 0; blk < 1 + ptiles; ++blk) {       // dQ, dP rows 0.., dP rows 128..
                        const int rows = blk == 0 ? p.B : p.N;
                        const int row0 = (blk == 0 ? 0 : 128 * (blk - 1)) + 32 * q;
                        const bool have = blk == 0 ? p.dQ != nullptr : p.dP != nullptr;
                        if (!have || row0 >= rows || col >= p.d) continue;
                        uint32_t v[32];
                        tmem_ld32(tmem + lane_addr + (blk == 0 ? COL_DQ : COL_DP + 64 * (blk - 1)) +
                                      32 * half, v);
                        if (n >= 2) {   // the store issued two blocks ago has read this buffer
                            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                            __syncwarp();
                        }
                        tmem_ld_wait();
                        const uint32_t buf = slot + (uint32_t)(n & 1) * 4096u;
                        stage_block(buf, v, p.out_scale, lane);
                        __syncwarp();
                        if (lane == 0) tma_store_3d(blk == 0 ? &mapDQ : &mapDP, buf, col, row0, 0);
                        ++n;
                    }
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
                    __syncwarp();
                }
            }
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
    if (warp == SM_MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     ::"r"(tmem), "r"((uint32_t)TMEM_COLS) : "memory");
    }
}

cudaError_t launch_small_bf16(const CUtensorMap& mq, const CUtensorMap& mp, const CUtensorMap& mdq,
                              const CUtensorMap& mdp, const SmallParams& p, dim3 grid,
                              cudaStream_t st) {
    static bool configured_on[64] = {false};      // the attribute belongs to (kernel, device)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured_on[dev]) {
        cudaError_t e = cudaFuncSetAttribute(small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)SM_DYN_SMEM);
        if (e != cudaSuccess) return e;
        configured_on[dev] = true;
    }
    return launch_chained(small_kernel, grid, SM_THREADS, SM_DYN_SMEM, 1, st, mq, mp, mdq, mdp, p);
}

}  // namespace

// GRADCACHE_PLAN=sweeps in the environment (read at every call) keeps every problem on the sweep
// kernels (or the FMA tiles): a diagnostic switch, so that small shapes can still exercise the
// kernels that large ones run.
static bool small_plans_enabled() {
    const char* e = getenv("GRADCACHE_PLAN");
    return !(e && strcmp(e, "sweeps") == 0);
}

bool small_applicable(int64_t B, int64_t N, int d, int dtype) {
    if (!small_plans_enabled()) return false;
    if (B > 128 || d % 8 != 0 || d > 1024) return false;
    return dtype == GC_BF16 ? N <= 256 : N <= 128;
}

// op: GC_OP_FWD (loss, row_lse, pos_logit), GC_OP_BWD (dQ, dP from row_lse_in) or GC_OP_BUILD.
cudaError_t launch_small(int op, const Problem& pr, const float* row_lse_in, float* loss,
                         float* row_lse, float* pos_logit, float* dQ, int64_t lddq, float* dP,
                         int64_t lddp, int* dev_status, cudaStream_t st) {
    if (pr.dtype == GC_F32)
        return launch_small_f32(op, pr, row_lse_in, loss, row_lse, pos_logit, dQ, lddq, dP, lddp, dev_status,
                                st);
    CUtensorMap mq, mp;
    if (!make_map(&mq, pr.Q, pr.B, pr.d, pr.ldq, 128) || !make_map(&mp, pr.P, pr.N, pr.d, pr.ldp, 128))
        return cudaErrorInvalidValue;
    // gradient outputs as [1][rows][d] for the epilogue's bulk tensor stores; a missing output
    // (gc_loss_fwd; gc_loss_bwd with one of the two) gets a map of the other, never written
    CUtensorMap mdq = mq, mdp = mp;
    if (dQ && !make_out_map(&mdq, dQ, pr.B, pr.d, lddq, 1)) return cudaErrorInvalidValue;
    if (dP && !make_out_map(&mdp, dP, pr.N, pr.d, lddp, 1)) return cudaErrorInvalidValue;
    SmallParams p{};
    p.B = (int)pr.B; p.N = (int)pr.N; p.d = pr.d;
    p.op = op;
    p.mask_mode = pr.mask_mode;
    p.mask_shift = (int)pr.mask_shift;
    p.scale2 = 1.4426950408889634f / pr.tau;
    p.inv_tau = 1.f / pr.tau;
    const float batch = (float)(pr.b_total > 0 ? pr.b_total : pr.B);
    p.out_scale = 1.f / (batch * pr.tau);
    p.inv_mean = 1.f / batch;
    p.pos_idx = pr.pos_idx;
    p.row_lse_in = row_lse_in;
    p.loss = loss; p.row_lse = row_lse; p.pos_logit = pos_logit;
    p.dQ = dQ; p.lddq = lddq; p.dP = dP; p.lddp = lddp;
    p.dev_status = dev_status;
    const dim3 grid(op == GC_OP_FWD ? 1u : (unsigned)((pr.d + 63) / 64));
    return launch_small_bf16(mq, mp, mdq, mdp, p, grid, st);
}

// Batches of several tiles that the strip plan takes whatever their width: fp32 while the planes of
// partial sums of tile pairs of 128 x 128 would stay within 2 GiB (beyond, the FMA tiles serve: they need
// no memory), bf16 of few tile pairs of 128 x 256.
bool small_tiled_applicable(int64_t B, int64_t N, int d, int dtype) {
    if (!small_plans_enabled()) return false;
    if (d % 8 != 0 || d > 4096 || small_applicable(B, N, d, dtype)) return false;
    if (B > (1 << 24) || N > (1 << 24)) return false;
    const int64_t xt = (B + 127) / 128, yt = dtype == GC_F32 ? (N + 127) / 128 : (N + 255) / 256;
    if (dtype == GC_F32) {
        const double plane_bytes = ((double)yt * (double)B + (double)xt * (double)N) * d * 4.0;
        return xt <= 65535 && yt <= 65535 && plane_bytes <= 2147483648.0;
    }
    return dtype == GC_BF16 && xt * yt <= 64 && xt * yt * ((d + 63) / 64) <= 2 * sm_count();
}

}  // namespace gc
