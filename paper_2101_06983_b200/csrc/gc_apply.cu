// Step 3 of Gradient Cache for a linear encoder f(s) = W s (Section 3.3, Eq. 8; Eq. 9 for g):
// the representation gradients of one sub-batch, read from the cache, times the sub-batch's
// encoder inputs,
//
//     dW[a][b] (+)= sum_i U[i][a] X[i][b]          U: rows x d fp32 (cache slice), X: rows x d_in bf16
//
// The cache is fp32 and the tensor cores take bf16, so every u is used as two bf16 terms,
// hi = rn(u) and lo = rn(u - hi), whose sum misses u by at most 2^-17 |u|; both terms accumulate
// into the same fp32 accumulator.
//
// A CTA pair owns a tile of 256 output rows (columns of U) x 256 output columns (columns of X) and
// one part of the contraction range (the rows of the sub-batch), in blocks of 64 rows:
//   16 converter warps read U straight from global memory (two blocks ahead, in registers), form hi and
//                   lo and write them as two MN-major A operands in the 128-byte swizzle; they run the
//                   epilogue too
//   producer warp   bulk tensor loads of X, an MN-major B operand as it lies in memory
//   MMA warp        the leader's: 8 instructions of M = 256, N = 256 per block
// With one part the tile goes to dW; otherwise each part is a plane of the workspace and a second
// kernel adds the planes in order.  No atomics, deterministic, every mbarrier wait is bounded.
//
// What bounds it at 4096 x 768 x 768 (9 tiles x 8 parts, 18.8 us): reading U and X once (3 us from
// memory, 3.6 until the first product), a block each 0.72 us against 0.55 of products, 3.8 us from the
// last product to the stored planes, 5 us for the second launch.  Sixteen converter warps, a float4
// of a row per lane: with eight, and two float4 per lane, a block took 0.85-1.1 us.  Before, one launch
// of clusters of single CTAs that exchanged their parts through shared memory: 22.8 us (32768 x 384 x
// 384: 84 / 35, 8192 x 128 x 384: 31 / 15, 4096 x 2048 x 2048: 93 / 50).
#include <cuda_bf16.h>

#include "tc_common.cuh"

namespace gc {

namespace {

constexpr int AP_KB = 64;                      // contraction rows per stage
constexpr int AP_CONV = 16;                    // converter / epilogue warps
constexpr int AP_PROD_WARP = AP_CONV;
constexpr int AP_MMA_WARP = AP_CONV + 1;
constexpr int AP_THREADS = 32 * (AP_CONV + 2);
constexpr int AP_STAGES = 3;
constexpr int AP_AHEAD = 3;                    // blocks of U held in registers
constexpr uint32_t AP_ATOM = 64 * 128;         // 64 contraction rows x 64 columns of bf16
constexpr uint32_t AP_STAGE = 6 * AP_ATOM;     // hi (2 atoms), lo (2 atoms), X (2 atoms)
constexpr size_t AP_SMEM = 1024 + (size_t)AP_STAGES * AP_STAGE + AP_CONV * 4096;
constexpr int AP_MAX_PARTS = 32;

static_assert(AP_SMEM <= SMEM_LIMIT - 1024, "shared memory budget");

struct ApplyParams {
    const float* U;
    int64_t ldu, rows;
    int d, d_in;
    int tiles_n, tiles;           // column tiles, all tiles
    int parts, kblocks;
    int add;                      // one part: add to dW
    int* dev_status;
};

struct __align__(16) ApplyBars {
    uint64_t signal[2 * AP_CONV];         // what the second CTA's converters send along with their signal
    uint64_t full[AP_STAGES];             // leader: X of both CTAs
    uint64_t conv[AP_STAGES];             // leader: hi and lo of both CTAs
    uint64_t empty[AP_STAGES];
    uint64_t acc_full;
    uint64_t acc_free, acc_free_peer;
};

__global__ void __launch_bounds__(AP_THREADS, 1)
apply_kernel(const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapO,
             const ApplyParams p) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ ApplyBars bars;
    __shared__ uint32_t tmem_s;
    __shared__ int abort_s;
    volatile int* abort_flag = &abort_s;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const uint32_t smem = (smem_u32(smem_raw) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < AP_STAGES; ++s) {
            mbar_init(smem_u32(&bars.full[s]), 1);
            mbar_init(smem_u32(&bars.conv[s]), AP_CONV);
            mbar_init(smem_u32(&bars.empty[s]), 1);
        }
        mbar_init(smem_u32(&bars.acc_full), 1);
        mbar_init(smem_u32(&bars.acc_free), AP_CONV);
        mbar_init(smem_u32(&bars.acc_free_peer), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == AP_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_s)), "r"(256u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after();
    const uint32_t tmem = tmem_s;
    dep_release();
    dep_wait();

    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    const int units = p.tiles * p.parts;           // unit: (part, tile), tiles fastest
    struct Unit { int m0, n0, bw, part, kb, kb_end; };
    auto unit_at = [&](int u) {
        Unit t;
        t.part = u / p.tiles;
        const int tile = u - t.part * p.tiles;
        t.m0 = tile / p.tiles_n * 256 + (int)rank * 128;
        t.n0 = tile % p.tiles_n * 256;
        t.bw = p.d_in - t.n0 <= 128 ? 64 : 128;    // columns of X this CTA loads
        t.kb = (int)((int64_t)p.kblocks * t.part / p.parts);
        t.kb_end = (int)((int64_t)p.kblocks * (t.part + 1) / p.parts);
        return t;
    };

    if (warp == AP_PROD_WARP) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int u = pair; u < units && ok; u += pairs) {
            const Unit t = unit_at(u);
            for (int kb = t.kb; kb < t.kb_end; ++kb) {
                ok = mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag);
                if (!ok) break;
                const uint32_t full = smem_u32(&bars.full[stage]), full_leader = mapa_u32(full, 0);
                const uint32_t dst = smem + stage * AP_STAGE + 4 * AP_ATOM;
                const int n = t.n0 + (int)rank * t.bw;
                if (elect_one()) {
                    if (rank == 0) mbar_expect_tx(full, 2u * 128u * (uint32_t)t.bw);
                    tma_load_2d_pair(dst, &mapX, n, kb * AP_KB, full_leader);
                    if (t.bw == 128) tma_load_2d_pair(dst + AP_ATOM, &mapX, n + 64, kb * AP_KB, full_leader);
                }
                if (++stage == AP_STAGES) { stage = 0; phase ^= 1u; }
            }
        }
        // the last commits that give stages back, from the leader into both CTAs, have arrived
        for (int n = 0; n < AP_STAGES && ok; ++n) {
            ok = mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag);
            if (++stage == AP_STAGES) { stage = 0; phase ^= 1u; }
        }
    } else if (warp == AP_MMA_WARP) {
        int n_unit = 0;
        bool ok = true;
        if (rank == 0) {
            int stage = 0;
            uint32_t phase = 0;
            for (int u = pair; u < units && ok; u += pairs, ++n_unit) {
                const Unit t = unit_at(u);
                const uint32_t idesc = instr_desc(2 * t.bw, true, 256, true);
                const uint32_t par = ((uint32_t)n_unit & 1u) ^ 1u;
                ok = mbar_wait(smem_u32(&bars.acc_free), par, abort_flag) &&
                     mbar_wait(smem_u32(&bars.acc_free_peer), par, abort_flag);
                if (!ok) break;
                tc_fence_after();
                for (int kb = t.kb; kb < t.kb_end; ++kb) {
                    ok = mbar_wait(smem_u32(&bars.full[stage]), phase, abort_flag) &&
                         mbar_wait(smem_u32(&bars.conv[stage]), phase, abort_flag);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t a = desc_lo(smem + stage * AP_STAGE, AP_ATOM);
                    const uint32_t b = desc_lo(smem + stage * AP_STAGE + 4 * AP_ATOM, AP_ATOM);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < AP_KB / 16; ++k) {
                            if (k == 0 && kb == t.kb) mma_ss<false, true>(tmem, a, b, idesc);
                            else mma_ss<true, true>(tmem, a + 128 * k, b + 128 * k, idesc);
                            mma_ss<true, true>(tmem, a + (2 * AP_ATOM >> 4) + 128 * k, b + 128 * k, idesc);
                        }
                        tc_commit_pair(smem_u32(&bars.empty[stage]));
                        if (kb == t.kb_end - 1) tc_commit_pair(smem_u32(&bars.acc_full));
                    }
                    if (++stage == AP_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
        } else {
            // what the leader waits for: every unit's "accumulator read" but the last one's
            for (int u = pair; u + pairs < units && ok; u += pairs, ++n_unit) {
                ok = mbar_wait(smem_u32(&bars.acc_free), (uint32_t)n_unit & 1u, abort_flag);
                if (ok && elect_one()) mbar_arrive_cluster(mapa_u32(smem_u32(&bars.acc_free_peer), 0));
            }
        }
    } else {
        // Piece of a block: one contraction row x 4 columns of U, one 16-byte load in, one 8-byte store
        // per term out.  A warp takes whole rows of 128 columns: loads are contiguous, and the stores of
        // a half warp fall on distinct banks.
        constexpr int ROWS = AP_KB / AP_CONV;      // of a warp: warp, warp + 16, ...
        const int col = lane * 4, row0 = warp;
        const int q = warp & 3, group = warp >> 2; // epilogue: lane quarter, quarter of the columns
        // the same place in every row and stage: 16 rows further is the same phase of the swizzle
        const uint32_t place = (uint32_t)(col >> 6) * AP_ATOM + (uint32_t)row0 * 128u +
                               (uint32_t)((((col & 63) >> 3) ^ (row0 & 7)) << 4) + (uint32_t)(col & 4) * 2u;
        const int64_t step = (int64_t)AP_CONV * p.ldu;
        const uint32_t slot = smem + AP_STAGES * AP_STAGE + (uint32_t)warp * 4096u;
        int stage = 0, n_unit = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int u = pair; u < units && ok; u += pairs, ++n_unit) {
            const Unit t = unit_at(u);
            const bool live = t.m0 + col < p.d;    // d is a multiple of 8
            const float* src = p.U + (live ? t.m0 + col : 0) + ((int64_t)t.kb * AP_KB + row0) * p.ldu;
            float4 x[AP_AHEAD][ROWS];
            // block kb; called once for every block in order
            auto fetch = [&](float4 (&v)[ROWS], int kb) {
                const int64_t left = p.rows - (int64_t)kb * AP_KB;         // rows from the block's first on
                if (kb < t.kb_end && live && left >= AP_KB) {
#pragma unroll
                    for (int i = 0; i < ROWS; ++i) v[i] = __ldcg(reinterpret_cast<const float4*>(src + i * step));
                } else {
#pragma unroll
                    for (int i = 0; i < ROWS; ++i) {
                        const bool in = kb < t.kb_end && live && row0 + AP_CONV * i < left;
                        v[i] = in ? __ldcg(reinterpret_cast<const float4*>(src + i * step))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
                src += (int64_t)AP_KB * p.ldu;
            };
            auto convert = [&](const float4 (&v)[ROWS]) {
                const uint32_t dst0 = smem + stage * AP_STAGE + place;
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    const float f[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
                    uint32_t hi[2], lo[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
                        hi[e] = *reinterpret_cast<const uint32_t*>(&h);
                        const __nv_bfloat162 g =
                            __floats2bfloat162_rn(f[2 * e] - __uint_as_float(hi[e] << 16),
                                                  f[2 * e + 1] - __uint_as_float(hi[e] & 0xffff0000u));
                        lo[e] = *reinterpret_cast<const uint32_t*>(&g);
                    }
                    const uint32_t dst = dst0 + (uint32_t)i * (AP_CONV * 128u);
                    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst), "r"(hi[0]), "r"(hi[1]) : "memory");
                    asm volatile("st.shared.v2.b32 [%0], {%1, %2};"
                                 ::"r"(dst + 2 * AP_ATOM), "r"(lo[0]), "r"(lo[1]) : "memory");
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                // a remote arrival would stall the warp; 16 bytes that the leader's barrier counts do not
                if (lane == 0) {
                    const uint32_t bar = smem_u32(&bars.conv[stage]);
                    const uint32_t box = smem_u32(&bars.signal[2 * warp]);
                    if (rank != 0)
                        asm volatile(
                            "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes "
                            "[%0], [%1], 16, [%2];"
                            ::"r"(mapa_u32(box, 0)), "r"(box), "r"(mapa_u32(bar, 0)) : "memory");
                    else if (warp == 0) mbar_expect_tx(bar, 16 * AP_CONV);
                    else                mbar_arrive(bar);
                }
            };
#pragma unroll
            for (int a = 0; a < AP_AHEAD; ++a) fetch(x[a], t.kb + a);
            for (int kb = t.kb; kb < t.kb_end && ok; kb += AP_AHEAD) {
#pragma unroll
                for (int a = 0; a < AP_AHEAD; ++a) {
                    if (kb + a >= t.kb_end) break;
                    ok = mbar_wait(smem_u32(&bars.empty[stage]), phase ^ 1u, abort_flag);
                    if (!ok) break;
                    convert(x[a]);
                    fetch(x[a], kb + a + AP_AHEAD);
                    if (++stage == AP_STAGES) { stage = 0; phase ^= 1u; }
                }
            }
            if (!ok) break;
            ok = mbar_wait(smem_u32(&bars.acc_full), (uint32_t)n_unit & 1u, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t src_t = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(group * (t.bw / 2));
            const int r_out = t.m0 + 32 * q;
            for (int cb = 0; 32 * cb < t.bw / 2; ++cb) {
                uint32_t v[32];
                tmem_ld32(src_t + 32 * cb, v);
                if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
                tmem_ld_wait();
                stage_block(slot, v, 1.f, lane);
                __syncwarp();
                const int c_out = t.n0 + group * (t.bw / 2) + 32 * cb;
                if (lane == 0 && r_out < p.d && c_out < p.d_in) {
                    if (p.add) {
                        asm volatile(
                            "cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.bulk_group "
                            "[%0, {%2, %3, %4}], [%1];"
                            ::"l"(reinterpret_cast<uint64_t>(&mapO)), "r"(slot), "r"(c_out), "r"(r_out), "r"(0)
                            : "memory");
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                    } else {
                        tma_store_3d(&mapO, slot, c_out, r_out, p.parts > 1 ? t.part : 0);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&bars.acc_free));
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
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
    cluster_meet();       // every load, signal, product, commit and arrival between the CTAs has been waited for
    if (warp == AP_MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;"
                     ::"r"(tmem), "r"(256u) : "memory");
    }
}

// dW (+)= sum of the planes, in order.
__global__ void __launch_bounds__(256)
apply_reduce_kernel(const float4* planes, int parts, int64_t plane, int n4,
                    float* __restrict__ dW, int64_t lddw, int add) {
    dep_release();
    dep_wait();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < plane;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / n4;
        float4* dst = reinterpret_cast<float4*>(dW + r * lddw) + (e - r * n4);
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        if (add) s = *dst;
#pragma unroll 8
        for (int g = 0; g < parts; ++g) {
            const float4 v = __ldcg(planes + g * plane + e);
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *dst = s;
    }
}

struct ApplyPlan {
    int tiles_m, tiles_n, parts, kblocks;
};

// As many parts as pairs are left per tile (one wave), up to AP_MAX_PARTS and one block each: the
// products of a second wave would cost more than the planes of a part save.
int most_parts(int64_t tiles) {
    const int64_t per = sm_count() / 2 / tiles;
    return per < 1 ? 1 : per > AP_MAX_PARTS ? AP_MAX_PARTS : (int)per;
}
size_t plane_bytes(int d, int d_in) { return (size_t)d * (size_t)d_in * 4; }
// ws_bytes: of a workspace that may hold fewer planes than that
ApplyPlan make_apply_plan(int64_t rows, int d, int d_in, size_t ws_bytes) {
    ApplyPlan pl{};
    pl.tiles_m = (d + 255) / 256;
    pl.tiles_n = (d_in + 255) / 256;
    pl.kblocks = (int)((rows + AP_KB - 1) / AP_KB);
    pl.parts = most_parts((int64_t)pl.tiles_m * pl.tiles_n);
    if (pl.parts > pl.kblocks) pl.parts = pl.kblocks;
    const size_t room = ws_bytes / plane_bytes(d, d_in);
    if ((size_t)pl.parts > room) pl.parts = room < 2 ? 1 : (int)room;
    return pl;
}

bool apply_shape_ok(int64_t rows, int d, int d_in) {
    return rows > 0 && rows <= ((int64_t)1 << 30) && d > 0 && d_in > 0 && d <= (1 << 20);
}

// The planes of the most parts these widths can take, whatever the rows.
size_t apply_ws(int d, int d_in) {
    const int parts = most_parts((int64_t)((d + 255) / 256) * ((d_in + 255) / 256));
    if (parts == 1) return 256;
    return ((size_t)parts * plane_bytes(d, d_in) + 255) & ~(size_t)255;
}

}  // namespace

}  // namespace gc

using namespace gc;

extern "C" {

size_t gc_cache_apply_workspace_bytes(int64_t rows, int d, int d_in) {
    if (!apply_shape_ok(rows, d, d_in) || d % 8 != 0 || d_in % 64 != 0 || d_in > 4096) return 0;
    return apply_ws(d, d_in);
}

int gc_cache_apply(const float* U, int64_t ldu, const void* X, int64_t ldx, int64_t rows, int d,
                   int d_in, int x_dtype, float* dW, int64_t lddw, int accumulate, void* ws,
                   size_t ws_bytes, int* dev_status, void* cuda_stream) {
    if (!U || !X || !dW) return GC_ERR_NULL;
    if (x_dtype != GC_BF16) return GC_ERR_DTYPE;
    if (!apply_shape_ok(rows, d, d_in) || ldu < d || ldx < d_in || lddw < d_in) return GC_ERR_SHAPE;
    if (d % 8 != 0 || d_in % 64 != 0 || d_in > 4096) return GC_ERR_LIMIT;
    if (((uintptr_t)U & 15) || ((uintptr_t)X & 15) || ((uintptr_t)dW & 15) || (ldu * 4) % 16 ||
        (ldx * 2) % 16 || (lddw * 4) % 16)
        return GC_ERR_ALIGN;
    if (!ws || ((uintptr_t)ws & 255) || ws_bytes < 256) return GC_ERR_WORKSPACE;
    int dev = 0, major = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) {
        cudaGetLastError();
        return GC_ERR_CUDA;
    }
    if (major != 10) return GC_ERR_ARCH;
    if (dev < 0 || dev >= 64) return GC_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const ApplyPlan pl = make_apply_plan(rows, d, d_in, ws_bytes);
    float* planes = static_cast<float*>(ws);
    CUtensorMap mx, mo;
    if (!make_map(&mx, X, rows, d_in, ldx, AP_KB) ||
        !(pl.parts > 1 ? make_out_map(&mo, planes, d, d_in, d_in, pl.parts)
                       : make_out_map(&mo, dW, d, d_in, lddw, 1)))
        return GC_ERR_CUDA;
    ApplyParams p{};
    p.U = U; p.ldu = ldu; p.rows = rows; p.d = d; p.d_in = d_in;
    p.tiles_n = pl.tiles_n; p.tiles = pl.tiles_m * pl.tiles_n;
    p.parts = pl.parts; p.kblocks = pl.kblocks;
    p.add = pl.parts == 1 && accumulate;
    p.dev_status = dev_status;

    static bool configured_on[64] = {false};      // the attribute belongs to (kernel, device)
    if (!configured_on[dev]) {
        if (cudaFuncSetAttribute(apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)AP_SMEM) != cudaSuccess) {
            cudaGetLastError();
            return GC_ERR_CUDA;
        }
        configured_on[dev] = true;
    }
    const int64_t units = (int64_t)p.tiles * p.parts, pairs = sm_count() / 2;
    cudaError_t e = launch_chained(apply_kernel, dim3(2u * (unsigned)(units < pairs ? units : pairs)),
                                   AP_THREADS, AP_SMEM, 2, st, mx, mo, p);
    if (e == cudaSuccess && pl.parts > 1) {
        const int64_t plane = (int64_t)d * (d_in / 4);
        const int64_t blocks = (plane + 255) / 256, most = 8 * (int64_t)sm_count();
        e = launch_chained(apply_reduce_kernel, dim3((unsigned)(blocks < most ? blocks : most)), 256, 0, 1,
                           st, reinterpret_cast<const float4*>(planes), pl.parts, plane, d_in / 4, dW, lddw,
                           accumulate ? 1 : 0);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return GC_ERR_CUDA;
    }
    return GC_OK;
}

}  // extern "C"
