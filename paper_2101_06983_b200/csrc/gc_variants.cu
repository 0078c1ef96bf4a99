// Loss variants around the Step 2 sweeps (Section 3.3: the loss on the stored representations may
// vary; the paper leaves its derivative to automatic differentiation).  Two of them need nothing
// from the sweeps but their inputs and outputs:
//
//   cosine similarity    S_ij = <q_i/|q_i|, p_j/|p_j|> / tau.  gc_row_normalize forms the unit rows
//                        the sweeps then see; gc_cosine_bwd takes the gradient with respect to the
//                        unit rows back through the normalisation, dx = (g - n <n, g>) / |x|.
//   learnable tau        dL/dtau = -(1/tau) sum_ij G_ij S_ij = -(1/tau) sum_i <q_i, dQ_i>, because
//                        <q_i, dQ_i> = sum_j G_ij <q_i, p_j> / tau (Eq. 5).  gc_dtau reduces the
//                        cache rows against the rows they belong to, in a fixed order.
//
// All three are bound by HBM traffic, or by launch and load latency for small batches: one warp per row,
// which may hold its pieces in registers, fp32 arithmetic, launched early (programmatic dependent launch).
#include <cuda_bf16.h>
#include <math.h>

#include "gc_internal.h"

namespace gc {
namespace {

__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// element k .. k + 3 of a row as floats (d is a multiple of 4; rows start on 16-byte boundaries)
template <bool BF16>
__device__ __forceinline__ float4 load4(const void* row, int k) {
    if (BF16) {
        const uint2 raw = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(row) + k);
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&raw.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return *reinterpret_cast<const float4*>(static_cast<const float*>(row) + k);
}
template <bool BF16>
__device__ __forceinline__ void store4(void* row, int k, float4 v) {
    if (BF16) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        uint2 raw;
        raw.x = *reinterpret_cast<uint32_t*>(&a);
        raw.y = *reinterpret_cast<uint32_t*>(&b);
        *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(row) + k) = raw;
    } else {
        *reinterpret_cast<float4*>(static_cast<float*>(row) + k) = v;
    }
}

// A lane's pieces of a row: 4 columns at 4 lane + 128 x, x < ROW_KEEP, held in registers; the rest is
// loaded each time it is asked for.  What is held saves the second read of a row and the wait for it, and costs
// warps per SM: see keep_normalize, keep_cosine; row_dot_kernel:
// none for bf16 and beyond 1024 columns, else 4 up to 512, 8.
template <int ROW_KEEP, typename Load>
struct RowPieces {
    float4 v[ROW_KEEP > 0 ? ROW_KEEP : 1];
    Load load;
    int d, k0;
    __device__ __forceinline__ RowPieces(Load l, int d_, int lane) : load(l), d(d_), k0(4 * lane) {
#pragma unroll
        for (int x = 0; x < ROW_KEEP; ++x)
            if (k0 + 128 * x < d) v[x] = load(k0 + 128 * x);
    }
};
template <int KEEP, typename Load>
__device__ __forceinline__ RowPieces<KEEP, Load> row_pieces(Load l, int d, int lane) {
    return RowPieces<KEEP, Load>(l, d, lane);
}
// f(k, piece of a, piece of b) for this lane's pieces in ascending order
template <int ROW_KEEP, typename A, typename B, typename F>
__device__ __forceinline__ void each_piece(const RowPieces<ROW_KEEP, A>& a, const RowPieces<ROW_KEEP, B>& b,
                                           F f) {
#pragma unroll
    for (int x = 0; x < ROW_KEEP; ++x)
        if (a.k0 + 128 * x < a.d) f(a.k0 + 128 * x, a.v[x], b.v[x]);
    for (int k = a.k0 + 128 * ROW_KEEP; k < a.d; k += 128) f(k, a.load(k), b.load(k));
}

template <bool BF16, int KEEP>
__global__ void __launch_bounds__(256)
row_normalize_kernel(const void* X, int64_t ldx, int64_t rows, int d,
                     void* __restrict__ Xn, int64_t ldxn, float* __restrict__ inv_norm) {
    const int lane = threadIdx.x & 31;
    const size_t es = BF16 ? 2 : 4;
    dep_release();
    dep_wait();
    for (int64_t i = blockIdx.x * 8 + (threadIdx.x >> 5); i < rows; i += (int64_t)gridDim.x * 8) {
        const char* src = static_cast<const char*>(X) + (size_t)i * (size_t)ldx * es;
        const auto x = row_pieces<KEEP>([&](int k) { return load4<BF16>(src, k); }, d, lane);
        float ss = 0.f;
        each_piece(x, x, [&](int, const float4& v, const float4&) {
            ss = fmaf(v.x, v.x, ss); ss = fmaf(v.y, v.y, ss);
            ss = fmaf(v.z, v.z, ss); ss = fmaf(v.w, v.w, ss);
        });
        ss = warp_sum(ss);
        const float inv = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;       // a zero row stays zero
        if (lane == 0) inv_norm[i] = inv;
        char* dst = static_cast<char*>(Xn) + (size_t)i * (size_t)ldxn * es;
        each_piece(x, x, [&](int k, const float4& v, const float4&) {
            store4<BF16>(dst, k, make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv));
        });
    }
}

// dX_i = inv_i (g_i - n_i <n_i, g_i>) with n_i = inv_i x_i formed in fp32 from the original row
template <bool BF16, int KEEP>
__global__ void __launch_bounds__(256)
cosine_bwd_kernel(const void* X, int64_t ldx, const float* inv_norm,
                  const float* G, int64_t ldg, int64_t rows, int d, float* dX, int64_t lddx) {
    const int lane = threadIdx.x & 31;
    const size_t es = BF16 ? 2 : 4;
    dep_release();
    dep_wait();
    for (int64_t i = blockIdx.x * 8 + (threadIdx.x >> 5); i < rows; i += (int64_t)gridDim.x * 8) {
        const char* src = static_cast<const char*>(X) + (size_t)i * (size_t)ldx * es;
        const float* g = G + i * ldg;
        const float inv = inv_norm[i];
        const auto xs = row_pieces<KEEP>([&](int k) { return load4<BF16>(src, k); }, d, lane);
        const auto gs = row_pieces<KEEP>([&](int k) { return *reinterpret_cast<const float4*>(g + k); }, d, lane);
        float dot = 0.f;
        each_piece(xs, gs, [&](int, const float4& x, const float4& gv) {
            dot = fmaf(x.x * inv, gv.x, dot); dot = fmaf(x.y * inv, gv.y, dot);
            dot = fmaf(x.z * inv, gv.z, dot); dot = fmaf(x.w * inv, gv.w, dot);
        });
        dot = warp_sum(dot);
        float* out = dX + i * lddx;
        each_piece(xs, gs, [&](int k, const float4& x, const float4& gv) {
            float4 o;
            o.x = inv * (gv.x - x.x * inv * dot); o.y = inv * (gv.y - x.y * inv * dot);
            o.z = inv * (gv.z - x.z * inv * dot); o.w = inv * (gv.w - x.w * inv * dot);
            *reinterpret_cast<float4*>(out + k) = o;
        });
    }
}

// row_dot[i] = <q_i, dQ_i>
template <bool BF16, int KEEP>
__global__ void __launch_bounds__(256)
row_dot_kernel(const void* Q, int64_t ldq, const float* dQ, int64_t lddq,
               int64_t rows, int d, float* __restrict__ row_dot) {
    const int lane = threadIdx.x & 31;
    const size_t es = BF16 ? 2 : 4;
    dep_release();
    dep_wait();
    for (int64_t i = blockIdx.x * 8 + (threadIdx.x >> 5); i < rows; i += (int64_t)gridDim.x * 8) {
        const char* src = static_cast<const char*>(Q) + (size_t)i * (size_t)ldq * es;
        const float* g = dQ + i * lddq;
        const auto xs = row_pieces<KEEP>([&](int k) { return load4<BF16>(src, k); }, d, lane);
        const auto gs = row_pieces<KEEP>([&](int k) { return *reinterpret_cast<const float4*>(g + k); }, d, lane);
        float dot = 0.f;
        each_piece(xs, gs, [&](int, const float4& x, const float4& gv) {
            dot = fmaf(x.x, gv.x, dot); dot = fmaf(x.y, gv.y, dot);
            dot = fmaf(x.z, gv.z, dot); dot = fmaf(x.w, gv.w, dot);
        });
        dot = warp_sum(dot);
        if (lane == 0) row_dot[i] = dot;
    }
}
// *out = scale * sum_i v[i]: one block, every thread a fixed strided share, then fixed trees
__global__ void __launch_bounds__(1024)
ordered_sum_kernel(const float* v, int64_t n, float scale, float* __restrict__ out) {
    __shared__ float part[32];
    dep_release();
    dep_wait();
    float s = 0.f;
#pragma unroll 8
    for (int64_t i = threadIdx.x; i < n; i += 1024) s += __ldcg(v + i);
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        float t = warp_sum(part[threadIdx.x]);
        if (threadIdx.x == 0) *out = t * scale;
    }
}

// Pieces to hold.  Measured, us per launch with none / 4 / 8 held (before they were: with none and not chained):
//   cosine_bwd  bf16  65536 x 128    13 / 17 / 41      4096 x 512     5.5 / 5.4 / 5.5    4096 x 1024  7.9 / 7.4 / 6.1
//                     32768 x 640    37 / 36 / 49      65536 x 2048   285 / 230 / 304
//               fp32  16384 x 256   6.4 / 5.7 / 11     32768 x 1024    59 / 56 / 53 and more for narrower, 1536 even
//   normalize   bf16  65536 x 768    35 / 39 / 38      32768 x 512    9.8 / 8.6 / 11     65536 x 2048 110 / 99 / 92
//               fp32  65536 x 512    49 / 44 / 44      65536 x 768     77 / 66 / 64
//   row_dot     bf16  32768 x 640    25 / 26 / 30      65536 x 2048   127 / 136 / 197    (one read of a row: nothing
//               fp32  65536 x 512    50 / 46 / 47      65536 x 1024    95 / 85 / 83       to save but the wait)
//                     32768 x 4096  169 / 176 / 230
int keep_cosine(int64_t rows, int d, int dtype) {
    if (dtype == GC_F32) return d <= 512 ? 4 : 8;
    return d <= 256 ? 0 : d > 768 && d <= 1536 && rows <= 4096 ? 8 : 4;
}
int keep_normalize(int64_t rows, int d, int dtype) {
    if (dtype == GC_BF16 && d <= 768 && rows * d > 20000000) return 0;      // neither rows nor unit rows stay in the L2
    return d <= 512 ? 4 : 8;
}
// go(kernel<BF16, KEEP>)
#define GC_KEEP_CALL(kernel, keep)                                                                               \
    (dtype == GC_F32 ? ((keep) == 4 ? go(kernel<false, 4>) : go(kernel<false, 8>))                               \
                     : ((keep) == 0 ? go(kernel<true, 0>) : (keep) == 4 ? go(kernel<true, 4>) : go(kernel<true, 8>)))

int grid_for(int64_t rows) {
    int64_t blocks = (rows + 7) / 8;
    const int cap = sm_count() * 8;
    return (int)(blocks > cap ? cap : blocks);
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

int check_rows(const void* X, int64_t ldx, int64_t rows, int d, int dtype) {
    if (!X) return GC_ERR_NULL;
    if (dtype != GC_F32 && dtype != GC_BF16) return GC_ERR_DTYPE;
    if (rows <= 0 || d <= 0 || ldx < d) return GC_ERR_SHAPE;
    const int es = dtype == GC_BF16 ? 2 : 4;
    if (!aligned16(X) || (ldx * es) % 16 != 0) return GC_ERR_ALIGN;
    if (d % 8 != 0) return GC_ERR_LIMIT;
    return GC_OK;
}
int check_f32(const float* X, int64_t ldx, int d) {
    if (!X) return GC_ERR_NULL;
    if (ldx < d) return GC_ERR_SHAPE;
    if (!aligned16(X) || (ldx * 4) % 16 != 0) return GC_ERR_ALIGN;
    return GC_OK;
}

}  // namespace
}  // namespace gc

using namespace gc;

extern "C" {

int gc_row_normalize(const void* X, int64_t ldx, int64_t rows, int d, int dtype, void* Xn,
                     int64_t ldxn, float* inv_norm, void* cuda_stream) {
    int rc = check_rows(X, ldx, rows, d, dtype);
    if (rc) return rc;
    if ((rc = check_rows(Xn, ldxn, rows, d, dtype))) return rc;
    if (!inv_norm) return GC_ERR_NULL;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e;
    auto go = [&](auto kernel) {
        return launch_chained(kernel, dim3(grid_for(rows)), 256, 0, 1, st, X, ldx, rows, d, Xn, ldxn,
                              inv_norm);
    };
    const int keep = keep_normalize(rows, d, dtype);
    e = GC_KEEP_CALL(row_normalize_kernel, keep);
    return e == cudaSuccess ? GC_OK : GC_ERR_CUDA;
}

int gc_cosine_bwd(const void* X, int64_t ldx, int64_t rows, int d, int dtype, const float* inv_norm,
                  const float* dXn, int64_t lddxn, float* dX, int64_t lddx, void* cuda_stream) {
    int rc = check_rows(X, ldx, rows, d, dtype);
    if (rc) return rc;
    if (!inv_norm) return GC_ERR_NULL;
    if ((rc = check_f32(dXn, lddxn, d))) return rc;
    if ((rc = check_f32(dX, lddx, d))) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e;
    auto go = [&](auto kernel) {
        return launch_chained(kernel, dim3(grid_for(rows)), 256, 0, 1, st, X, ldx, inv_norm, dXn, lddxn,
                              rows, d, dX, lddx);
    };
    const int keep = keep_cosine(rows, d, dtype);
    e = GC_KEEP_CALL(cosine_bwd_kernel, keep);
    return e == cudaSuccess ? GC_OK : GC_ERR_CUDA;
}

size_t gc_dtau_workspace_bytes(int64_t B) {
    return B > 0 ? (((size_t)B * sizeof(float)) + 255) & ~(size_t)255 : 0;
}

int gc_dtau(const void* Q, int64_t ldq, const float* dQ, int64_t lddq, int64_t B, int d, float tau,
            int dtype, float* dtau, void* ws, size_t ws_bytes, void* cuda_stream) {
    int rc = check_rows(Q, ldq, B, d, dtype);
    if (rc) return rc;
    if ((rc = check_f32(dQ, lddq, d))) return rc;
    if (!dtau) return GC_ERR_NULL;
    if (!(tau > 0.f) || !isfinite(tau)) return GC_ERR_SHAPE;
    if (!ws || ((uintptr_t)ws & 255) != 0 || ws_bytes < gc_dtau_workspace_bytes(B)) return GC_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e;
    float* row_dot = static_cast<float*>(ws);
    auto go = [&](auto kernel) {
        return launch_chained(kernel, dim3(grid_for(B)), 256, 0, 1, st, Q, ldq, dQ, lddq, B, d, row_dot);
    };
    if (dtype == GC_BF16) e = go(row_dot_kernel<true, 0>);
    else e = d > 1024 ? go(row_dot_kernel<false, 0>) : d <= 512 ? go(row_dot_kernel<false, 4>) : go(row_dot_kernel<false, 8>);
    if (e != cudaSuccess) return GC_ERR_CUDA;
    e = launch_chained(ordered_sum_kernel, dim3(1), 1024, 0, 1, st, row_dot, B, -1.f / tau, dtau);
    return e == cudaSuccess ? GC_OK : GC_ERR_CUDA;
}

}  // extern "C"
