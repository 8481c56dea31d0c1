// residual.cu -- Freivalds residual r = C x - A (B x) of a computed product.
//
// Three row-times-vector passes, each one block per matrix row with coalesced
// reads along the row: y = B x (K entries), z = A y (M), w = C x (M), r = w - z.
// Accumulation in fp32 (rowdot_kernel), or in fp64 for the optional refinement
// (rowdot64_kernel: O(mn + mk + kn) fp64 operations; the fp64 pipe, not HBM, sets
// its time).  One
// pass over A, B and C: bandwidth-bound in fp32.
#include "../../include/fmm.h"
#include "fmm_internal.h"
#include "ptx.cuh"

#include <cstdint>
#include <type_traits>

namespace fmm {
namespace {

// One block of 256 threads per row: out[row] = sum_c X[row][c] v[c] (minus
// sub[row]).  When the rows and v are 16-byte aligned, thread t reads columns
// 4g .. 4g + 3 for g = t, t + 256, ... (a block-wide coalesced sweep of the
// row, several 16-byte loads in flight per thread) into four independent
// partial sums; the last cols % 4 columns, or every column of unaligned rows,
// go one at a time.  Warp sums, then the 8 warp sums in a fixed order.  One
// row per block keeps the grid many waves deep (16384 rows: 13.5 waves).
template <typename Acc, typename Vec, typename Out>
__global__ void __launch_bounds__(256) rowdot_kernel(const float* X, long long ld, long long rows,
                                                     long long cols, const Vec* v,
                                                     Out* __restrict__ out, const double* sub,
                                                     int vec4) {
    __shared__ Acc warp_sum[8];
    dep_start();
    const long long row = blockIdx.x;
    const int t = threadIdx.x;
    const float* xr = X + row * ld;
    Acc a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    long long c0 = 0;
    if (vec4) {
        const long long groups = cols >> 2;
        const float4* x4 = reinterpret_cast<const float4*>(xr);
#pragma unroll 4
        for (long long g = t; g < groups; g += 256) {
            const float4 xv = x4[g];
            Acc v0, v1, v2, v3;
            if constexpr (std::is_same<Vec, float>::value) {
                const float4 q = reinterpret_cast<const float4*>(v)[g];
                v0 = q.x; v1 = q.y; v2 = q.z; v3 = q.w;
            } else {
                const double2 q0 = reinterpret_cast<const double2*>(v)[2 * g];
                const double2 q1 = reinterpret_cast<const double2*>(v)[2 * g + 1];
                v0 = (Acc)q0.x; v1 = (Acc)q0.y; v2 = (Acc)q1.x; v3 = (Acc)q1.y;
            }
            a0 += (Acc)xv.x * v0;
            a1 += (Acc)xv.y * v1;
            a2 += (Acc)xv.z * v2;
            a3 += (Acc)xv.w * v3;
        }
        c0 = groups << 2;
    }
    for (long long c = c0 + t; c < cols; c += 256) a0 += (Acc)xr[c] * (Acc)v[c];
    Acc acc = (a0 + a1) + (a2 + a3);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((t & 31) == 0) warp_sum[t >> 5] = acc;
    __syncthreads();
    if (t == 0) {
        Acc s = warp_sum[0];
#pragma unroll
        for (int w = 1; w < 8; ++w) s += warp_sum[w];
        if (sub) out[row] = (Out)((double)s - sub[row]);
        else out[row] = (Out)s;
    }
}

// float -> double without the FP64 pipe's conversion instruction: a normal
// value's bits are moved and its exponent rebiased by integer operations.
__device__ __forceinline__ bool is_normal(float x) {
    return (__float_as_uint(x) << 1) - 0x01000000u < 0xFE000000u;
}
__device__ __forceinline__ double widen_normal(float x) {
    const uint32_t u = __float_as_uint(x);
    return __hiloint2double((int)((((u & 0x7FFFFFFFu) >> 3) + 0x38000000u) | (u & 0x80000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen_any(float x) {   // zeros, subnormals, infinities, NaN too
    double d;
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(x));
    return d;
}
template <int N>
__device__ __forceinline__ void widen(const float (&x)[N], double (&d)[N]) {
    bool normal = true;
#pragma unroll
    for (int i = 0; i < N; ++i) normal = normal && is_normal(x[i]);
    if (normal) {
#pragma unroll
        for (int i = 0; i < N; ++i) d[i] = widen_normal(x[i]);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) d[i] = widen_any(x[i]);
    }
}

// rowdot_kernel in fp64: R consecutive rows per block, each with the sums and
// the order that kernel gives it, so v is read (and a float v widened) once for
// R rows.  Bound: the FP64 pipe (ncu: 91 % busy), which with one
// conversion per element of X and of v beside the FMA took 1.72 ms for the three
// passes at 12000 x 9001 x 10500, and with the FMA alone 0.74 ms.  R = 4 on
// 16-byte rows (four sums a row), 8 on others (one sum a row; two rows took
// 1.6 times as long as four); below 304 blocks of that, one row per block, off the
// 16-byte grid with eight of its columns per thread in flight (1024 x 16001 x 1025 94 us;
// 240 with one column at a time, 215 with a conversion per element).
template <typename Vec, int R, bool VEC4, bool STEP8 = false>
__global__ void __launch_bounds__(256, 3) rowdot64_kernel(const float* X, long long ld,
                                                                     long long rows, long long cols,
                                                                     const Vec* v,
                                                                     double* __restrict__ out,
                                                                     const double* sub) {
    __shared__ double warp_sum[8][R];
    dep_start();
    const long long row0 = (long long)blockIdx.x * R;
    const int t = threadIdx.x, nr = rows - row0 < R ? (int)(rows - row0) : R;
    const float* xr[R];
#pragma unroll
    for (int r = 0; r < R; ++r) xr[r] = X + (row0 + (r < nr ? r : 0)) * ld;   // rows past the end read the first one
    double a[R][VEC4 ? 4 : 1] = {};
    long long c0 = 0;
    if constexpr (VEC4) {
        const long long groups = cols >> 2;
#pragma unroll 1
        for (long long g = t; g < groups; g += 256) {
            float4 q[R];
#pragma unroll
            for (int r = 0; r < R; ++r) q[r] = reinterpret_cast<const float4*>(xr[r])[g];
            double w[4];
            if constexpr (std::is_same<Vec, float>::value) {
                const float4 f = reinterpret_cast<const float4*>(v)[g];
                const float ff[4] = {f.x, f.y, f.z, f.w};
                widen(ff, w);
            } else {
                const double2 d0 = reinterpret_cast<const double2*>(v)[2 * g];
                const double2 d1 = reinterpret_cast<const double2*>(v)[2 * g + 1];
                w[0] = d0.x; w[1] = d0.y; w[2] = d1.x; w[3] = d1.y;
            }
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float qq[4] = {q[r].x, q[r].y, q[r].z, q[r].w};
                double d[4];
                widen(qq, d);
#pragma unroll
                for (int i = 0; i < 4; ++i) a[r][i] += d[i] * w[i];
            }
        }
        c0 = groups << 2;
    }
    long long c = c0 + t;
    if constexpr (STEP8) {
        // one row: eight loads in flight come from eight of its columns (widen's branch
        // keeps a later column's loads behind it)
        for (; c + 7 * 256 < cols; c += 8 * 256) {
            float q[8];
            double d[8], w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) q[i] = xr[0][c + 256 * i];
            if constexpr (std::is_same<Vec, float>::value) {
                float f[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) f[i] = v[c + 256 * i];
                widen(f, w);
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) w[i] = v[c + 256 * i];
            }
            widen(q, d);
#pragma unroll
            for (int i = 0; i < 8; ++i) a[0][0] += d[i] * w[i];
        }
    }
#pragma unroll 2
    for (; c < cols; c += 256) {
        float q[R];
#pragma unroll
        for (int r = 0; r < R; ++r) q[r] = xr[r][c];
        double d[R], w[1];
        if constexpr (std::is_same<Vec, float>::value) {
            const float f[1] = {v[c]};
            widen(f, w);
        } else {
            w[0] = v[c];
        }
        widen(q, d);
#pragma unroll
        for (int r = 0; r < R; ++r) a[r][0] += d[r] * w[0];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        double acc = a[r][0];
        if constexpr (VEC4) acc = (a[r][0] + a[r][1]) + (a[r][2] + a[r][3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((t & 31) == 0) warp_sum[t >> 5][r] = acc;
    }
    __syncthreads();
    if (t < nr) {
        double s = warp_sum[0][t];
#pragma unroll
        for (int w = 1; w < 8; ++w) s += warp_sum[w][t];
        out[row0 + t] = sub ? s - sub[row0 + t] : s;
    }
}

template <typename Vec>
void rowdot64(const float* X, long long ld, long long rows, long long cols, const Vec* v, double* out,
              const double* sub, int vec4, cudaStream_t s) {
    const int R = vec4 ? 4 : 8;
    const bool wide = rows >= 304LL * R;
    const unsigned grid = (unsigned)(wide ? (rows + R - 1) / R : rows);
    if (vec4) {
        if (wide) launch_dep(rowdot64_kernel<Vec, 4, true>, grid, 256, 0, s, X, ld, rows, cols, v, out, sub);
        else launch_dep(rowdot64_kernel<Vec, 1, true>, grid, 256, 0, s, X, ld, rows, cols, v, out, sub);
    } else {
        if (wide) launch_dep(rowdot64_kernel<Vec, 8, false>, grid, 256, 0, s, X, ld, rows, cols, v, out, sub);
        // shorter rows take no step of eight, and fit more blocks on an SM without it
        else if (cols > 7 * 256) launch_dep(rowdot64_kernel<Vec, 1, false, true>, grid, 256, 0, s, X, ld, rows, cols, v, out, sub);
        else launch_dep(rowdot64_kernel<Vec, 1, false>, grid, 256, 0, s, X, ld, rows, cols, v, out, sub);
    }
}

inline int aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 ? 1 : 0; }

// y = B x ; z = A y ; r = C x - z.  y is kept in the accumulation type: an
// fp32 sum is exactly representable either way, and a float y keeps the
// middle pass off the FP64 pipe (a double-to-float conversion per element).
template <typename Acc>
cudaError_t residual_impl(long long M, long long N, long long K, const float* A, long long lda, const float* B,
                          long long ldb, const float* C, long long ldc, const float* x, double* r, double* y_ws,
                          double* z, cudaStream_t s) {
    Acc* y = reinterpret_cast<Acc*>(y_ws);   // K entries (the workspace holds K doubles)
    const int vx = aligned16(x), vy = aligned16(y);
    const int bv = vx & aligned16(B) & (ldb % 4 == 0), av = vy & aligned16(A) & (lda % 4 == 0),
              cv = vx & aligned16(C) & (ldc % 4 == 0);
    if constexpr (std::is_same<Acc, double>::value) {
        if (K > 0) rowdot64<float>(B, ldb, K, N, x, y, nullptr, bv, s);
        rowdot64<double>(A, lda, M, K, y, z, nullptr, av, s);
        rowdot64<float>(C, ldc, M, N, x, r, z, cv, s);
    } else {
        if (K > 0) launch_dep(rowdot_kernel<Acc, float, Acc>, (unsigned)K, 256, 0, s, B, ldb, K, N, x, y, nullptr, bv);
        launch_dep(rowdot_kernel<Acc, Acc, double>, (unsigned)M, 256, 0, s, A, lda, M, K, y, z, nullptr, av);
        launch_dep(rowdot_kernel<Acc, float, double>, (unsigned)M, 256, 0, s, C, ldc, M, N, x, r, z, cv);
    }
    return cudaGetLastError();
}

}  // namespace
}  // namespace fmm

extern "C" fmm_status_t fmm_residual(int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B,
                                     int64_t ldb, const float* C, int64_t ldc, const float* x, double* r,
                                     void* workspace, size_t workspace_bytes, size_t* workspace_needed, int fp64,
                                     fmm_stream_t stream) {
    if (M < 0 || N < 0 || K < 0) return FMM_ERR_INVALID_ARG;
    if (lda < (K > 0 ? K : 1) || ldb < (N > 0 ? N : 1) || ldc < (N > 0 ? N : 1)) return FMM_ERR_INVALID_ARG;
    const size_t need = ((size_t)(K > 0 ? K : 1) + (size_t)(M > 0 ? M : 1)) * sizeof(double) + 256;
    if (workspace_needed) *workspace_needed = need;
    if (!workspace && !r) return FMM_OK;  // size query
    if (M == 0) return FMM_OK;
    if (!A || !B || !C || !x || !r) return FMM_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < need) return FMM_ERR_WORKSPACE;
    double* y = static_cast<double*>(workspace);
    double* z = y + (K > 0 ? K : 1);
    cudaError_t e = fp64 ? fmm::residual_impl<double>(M, N, K, A, lda, B, ldb, C, ldc, x, r, y, z, (cudaStream_t)stream)
                         : fmm::residual_impl<float>(M, N, K, A, lda, B, ldb, C, ldc, x, r, y, z, (cudaStream_t)stream);
    return e == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}
