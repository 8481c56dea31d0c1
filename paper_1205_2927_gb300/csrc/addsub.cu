// addsub.cu -- bandwidth-bound kernels of the recursion: the 8 pre-additions
// (S1..S4 on A, T1..T4 on B) and the 7 post-additions (U1..U7) of Winograd's
// variant of Strassen's algorithm, plus the copies the leaves need (transposed
// right operand, aligned left operand) and C <- beta*C.
//
// Quadrant naming follows Eq. 1: Q0 = X11 (top-left), Q1 = X12, Q2 = X21,
// Q3 = X22.  The right operand is kept transposed (Y = B^T, K-major) below the
// root, so B11 = Y11^T, B12 = Y21^T, B21 = Y12^T, B22 = Y22^T and
//   T1^T = Y21 - Y11,  T2^T = Y22 - T1^T,  T3^T = Y22 - Y21,  T4^T = T2^T - Y12.
// Child order (one child per product P1..P7):
//   A side: Q0, Q1, S4, Q3, S1, S2, S3        (sums only: S1, S2, S3, S4)
//   B side: Y0, Y1, Y3, T4, T1, T2, T3        (sums only: T1, T2, T3, T4)
// All streaming kernels move 16-byte vectors when the view allows it.
#include "fmm_internal.h"
#include "ptx.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace fmm {

namespace {

__device__ __forceinline__ float4 f4(float a, float b, float c, float d) { return make_float4(a, b, c, d); }
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return f4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 sub4(float4 a, float4 b) { return f4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }

// 4 consecutive elements (r, c..c+3) of quadrant q of node view `base`,
// zero outside valid rows/cols.
template <bool VEC>
__device__ __forceinline__ float4 load_q(const View& v, const float* base, long long r, long long c) {
    if (VEC) {
        if (r < v.valid_rows && c + 3 < v.valid_cols) return *reinterpret_cast<const float4*>(base + r * v.ld + c);
    }
    float t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = (r < v.valid_rows && c + j < v.valid_cols) ? base[r * v.ld + c + j] : 0.0f;
    return f4(t[0], t[1], t[2], t[3]);
}

__device__ __forceinline__ void store4(float* p, float4 v, bool vec, long long nvalid) {
    if (vec && nvalid >= 4) { *reinterpret_cast<float4*>(p) = v; return; }
    if (nvalid > 0) p[0] = v.x;
    if (nvalid > 1) p[1] = v.y;
    if (nvalid > 2) p[2] = v.z;
    if (nvalid > 3) p[3] = v.w;
}

// grid: x over column groups of 4, y over rows (strided), z over nodes.
template <bool VEC, int SIDE_B, bool FULL>
__global__ void __launch_bounds__(128) pre_add_kernel(View P, long long h, long long w, Stack out, int dep) {
    if (dep) dep_start();
    const long long c = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (c >= w) return;
    const long long node = blockIdx.z;
    const float* base = P.ptr + node * P.node_stride;
    const float* q1p = base + w;
    const float* q2p = base + h * P.ld;
    const float* q3p = q2p + w;
    // quadrant views share the node's validity window, shifted
    View v0 = P, v1 = P, v2 = P, v3 = P;
    v1.valid_cols = P.valid_cols - w;
    v2.valid_rows = P.valid_rows - h;
    v3.valid_rows = P.valid_rows - h;
    v3.valid_cols = P.valid_cols - w;
    const long long nvalid = w - c;
    for (long long r = blockIdx.y; r < h; r += gridDim.y) {
        const float4 Q0 = load_q<VEC>(v0, base, r, c);
        const float4 Q1 = load_q<VEC>(v1, q1p, r, c);
        const float4 Q2 = load_q<VEC>(v2, q2p, r, c);
        const float4 Q3 = load_q<VEC>(v3, q3p, r, c);
        float4 X1, X2, X3, X4;  // S1..S4 or T1^T..T4^T
        if (!SIDE_B) {
            X1 = add4(Q2, Q3);   // S1 = A21 + A22
            X2 = sub4(X1, Q0);   // S2 = S1 - A11
            X3 = sub4(Q0, Q2);   // S3 = A11 - A21
            X4 = sub4(Q1, X2);   // S4 = A12 - S2
        } else {
            X1 = sub4(Q2, Q0);   // T1^T = Y21 - Y11  (B12 - B11)
            X2 = sub4(Q3, X1);   // T2^T = Y22 - T1^T (B22 - T1)
            X3 = sub4(Q3, Q2);   // T3^T = Y22 - Y21  (B22 - B12)
            X4 = sub4(X2, Q1);   // T4^T = T2^T - Y12 (T2 - B21)
        }
        float* o = out.ptr + (node * out.nchild) * out.child_stride + r * out.ld + c;
        const long long cs = out.child_stride;
        if (FULL) {
            store4(o + 0 * cs, Q0, VEC, nvalid);
            store4(o + 1 * cs, Q1, VEC, nvalid);
            if (!SIDE_B) {
                store4(o + 2 * cs, X4, VEC, nvalid);  // P3 = S4 B22
                store4(o + 3 * cs, Q3, VEC, nvalid);  // P4 = A22 T4
            } else {
                store4(o + 2 * cs, Q3, VEC, nvalid);  // P3: B22
                store4(o + 3 * cs, X4, VEC, nvalid);  // P4: T4
            }
            store4(o + 4 * cs, X1, VEC, nvalid);
            store4(o + 5 * cs, X2, VEC, nvalid);
            store4(o + 6 * cs, X3, VEC, nvalid);
        } else {
            store4(o + 0 * cs, X1, VEC, nvalid);
            store4(o + 1 * cs, X2, VEC, nvalid);
            store4(o + 2 * cs, X3, VEC, nvalid);
            store4(o + 3 * cs, X4, VEC, nvalid);
        }
    }
}

// Root B side: B is K x N row-major (ldb).  Tile of 32 (k) x 32 (n) in the
// half domain; reads the four quadrants coalesced along n, writes the
// transposed children coalesced along k.  blockDim = (32, 8).
template <bool FULL>
__global__ void __launch_bounds__(256) pre_add_b_root_kernel(const float* B, long long ldb, long long K,
                                                             long long N, long long kh, long long nh, Stack out) {
    dep_start();
    constexpr int NC = FULL ? 7 : 4;
    __shared__ float tile[NC][32][33];
    const long long k0 = (long long)blockIdx.y * 32, n0 = (long long)blockIdx.x * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int kl = ty + 8 * i;
        const long long k = k0 + kl, n = n0 + tx;
        float b11 = 0.f, b12 = 0.f, b21 = 0.f, b22 = 0.f;
        if (k < kh && n < nh) {
            const long long kk2 = k + kh, nn2 = n + nh;
            if (k < K && n < N) b11 = B[k * ldb + n];
            if (k < K && nn2 < N) b12 = B[k * ldb + nn2];
            if (kk2 < K && n < N) b21 = B[kk2 * ldb + n];
            if (kk2 < K && nn2 < N) b22 = B[kk2 * ldb + nn2];
        }
        const float t1 = b12 - b11;  // T1 = B12 - B11
        const float t2 = b22 - t1;   // T2 = B22 - T1
        const float t3 = b22 - b12;  // T3 = B22 - B12
        const float t4 = t2 - b21;   // T4 = T2 - B21
        if (FULL) {
            tile[0][kl][tx] = b11; tile[1][kl][tx] = b21; tile[2][kl][tx] = b22; tile[3][kl][tx] = t4;
            tile[4][kl][tx] = t1;  tile[5][kl][tx] = t2;  tile[6][kl][tx] = t3;
        } else {
            tile[0][kl][tx] = t1; tile[1][kl][tx] = t2; tile[2][kl][tx] = t3; tile[3][kl][tx] = t4;
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int nl = ty + 8 * i;
        const long long n = n0 + nl, k = k0 + tx;
        if (n < nh && k < kh) {
#pragma unroll
            for (int c = 0; c < NC; ++c) out.ptr[c * out.child_stride + n * out.ld + k] = tile[c][tx][nl];
        }
    }
}

// Post-additions: per node, children P1..P7 (h x w each) -> node output.
template <bool VEC, bool ROOT>
__global__ void __launch_bounds__(128) post_add_kernel(const float* P, long long ld_in, long long cs,
                                                       long long h, long long w, float* __restrict__ out, long long ld_out,
                                                       long long out_ns, long long valid_rows, long long valid_cols,
                                                       float alpha, float beta) {
    dep_start();
    const long long c = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (c >= w) return;
    const long long node = blockIdx.z;
    const float* base = P + node * 7 * cs;
    float* o = out + node * out_ns;
    for (long long r = blockIdx.y; r < h; r += gridDim.y) {
        const float* pr = base + r * ld_in + c;
        float4 p[7];
        if (VEC) {
#pragma unroll
            for (int i = 0; i < 7; ++i) p[i] = *reinterpret_cast<const float4*>(pr + i * cs);
        } else {
#pragma unroll
            for (int i = 0; i < 7; ++i) {
                float t[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) t[j] = (c + j < w) ? pr[i * cs + j] : 0.0f;
                p[i] = f4(t[0], t[1], t[2], t[3]);
            }
        }
        const float4 U1 = add4(p[0], p[1]);   // P1 + P2
        const float4 U2 = add4(p[0], p[5]);   // P1 + P6
        const float4 U3 = add4(U2, p[6]);     // U2 + P7
        const float4 U4 = add4(U2, p[4]);     // U2 + P5
        const float4 U5 = add4(U4, p[2]);     // U4 + P3
        const float4 U6 = sub4(U3, p[3]);     // U3 - P4
        const float4 U7 = add4(U3, p[4]);     // U3 + P5
        const float4 quad[4] = {U1, U5, U6, U7};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const long long rr = r + (q >> 1) * h;
            const long long cc = c + (q & 1) * w;
            float4 v = quad[q];
            if (!ROOT) {
                store4(o + rr * ld_out + cc, v, VEC, w - c);
            } else {
                if (rr >= valid_rows || cc >= valid_cols) continue;
                const long long nv = min(min(4LL, w - c), valid_cols - cc);
                float* dst = o + rr * ld_out + cc;
                const bool vec = VEC && nv == 4 && ((reinterpret_cast<uintptr_t>(dst) & 15) == 0);
                if (vec) {
                    float4 r4 = f4(alpha * v.x, alpha * v.y, alpha * v.z, alpha * v.w);
                    if (beta != 0.0f) {
                        const float4 old = *reinterpret_cast<const float4*>(dst);
                        r4.x += beta * old.x; r4.y += beta * old.y; r4.z += beta * old.z; r4.w += beta * old.w;
                    }
                    *reinterpret_cast<float4*>(dst) = r4;
                } else {
                    const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (j < nv) {
                            float x = alpha * vv[j];
                            if (beta != 0.0f) x += beta * dst[j];
                            dst[j] = x;
                        }
                    }
                }
            }
        }
    }
}

// Bt (rows_out x cols_out, >= N x K) = B^T, zeros outside the N x K valid part.
__global__ void __launch_bounds__(256) transpose_kernel(const float* B, long long ldb, long long K,
                                                        long long N, float* __restrict__ Bt, long long ldt,
                                                        long long rows_out, long long cols_out) {
    dep_start();
    // one 128 (k) x 32 (n) block of B per CTA: 16 loads in flight per thread,
    // then 32 rows of B^T written as 512 contiguous bytes each
    __shared__ float tile[32][129];   // [n][k]
    const long long k0 = (long long)blockIdx.y * 128, n0 = (long long)blockIdx.x * 32;
    const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
    float x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const long long k = k0 + warp + 8 * i, n = n0 + lane;
        x[i] = (k < K && n < N) ? B[k * ldb + n] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) tile[lane][warp + 8 * i] = x[i];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int v = tid + 256 * j;   // row v / 128 of the B^T block, column v % 128
        const long long n = n0 + (v >> 7), k = k0 + (v & 127);
        if (n < rows_out && k < cols_out) Bt[n * ldt + k] = tile[v >> 7][v & 127];
    }
}

__global__ void copy2d_kernel(const float* A, long long lda, long long M, long long K, float* dst,
                              long long ldd) {
    dep_start();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long r = blockIdx.y; r < M; r += gridDim.y)
        if (c < K) dst[r * ldd + c] = A[r * lda + c];
}

__global__ void scale_kernel(float* C, long long ldc, long long M, long long N, float beta) {
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (long long r = blockIdx.y; r < M; r += gridDim.y)
        if (c < N) C[r * ldc + c] = (beta == 0.0f) ? 0.0f : beta * C[r * ldc + c];
}

__global__ void __launch_bounds__(256) batched_copy_kernel(const CopyJob* __restrict__ jobs, int njobs) {
    __shared__ float tile[32][33];
    const long long t = blockIdx.x;
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].tile_begin <= t) lo = mid; else hi = mid - 1;
    }
    const CopyJob J = jobs[lo];
    const long long local = t - J.tile_begin;
    const long long r0 = (local / J.tiles_c) * 32, c0 = (local % J.tiles_c) * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;
    if (!J.transpose) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const long long r = r0 + ty + 8 * i, c = c0 + tx;
            if (r < J.rows && c < J.cols) J.dst[r * J.ldd + c] = J.src[r * J.lds + c];
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long r = r0 + ty + 8 * i, c = c0 + tx;
        tile[ty + 8 * i][tx] = (r < J.rows && c < J.cols) ? J.src[r * J.lds + c] : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const long long c = c0 + ty + 8 * i, r = r0 + tx;
        if (c < J.cols && r < J.rows) J.dst[c * J.ldd + r] = tile[tx][ty + 8 * i];
    }
}

__global__ void fill_kernel(float* p, size_t n, unsigned seed) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        unsigned x = (unsigned)i * 2654435761u ^ seed;   // integer hash (xorshift-multiply)
        x ^= x >> 16; x *= 0x7feb352du; x ^= x >> 15; x *= 0x846ca68bu; x ^= x >> 16;
        p[i] = (float)(x >> 8) * (2.0f / 16777216.0f) - 1.0f;
    }
}

// max |x| of A and of B in one launch, folded into mx[0] and mx[1] (float bits;
// non-negative floats order like unsigned integers).  Blocks stride over 32 x 128
// blocks of both operands, two at a time: eight 16-byte loads per thread in
// flight where the rows allow; one atomic per block and operand.  Bound: HBM.
// n = 8192: 78 us, against 70 + 70 for one launch per operand with two loads
// in flight.
struct MaxOperand {
    const float* X;
    long long ld, rows, cols, tiles_c, tiles;   // tiles_c 128-column blocks per 32-row band
};
__device__ __forceinline__ void absmax_load(const MaxOperand& o, bool vec, long long tile, int tid, float4 (&v)[4]) {
    const long long band = tile / o.tiles_c, r0 = band * 32, c0 = (tile - band * o.tiles_c) * 128;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int g = tid + 256 * j;   // row g / 32 of the block, columns 4 (g % 32) .. + 3
        const long long r = r0 + (g >> 5), c = c0 + 4 * (g & 31);
        v[j] = f4(0.f, 0.f, 0.f, 0.f);
        if (r >= o.rows || c >= o.cols) continue;
        const float* src = o.X + r * o.ld + c;
        if (vec && c + 3 < o.cols) {
            v[j] = __ldg(reinterpret_cast<const float4*>(src));
        } else {
            v[j].x = __ldg(src);
            if (c + 1 < o.cols) v[j].y = __ldg(src + 1);
            if (c + 2 < o.cols) v[j].z = __ldg(src + 2);
            if (c + 3 < o.cols) v[j].w = __ldg(src + 3);
        }
    }
}
__global__ void __launch_bounds__(256) absmax_kernel(MaxOperand A, MaxOperand B, unsigned* mx) {
    __shared__ float warp_max[8];
    dep_trigger();
    const int tid = threadIdx.x;
#pragma unroll 1
    for (int which = 0; which < 2; ++which) {
        const MaxOperand& o = which ? B : A;
        const bool vec = (reinterpret_cast<uintptr_t>(o.X) & 15) == 0 && (o.ld & 3) == 0;
        float m = 0.f;
        for (long long t = blockIdx.x; t < o.tiles; t += 2LL * gridDim.x) {
            float4 v[2][4];
            absmax_load(o, vec, t, tid, v[0]);
            absmax_load(o, vec, min(t + gridDim.x, o.tiles - 1), tid, v[1]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 x = v[i >> 2][i & 3];
                m = fmaxf(fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y))), fmaxf(fabsf(x.z), fabsf(x.w)));
            }
        }
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, s));
        if ((tid & 31) == 0) warp_max[tid >> 5] = m;
        __syncthreads();
        if (tid == 0) {
#pragma unroll
            for (int w = 1; w < 8; ++w) m = fmaxf(m, warp_max[w]);
            if (blockIdx.x < o.tiles) atomicMax(mx + which, __float_as_uint(m));
        }
        __syncthreads();
    }
}

// Largest power of two s with m * s <= 2^14 (1 for m = 0 or not finite).
__device__ __forceinline__ float fp16_scale_of(float m) {
    if (!(m > 0.f) || !isfinite(m)) return 1.0f;
    int x;
    frexpf(m, &x);                   // m = f * 2^x, 0.5 <= f < 1
    int e = 14 - x;                  // largest e with m * 2^e <= 2^14
    e = max(-100, min(100, e));
    return ldexpf(1.0f, e);
}

__global__ void fp16_scale_kernel(const unsigned* mx, float bound_mult, float* scale) {
    dep_start();
    const int i = threadIdx.x;
    if (i > 1) return;
    scale[i] = fp16_scale_of(__uint_as_float(mx[i]) * bound_mult);
}

// Batched maxima: every block takes a run of consecutive 32 x 128 blocks (found once
// by binary search), two at a time as in absmax_kernel, and folds what it saw of a
// job into the job's slot when the run leaves it.  Bound: HBM.  512 FP16x3 products,
// 5.8 GB of operands: a call 6.38 ms with one 32 x 128 block per CTA, now 6.12.
__global__ void __launch_bounds__(256) batched_absmax_kernel(const AbsJob* __restrict__ jobs, int njobs, long long total) {
    __shared__ float warp_max[8];
    dep_trigger();
    const long long per = (total + gridDim.x - 1) / gridDim.x;
    long long t = blockIdx.x * per;
    const long long stop = min(total, t + per);
    if (t >= stop) return;
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].tile_begin <= t) lo = mid; else hi = mid - 1;
    }
    const int tid = threadIdx.x;
    for (; t < stop; ++lo) {
        const AbsJob J = jobs[lo];
        const long long end = lo + 1 < njobs ? min(stop, jobs[lo + 1].tile_begin) : stop;
        const MaxOperand o{J.src, J.lds, J.rows, J.cols, J.tiles_c, 0};
        const bool vec = (reinterpret_cast<uintptr_t>(J.src) & 15) == 0 && (J.lds & 3) == 0;
        float m = 0.f;
        for (; t < end; t += 2) {
            float4 v[2][4];
            absmax_load(o, vec, t - J.tile_begin, tid, v[0]);
            absmax_load(o, vec, min(t + 1, end - 1) - J.tile_begin, tid, v[1]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 x = v[i >> 2][i & 3];
                m = fmaxf(fmaxf(m, fmaxf(fabsf(x.x), fabsf(x.y))), fmaxf(fabsf(x.z), fabsf(x.w)));
            }
        }
        t = end;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, s));
        if ((tid & 31) == 0) warp_max[tid >> 5] = m;
        __syncthreads();
        if (tid == 0) {
#pragma unroll
            for (int w = 1; w < 8; ++w) m = fmaxf(m, warp_max[w]);
            atomicMax(J.slot, __float_as_uint(m));
        }
        __syncthreads();
    }
}

__global__ void batched_fp16_scale_kernel(const unsigned* maxima, const float* bound,
                                          float* __restrict__ scales, int count) {
    dep_start();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 2 * count) return;
    scales[i] = fp16_scale_of(__uint_as_float(maxima[i]) * bound[i >> 1]);
}

// Root pre-additions of the host-streamed schedule: the four quadrants are
// separate row-major buffers (h x w, row stride ld), and a launch forms the sums
// whose quadrants have arrived.
//   A side: S1 = Q2 + Q3, S2 = S1 - Q0, S3 = Q0 - Q2, then S4 = Q1 - S2
//   B side: T1 = Q1 - Q0, then T2 = Q3 - T1, T3 = Q3 - Q1, then T4 = T2 - Q2
template <QuadSums SUMS>
__global__ void __launch_bounds__(128) quad_pre_kernel(QuadPre q) {
    const long long c = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (c >= q.w) return;
    for (long long r = blockIdx.y; r < q.h; r += gridDim.y) {
        const long long o = r * q.ld + c;
        auto Q = [&](int i) { return *reinterpret_cast<const float4*>(q.in[i] + o); };
        auto X = [&](int i) { return *reinterpret_cast<const float4*>(q.out[i - 1] + o); };
        auto put = [&](int i, float4 v) { *reinterpret_cast<float4*>(q.out[i - 1] + o) = v; };
        if constexpr (SUMS == kQuadS123) {
            const float4 Q0 = Q(0), Q2 = Q(2), S1 = add4(Q2, Q(3));
            put(1, S1);
            put(2, sub4(S1, Q0));
            put(3, sub4(Q0, Q2));
        } else if constexpr (SUMS == kQuadS4) {
            put(4, sub4(Q(1), X(2)));
        } else if constexpr (SUMS == kQuadT1) {
            put(1, sub4(Q(1), Q(0)));
        } else if constexpr (SUMS == kQuadT23) {
            const float4 Q3 = Q(3), T1 = X(1), Q1 = Q(1);
            put(2, sub4(Q3, T1));
            put(3, sub4(Q3, Q1));
        } else {
            put(4, sub4(X(2), Q(2)));
        }
    }
}

// Root post-additions of the host-streamed schedule from the seven product
// buffers (h x w, row stride ld) into one quadrant buffer of C (same layout),
// with the U-chain's operation order, so each quadrant can be formed (and
// copied out) as soon as its products exist:
//   part 0: C11 = alpha * U1 + beta * C11, U1 = P1 + P2
//   part 1: C12 = alpha * U5 + beta * C12, U5 = ((P1 + P6) + P5) + P3
//   part 2: C21 = alpha * U6 + beta * C21, U6 = ((P1 + P6) + P7) - P4
//   part 3: C22 = alpha * U7 + beta * C22, U7 = ((P1 + P6) + P7) + P5
template <int PART>
__global__ void __launch_bounds__(128) quad_post_kernel(QuadPost q) {
    const long long c = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (c >= q.w) return;
    for (long long r = blockIdx.y; r < q.h; r += gridDim.y) {
        const long long o = r * q.ld + c;
        auto P = [&](int i) { return *reinterpret_cast<const float4*>(q.p[i] + o); };
        auto put = [&](float* dst, float4 u) {
            float4 v = f4(q.alpha * u.x, q.alpha * u.y, q.alpha * u.z, q.alpha * u.w);
            if (q.beta != 0.0f) {
                const float4 old = *reinterpret_cast<const float4*>(dst + o);
                v.x += q.beta * old.x; v.y += q.beta * old.y; v.z += q.beta * old.z; v.w += q.beta * old.w;
            }
            *reinterpret_cast<float4*>(dst + o) = v;
        };
        if (PART == 0) {
            put(q.c[0], add4(P(0), P(1)));
        } else {
            const float4 U2 = add4(P(0), P(5));
            if (PART == 1) {
                put(q.c[1], add4(add4(U2, P(4)), P(2)));   // U5 = U4 + P3, U4 = U2 + P5
            } else {
                const float4 U3 = add4(U2, P(6));
                if (PART == 2) put(q.c[2], sub4(U3, P(3)));   // U6 = U3 - P4
                else put(q.c[3], add4(U3, P(4)));             // U7 = U3 + P5
            }
        }
    }
}

// ---------------------------------------------------------------- 16-bit hi/lo planes
// Split four consecutive values into the planes at element offset o.
//   bf16 / fp16: x * s = hi + lo (+ residual), hi = rn16(x s), lo = rn16(x s - hi)
//   tf32:        hi = x (the tensor core reads trunc_tf32(x)), lo = rn_tf32(x - trunc_tf32(x))
// The planes are written with evict-first (streaming) stores: they are read by
// the leaf launch only after far more data than L2 holds has passed, and they
// must not push out the operand lines a fused pass reads again.
//   tf32x:       hi = rn_tf32(x), and in the other plane bf16(hi) and bf16(x - hi), 32 columns of
//                each per 128-byte line (zeros for an infinity, which the hi plane alone carries)
// Two values to bf16, nearest even, saturating at the largest finite value.
__device__ __forceinline__ uint32_t bf16x2_sat(float x0, float x1) {
    uint32_t r;
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(x1), "f"(x0));
    return r;
}
// 16-bit offset of hi (lo: + 32) of the element at offset o of a tf32x correction plane.
__device__ __forceinline__ long long tf32x_off(long long o) { return 2 * (o & ~31LL) + (o & 31); }

// RAW (A of a depth-0 product): hi = x as for tf32, whether the leaves read the operand
// itself (no hi plane) or its copy, so that a product has the same bits at any alignment
// of A; tf32x corrections are then those of trunc_tf32(x).
template <int KIND, bool RAW = false>
__device__ __forceinline__ void split_store(void* hi_plane, void* lo_plane, long long o, float4 v, float sc) {
    if constexpr (KIND == kSplitTF32X) {
        float4 h = RAW ? f4(tf32_trunc(v.x), tf32_trunc(v.y), tf32_trunc(v.z), tf32_trunc(v.w))
                       : f4(tf32_round_hi(v.x), tf32_round_hi(v.y), tf32_round_hi(v.z), tf32_round_hi(v.w));
        if (hi_plane) __stcs(reinterpret_cast<float4*>(static_cast<float*>(hi_plane) + o), RAW ? v : h);
        // an infinity's product is its hi's alone: x - hi would be NaN
        float4 l = sub4(v, h);
        if (isinf(fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))))) {
            if (isinf(v.x)) h.x = l.x = 0.f;
            if (isinf(v.y)) h.y = l.y = 0.f;
            if (isinf(v.z)) h.z = l.z = 0.f;
            if (isinf(v.w)) h.w = l.w = 0.f;
        }
        uint16_t* hl = static_cast<uint16_t*>(lo_plane) + tf32x_off(o);
        __stcs(reinterpret_cast<uint2*>(hl), make_uint2(bf16x2_sat(h.x, h.y), bf16x2_sat(h.z, h.w)));
        __stcs(reinterpret_cast<uint2*>(hl + 32), make_uint2(bf16x2_sat(l.x, l.y), bf16x2_sat(l.z, l.w)));
        return;
    }
    if constexpr (KIND == kSplitTF32) {
        float4 l;
        l.x = tf32_round_rne(v.x - tf32_trunc(v.x));
        l.y = tf32_round_rne(v.y - tf32_trunc(v.y));
        l.z = tf32_round_rne(v.z - tf32_trunc(v.z));
        l.w = tf32_round_rne(v.w - tf32_trunc(v.w));
        // no hi plane: the leaves read the raw operand itself (hi = x)
        if (hi_plane) __stcs(reinterpret_cast<float4*>(static_cast<float*>(hi_plane) + o), v);
        __stcs(reinterpret_cast<float4*>(static_cast<float*>(lo_plane) + o), l);
        return;
    }
    uint16_t* hi = static_cast<uint16_t*>(hi_plane) + o;
    uint16_t* lo = static_cast<uint16_t*>(lo_plane) + o;
    const float x0 = v.x * sc, x1 = v.y * sc, x2 = v.z * sc, x3 = v.w * sc;
    uint32_t h01, h23, l01, l23;
    if constexpr (KIND == kSplitBF16) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(x0, x1), b = __floats2bfloat162_rn(x2, x3);
        const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
        const __nv_bfloat162 c = __floats2bfloat162_rn(x0 - fa.x, x1 - fa.y), d = __floats2bfloat162_rn(x2 - fb.x, x3 - fb.y);
        h01 = *reinterpret_cast<const uint32_t*>(&a); h23 = *reinterpret_cast<const uint32_t*>(&b);
        l01 = *reinterpret_cast<const uint32_t*>(&c); l23 = *reinterpret_cast<const uint32_t*>(&d);
    } else {
        const __half2 a = __floats2half2_rn(x0, x1), b = __floats2half2_rn(x2, x3);
        const float2 fa = __half22float2(a), fb = __half22float2(b);
        const __half2 c = __floats2half2_rn(x0 - fa.x, x1 - fa.y), d = __floats2half2_rn(x2 - fb.x, x3 - fb.y);
        h01 = *reinterpret_cast<const uint32_t*>(&a); h23 = *reinterpret_cast<const uint32_t*>(&b);
        l01 = *reinterpret_cast<const uint32_t*>(&c); l23 = *reinterpret_cast<const uint32_t*>(&d);
    }
    __stcs(reinterpret_cast<uint2*>(hi), make_uint2(h01, h23));
    __stcs(reinterpret_cast<uint2*>(lo), make_uint2(l01, l23));
}

// Columns a split pass writes of a matrix of `cols` columns: a tf32x correction
// plane is zero up to the next multiple of 32 (the planes' pitch covers it).
template <int KIND>
__host__ __device__ __forceinline__ long long plane_cols(long long cols) {
    return KIND == kSplitTF32X ? (cols + 31) & ~31LL : cols;
}

// Plain split (transpose = 0: rows x cols -> rows x ld planes) or transposed
// split (transpose = 1: X is rows(K) x cols(N), planes are cols x ld).  Every
// thread issues all of its loads before its first store.  Plain: one 32 x 128
// block per CTA, 16-byte loads straight to the planes.  Transposed: one
// 128 (row) x 32 (column) block staged in a shared tile, left as 32 plane rows
// of 128 elements (512 contiguous bytes each).
template <int KIND, bool TRANS>
__global__ void __launch_bounds__(256) split16_kernel(const float* X, long long ldx, long long rows,
                                                      long long cols, Stack16 out, const float* scale,
                                                      int which) {
    dep_start();
    const float sc = scale ? scale[which] : 1.0f;
    const int lane = threadIdx.x, warp = threadIdx.y, tid = warp * 32 + lane;
    if (!TRANS) {
        const long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 128;
        const bool vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0 && (ldx & 3) == 0;
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int g = tid + 256 * j;   // row g / 32 of the block, columns 4 (g % 32) .. + 3
            const long long r = r0 + (g >> 5), c = c0 + 4 * (g & 31);
            v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r >= rows || c >= cols) continue;
            const float* src = X + r * ldx + c;
            if (vec && c + 3 < cols) {
                v[j] = *reinterpret_cast<const float4*>(src);
            } else {
                v[j].x = *src;
                if (c + 1 < cols) v[j].y = src[1];
                if (c + 2 < cols) v[j].z = src[2];
                if (c + 3 < cols) v[j].w = src[3];
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int g = tid + 256 * j;
            const long long r = r0 + (g >> 5), c = c0 + 4 * (g & 31);
            // ld is a multiple of 8, so a group of 4 never crosses a row: padding columns get zeros
            if (r < rows && c < plane_cols<KIND>(cols)) split_store<KIND, true>(out.hi, out.lo, r * out.ld + c, v[j], sc);
        }
        return;
    }
    __shared__ float tile[32][129];   // [column of X][row of X]
    const long long r0 = (long long)blockIdx.y * 128, c0 = (long long)blockIdx.x * 32;
    float x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const long long r = r0 + warp + 8 * i, c = c0 + lane;
        x[i] = (r < rows && c < cols) ? X[r * ldx + c] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) tile[lane][warp + 8 * i] = x[i];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int g = tid + 256 * j;   // plane row g / 32 (a column of X), 4 consecutive plane columns
        const int a = g >> 5, q = (g & 31) * 4;
        const long long orow = c0 + a, ocol = r0 + q;
        if (orow < cols && ocol < plane_cols<KIND>(rows)) {
            const float4 v = make_float4(tile[a][q], tile[a][q + 1], tile[a][q + 2], tile[a][q + 3]);
            split_store<KIND>(out.hi, out.lo, orow * out.ld + ocol, v, sc);
        }
    }
}

// ---------------------------------------------------------------- two levels at once
// The 7 children of an operand from its 4 quadrants, in product order, with
// the same fp32 operations as pre_add_kernel (A: S1..S4; B^T: T1..T4).
template <int SIDE_B>
__device__ __forceinline__ void children7(const float4 (&Q)[4], float4 (&ch)[7]) {
    float4 X1, X2, X3, X4;
    if (!SIDE_B) {
        X1 = add4(Q[2], Q[3]); X2 = sub4(X1, Q[0]); X3 = sub4(Q[0], Q[2]); X4 = sub4(Q[1], X2);
    } else {
        X1 = sub4(Q[2], Q[0]); X2 = sub4(Q[3], X1); X3 = sub4(Q[3], Q[2]); X4 = sub4(X2, Q[1]);
    }
    ch[0] = Q[0]; ch[1] = Q[1];
    ch[2] = SIDE_B ? Q[3] : X4;
    ch[3] = SIDE_B ? X4 : Q[3];
    ch[4] = X1; ch[5] = X2; ch[6] = X3;
}

// 4 consecutive elements at (row, col) of a view, zero outside its valid window.
__device__ __forceinline__ float4 load_sub(const View& v, bool vec, long long row, long long col) {
    if (vec && row < v.valid_rows && col + 3 < v.valid_cols)
        return __ldg(reinterpret_cast<const float4*>(v.ptr + row * v.ld + col));
    float t[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) t[j] = (row < v.valid_rows && col + j < v.valid_cols) ? __ldg(v.ptr + row * v.ld + col + j) : 0.0f;
    return f4(t[0], t[1], t[2], t[3]);
}

// Child i (product order) of an operand from its four quadrants: the fp32
// operations of children7 computing only that child.
template <int SIDE_B>
__device__ __forceinline__ float4 child_of4(int i, float4 Q0, float4 Q1, float4 Q2, float4 Q3) {
    if (!SIDE_B) {
        switch (i) {
            case 0: return Q0;
            case 1: return Q1;
            case 2: return sub4(Q1, sub4(add4(Q2, Q3), Q0));   // S4 = Q1 - S2
            case 3: return Q3;
            case 4: return add4(Q2, Q3);                       // S1
            case 5: return sub4(add4(Q2, Q3), Q0);             // S2 = S1 - Q0
            default: return sub4(Q0, Q2);                      // S3
        }
    }
    switch (i) {
        case 0: return Q0;
        case 1: return Q1;
        case 2: return Q3;
        case 3: return sub4(sub4(Q3, sub4(Q2, Q0)), Q1);       // T4 = T2 - Q1, T2 = Q3 - T1
        case 4: return sub4(Q2, Q0);                           // T1
        case 5: return sub4(Q3, sub4(Q2, Q0));                 // T2
        default: return sub4(Q3, Q2);                          // T3
    }
}

// The 7^D children of one position (4 consecutive columns) of an operand's 2^D x 2^D
// sub-blocks X, split into planes from element offset o0 on, in product order.
template <int D, int SIDE_B, int KIND>
__device__ __forceinline__ void emit_children(const float4 (&X)[1 << D][1 << D], const Stack16& out, long long o0,
                                              float sc) {
    if constexpr (D == 1) {
        const float4 Q[4] = {X[0][0], X[0][1], X[1][0], X[1][1]};
        float4 ch[7];
        children7<SIDE_B>(Q, ch);
#pragma unroll
        for (int i = 0; i < 7; ++i) split_store<KIND>(out.hi, out.lo, o0 + i * out.child_stride, ch[i], sc);
    } else {
#pragma unroll 1
        for (int i = 0; i < 7; ++i) {
            float4 Q[4], ch[7];   // child i's quadrants, its children
#pragma unroll
            for (int q = 0; q < 4; ++q)
                Q[q] = child_of4<SIDE_B>(i, X[q >> 1][q & 1], X[q >> 1][2 + (q & 1)], X[2 + (q >> 1)][q & 1],
                                         X[2 + (q >> 1)][2 + (q & 1)]);
            children7<SIDE_B>(Q, ch);
#pragma unroll
            for (int j = 0; j < 7; ++j)
                split_store<KIND>(out.hi, out.lo, o0 + (i * 7 + j) * out.child_stride, ch[j], sc);
        }
    }
}

// Pre-additions of a whole depth-1 or depth-2 recursion, both sides in one launch:
// the caller's A (a view of 2^D h x 2^D w positions, zero outside its valid window)
// and row-major B (valid K x N, zero outside) -> the 7^D leaf operands of A and of
// B^T as split planes; the fp32 operations are those of one pass per level, and no
// level between is stored.
//   A blocks (the first a_blocks): a thread takes 4 consecutive columns of one leaf
//     row, 16-byte loads and stores.
//   B blocks: leaf position (n, k) of B^T sub-block (a, b) is B[b w + k][a h + n].
//     A block takes 16 (n) x 32 (k) positions, stages the sub-blocks' 32 rows x 64
//     bytes in shared memory (every load before the first store; 17 floats a row:
//     the reads are free of bank conflicts) and then, like an A thread, holds 4
//     consecutive k of one n and stores along k.
// Bound: HBM writes.  n = 8192, depth 2, FP32: both sides 606 us (3.83 GB, 3.29 of
// them written: 6.3 TB/s), against 284 + 334 us for one launch per side whose B pass
// turned each group of seven outputs through shared memory; n = 4096, depth 1: 43 +
// 49 -> 86 us; n = 1024, depth 2: 8.3 + 15.4 -> 11.5 us.
constexpr int kRootN = 16, kRootK = 32, kRootPitch = kRootN + 1;
struct RootB {
    const float* ptr;
    long long ld, K, N, h, w;   // valid K x N; leaf h (n) x w (k)
};
template <int D, int KIND>
__global__ void __launch_bounds__(128) pre_root_kernel(View P, long long h, long long w, Stack16 sa, RootB Bm, Stack16 sb,
                                                       long long a_blocks, long long tiles_n,
                                                       const float* __restrict__ scale) {
    dep_trigger();
    constexpr int S = 1 << D;
    __shared__ float tile[S * S][kRootK][kRootPitch];
    const int t = threadIdx.x;
    float4 X[S][S];
    if ((long long)blockIdx.x < a_blocks) {
        const bool vec = (reinterpret_cast<uintptr_t>(P.ptr) & 15) == 0 && (P.ld & 3) == 0;
        const long long w4 = plane_cols<KIND>(w) >> 2, e = (long long)blockIdx.x * 128 + t, r = e / w4;
        const long long c = (e - r * w4) * 4;
        if (r >= h) return;
        if (c >= w) P.valid_rows = 0;   // padding columns of a tf32x plane: zeros
#pragma unroll
        for (int a = 0; a < S; ++a)
#pragma unroll
            for (int b = 0; b < S; ++b) X[a][b] = load_sub(P, vec, a * h + r, b * w + c);
        emit_children<D, 0, KIND>(X, sa, r * sa.ld + c, scale ? scale[0] : 1.0f);
        return;
    }
    const long long blk = (long long)blockIdx.x - a_blocks;
    const long long n0 = blk % tiles_n * kRootN, k0 = blk / tiles_n * kRootK;
    const bool vec = (reinterpret_cast<uintptr_t>(Bm.ptr) & 15) == 0 && (Bm.ld & 3) == 0;
    // S * S sub-blocks x 32 rows x 4 groups of 4 floats over 128 threads
    float4 v[S * S];
#pragma unroll
    for (int j = 0; j < S * S; ++j) {
        const int kr = t >> 2, q = t & 3;              // sub-block j = S a + b
        const long long k = k0 + kr, n = n0 + 4 * q;   // h is a multiple of 4: n < h covers n + 3
        const long long row = (j % S) * Bm.w + k, col = (j / S) * Bm.h + n;
        v[j] = f4(0.f, 0.f, 0.f, 0.f);
        if (k < Bm.w && n < Bm.h && row < Bm.K && col < Bm.N) {
            const float* src = Bm.ptr + row * Bm.ld + col;
            if (vec && col + 3 < Bm.N) {
                v[j] = __ldg(reinterpret_cast<const float4*>(src));
            } else {
                v[j].x = __ldg(src);
                if (col + 1 < Bm.N) v[j].y = __ldg(src + 1);
                if (col + 2 < Bm.N) v[j].z = __ldg(src + 2);
                if (col + 3 < Bm.N) v[j].w = __ldg(src + 3);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < S * S; ++j) {
        float* d = &tile[j][t >> 2][4 * (t & 3)];
        d[0] = v[j].x; d[1] = v[j].y; d[2] = v[j].z; d[3] = v[j].w;
    }
    __syncthreads();
    const int nl = t >> 3, kq = (t & 7) * 4;
    const long long n = n0 + nl, k = k0 + kq;
    if (n >= Bm.h || k >= plane_cols<KIND>(Bm.w)) return;
#pragma unroll
    for (int a = 0; a < S; ++a)
#pragma unroll
        for (int b = 0; b < S; ++b)
            X[a][b] = f4(tile[a * S + b][kq][nl], tile[a * S + b][kq + 1][nl], tile[a * S + b][kq + 2][nl],
                         tile[a * S + b][kq + 3][nl]);
    emit_children<D, 1, KIND>(X, sb, n * sb.ld + k, scale ? scale[1] : 1.0f);
}

// Child i (product order) of an operand from its four quadrants, one element at
// a time: the same fp32 operations as children7 computing only that child.
template <int SIDE_B>
__device__ __forceinline__ float child_of1(int i, float Q0, float Q1, float Q2, float Q3) {
    if (!SIDE_B) {
        switch (i) {
            case 0: return Q0;
            case 1: return Q1;
            case 2: return Q1 - ((Q2 + Q3) - Q0);   // S4 = Q1 - S2
            case 3: return Q3;
            case 4: return Q2 + Q3;                 // S1
            case 5: return (Q2 + Q3) - Q0;          // S2 = S1 - Q0
            default: return Q0 - Q2;                // S3
        }
    }
    switch (i) {
        case 0: return Q0;
        case 1: return Q1;
        case 2: return Q3;
        case 3: return (Q3 - (Q2 - Q0)) - Q1;       // T4 = T2 - Q1, T2 = Q3 - T1
        case 4: return Q2 - Q0;                     // T1
        case 5: return Q3 - (Q2 - Q0);              // T2
        default: return Q3 - Q2;                    // T3
    }
}

// One value into the planes at element offset o (evict-first stores).
template <int KIND>
__device__ __forceinline__ void split_store1(void* hi_plane, void* lo_plane, long long o, float v, float sc) {
    if constexpr (KIND == kSplitTF32) {
        __stcs(static_cast<float*>(hi_plane) + o, v);
        __stcs(static_cast<float*>(lo_plane) + o, tf32_round_rne(v - tf32_trunc(v)));
        return;
    }
    const float x = v * sc;
    unsigned short h, l;
    if constexpr (KIND == kSplitBF16) {
        const __nv_bfloat16 a = __float2bfloat16_rn(x);
        const __nv_bfloat16 b = __float2bfloat16_rn(x - __bfloat162float(a));
        h = __bfloat16_as_ushort(a);
        l = __bfloat16_as_ushort(b);
    } else {
        const __half a = __float2half_rn(x);
        const __half b = __float2half_rn(x - __half2float(a));
        h = __half_as_ushort(a);
        l = __half_as_ushort(b);
    }
    __stcs(static_cast<unsigned short*>(hi_plane) + o, h);
    __stcs(static_cast<unsigned short*>(lo_plane) + o, l);
}

// Pre-additions of three consecutive levels in one pass (the whole recursion
// of a depth-3 plan): each node operand (8h x 8w, read through its view with
// zero outside the valid window) -> its 343 great-grandchildren (h x w), split
// planes at stack index node * 343 + (i * 7 + j) * 7 + l.  One element per
// thread: the node's 64 sub-block values are loaded once, level-1 child i's
// 4 x 4 sub-block values are formed from them, then level-2 child j's
// quadrants, then its 7 children; the fp32 operations are those of three
// pre_add passes.
template <int SIDE_B, int KIND>
__global__ void __launch_bounds__(256, 2) pre_add3_kernel(View P, long long h, long long w, Stack16 out,
                                                       const float* scale, int dep) {
    if (dep) dep_start();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= w) return;
    const float sc = scale ? scale[SIDE_B] : 1.0f;
    const long long node = blockIdx.z;
    const float* base = P.ptr + node * P.node_stride;
    for (long long r = blockIdx.y; r < h; r += gridDim.y) {
        const long long o0 = (node * 343) * out.child_stride + r * out.ld + c;
        float X[8][8];   // sub-block (a, b) of the node
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) {
                const long long row = a * h + r, col = b * w + c;
                X[a][b] = (row < P.valid_rows && col < P.valid_cols) ? base[row * P.ld + col] : 0.0f;
            }
#pragma unroll 1
        for (int i = 0; i < 7; ++i) {
            float Y[4][4];   // level-1 child i, sub-block (a, b)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    Y[a][b] = child_of1<SIDE_B>(i, X[a][b], X[a][4 + b], X[4 + a][b], X[4 + a][4 + b]);
#pragma unroll 1
            for (int j = 0; j < 7; ++j) {
                float Cj[4];   // level-2 child (i, j), quadrant t
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    Cj[t] = child_of1<SIDE_B>(j, Y[(t >> 1)][(t & 1)], Y[(t >> 1)][2 + (t & 1)],
                                              Y[2 + (t >> 1)][(t & 1)], Y[2 + (t >> 1)][2 + (t & 1)]);
#pragma unroll
                for (int l = 0; l < 7; ++l)
                    split_store1<KIND>(out.hi, out.lo, o0 + (i * 49 + j * 7 + l) * out.child_stride,
                                       child_of1<SIDE_B>(l, Cj[0], Cj[1], Cj[2], Cj[3]), sc);
            }
        }
    }
}

// Root B side of a depth-3 plan in one pass, straight from the caller's
// row-major B (valid K x N, zero outside) into the 343 leaf operands of B^T,
// split into planes.  Leaf position (n, k) of B^T sub-block (a, b) is
// B[b * w + k][a * h + n] (h = N0 / 8, w = K0 / 8).  A block takes an 8 (n) x
// 32 (k) patch of positions: it stages the 64 sub-block tiles of B that the
// patch needs (32 rows of k by 8 columns of n, one 32-byte sector per row) in
// shared memory, every load issued before the first store; each thread then
// reads its position's 64 values from there (rows padded to 9 floats, so the
// 32 lanes of a warp -- 32 consecutive k -- hit 32 banks) and runs
// pre_add3_kernel's chain, its leaf stores running along k, coalesced.  The
// fp32 operations are those of pre_add3_kernel<1> on a transposed copy.
constexpr int kBtN = 8, kBtK = 32, kBtPitch = 9;
constexpr size_t kBtSmem = (size_t)64 * kBtK * kBtPitch * sizeof(float);   // 73,728 bytes

template <int KIND>
__global__ void __launch_bounds__(256, 2) pre_add3_bt_kernel(const float* B, long long ldb, long long K,
                                                          long long N, long long h, long long w, long long tiles_n,
                                                          Stack16 out, const float* scale) {
    dep_start();
    extern __shared__ float bt_tile[];   // [64 sub-blocks][kBtK rows of k][kBtPitch]
    const float sc = scale ? scale[1] : 1.0f;
    const int t = threadIdx.x;
    const long long n0 = (long long)(blockIdx.x % tiles_n) * kBtN, k0 = (long long)(blockIdx.x / tiles_n) * kBtK;
    const bool vec = (reinterpret_cast<uintptr_t>(B) & 15) == 0 && (ldb & 3) == 0;
    // 64 tiles x 32 rows x 2 float4 = 4096 float4, 16 per thread
    float4 v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int L = t + 256 * j;   // sub-block L / 64 = 8 a + b, row (L % 64) / 2, half L % 2
        const int ab = L >> 6, kr = (L & 63) >> 1, q = L & 1;
        const long long k = k0 + kr, n = n0 + 4 * q;   // h is a multiple of 4: n < h covers n + 3
        const long long row = (ab & 7) * w + k, col = (ab >> 3) * h + n;
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < w && n < h && row < K && col < N) {
            const float* src = B + row * ldb + col;
            if (vec && col + 3 < N) {
                v[j] = *reinterpret_cast<const float4*>(src);
            } else {
                v[j].x = *src;
                if (col + 1 < N) v[j].y = src[1];
                if (col + 2 < N) v[j].z = src[2];
                if (col + 3 < N) v[j].w = src[3];
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int L = t + 256 * j;
        float* d = bt_tile + ((L >> 6) * kBtK + ((L & 63) >> 1)) * kBtPitch + 4 * (L & 1);
        d[0] = v[j].x; d[1] = v[j].y; d[2] = v[j].z; d[3] = v[j].w;
    }
    __syncthreads();
    const int tn = t >> 5, tk = t & 31;
    const long long n = n0 + tn, k = k0 + tk;
    if (n >= h || k >= w) return;
    float X[8][8];   // sub-block (a, b) of B^T at position (n, k)
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) X[a][b] = bt_tile[((a * 8 + b) * kBtK + tk) * kBtPitch + tn];
    const long long o0 = n * out.ld + k;
#pragma unroll 1
    for (int i = 0; i < 7; ++i) {
        float Y[4][4];   // level-1 child i, sub-block (a, b)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) Y[a][b] = child_of1<1>(i, X[a][b], X[a][4 + b], X[4 + a][b], X[4 + a][4 + b]);
#pragma unroll 1
        for (int j = 0; j < 7; ++j) {
            float Cj[4];   // level-2 child (i, j), quadrant t
#pragma unroll
            for (int q = 0; q < 4; ++q)
                Cj[q] = child_of1<1>(j, Y[(q >> 1)][(q & 1)], Y[(q >> 1)][2 + (q & 1)], Y[2 + (q >> 1)][(q & 1)],
                                     Y[2 + (q >> 1)][2 + (q & 1)]);
#pragma unroll
            for (int l = 0; l < 7; ++l)
                split_store1<KIND>(out.hi, out.lo, o0 + (i * 49 + j * 7 + l) * out.child_stride,
                                   child_of1<1>(l, Cj[0], Cj[1], Cj[2], Cj[3]), sc);
        }
    }
}

// Post-additions of two consecutive levels in one pass: for each node, its 49
// grandchild products P[(node * 7 + i) * 7 + j] (h x w, row stride ld_in) ->
// the node output (4h x 4w).  The children's quadrant values are formed with
// the same U-chain as post_add_kernel, then the node's; results are identical
// to two post_add passes and the middle level is never stored.
__device__ __forceinline__ float uchain_quadrant(int q, float P1, float P2, float P3, float P4, float P5, float P6,
                                                 float P7) {
    if (q == 0) return P1 + P2;                               // U1
    const float U2 = P1 + P6;
    if (q == 1) return (U2 + P5) + P3;                        // U5 = U4 + P3, U4 = U2 + P5
    const float U3 = U2 + P7;
    if (q == 2) return U3 - P4;                               // U6
    return U3 + P5;                                           // U7
}

// One element per thread: the 49 products of a position are loaded once.
// ROOT: out is the caller's C: alpha / beta and the valid window apply.
template <bool ROOT>
__global__ void __launch_bounds__(128) post_add2_kernel(const float* P, long long ld_in, long long cs,
                                                        long long h, long long w, float* __restrict__ out, long long ld_out,
                                                        long long out_ns, long long valid_rows, long long valid_cols,
                                                        float alpha, float beta) {
    dep_start();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= w) return;
    const long long node = blockIdx.z;
    const float* base = P + node * 49 * cs;
    float* o = out + node * out_ns;
    for (long long r = blockIdx.y; r < h; r += gridDim.y) {
        const float* pr = base + r * ld_in + c;
        float p[7][7];
#pragma unroll
        for (int i = 0; i < 7; ++i)
#pragma unroll
            for (int j = 0; j < 7; ++j) p[i][j] = pr[(i * 7 + j) * cs];
#pragma unroll
        for (int t = 0; t < 4; ++t) {            // sub-quadrant of every child quadrant
            float Ct[7];                          // child i's quadrant t
#pragma unroll
            for (int i = 0; i < 7; ++i)
                Ct[i] = uchain_quadrant(t, p[i][0], p[i][1], p[i][2], p[i][3], p[i][4], p[i][5], p[i][6]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {        // node quadrant q, its sub-quadrant t
                const long long rr = (long long)((q >> 1) * 2 + (t >> 1)) * h + r;
                const long long cc = (long long)((q & 1) * 2 + (t & 1)) * w + c;
                const float v = uchain_quadrant(q, Ct[0], Ct[1], Ct[2], Ct[3], Ct[4], Ct[5], Ct[6]);
                if (!ROOT) {
                    o[rr * ld_out + cc] = v;
                } else if (rr < valid_rows && cc < valid_cols) {
                    float* dst = o + rr * ld_out + cc;
                    *dst = (beta != 0.0f) ? alpha * v + beta * *dst : alpha * v;
                }
            }
        }
    }
}

// Post-additions of three consecutive levels in one pass (the whole recursion
// of a depth-3 plan, ROOT) or of a node's bottom three levels: for each node,
// its 343 great-grandchild products P[node * 343 + (i * 7 + j) * 7 + l] (h x w,
// row stride ld_in) -> the node output (8h x 8w).  One element per thread,
// every product loaded once.  Level-2 outputs (the U-chain over l), then each
// level-1 child's 16 values (the U-chain over j), then the node's 64 values
// (the U-chain over i): the fp32 operations of three post_add passes.
//
// The level-1 children are visited in the order P1, P6, P7, P5, P3, P4, P2, in
// which the node's U-chain needs them; the chain keeps three running values per
// position (P1, U2 then U4, U3) and each node quadrant is stored as soon as it
// is final (C22 = U7 after P5, C12 = U5 after P3, C21 = U6 after P4, C11 = U1
// after P2).  48 live values instead of the seven children's 112 leave room
// for four blocks per SM, i.e. twice the loads in flight.

// Level-1 child I's 16 values at (quadrant q1, sub-quadrant q2): o1[q1 * 4 + q2].
template <int I>
__device__ __forceinline__ void post3_child(const float* pr, long long cs, float (&o1)[16]) {
    float o2[7][4];   // level-2 child (I, j), quadrant q2
#pragma unroll
    for (int j = 0; j < 7; ++j) {
        float p[7];
#pragma unroll
        for (int l = 0; l < 7; ++l) p[l] = pr[((I * 7 + j) * 7 + l) * cs];
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) o2[j][q2] = uchain_quadrant(q2, p[0], p[1], p[2], p[3], p[4], p[5], p[6]);
    }
#pragma unroll
    for (int q1 = 0; q1 < 4; ++q1)
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2)
            o1[q1 * 4 + q2] = uchain_quadrant(q1, o2[0][q2], o2[1][q2], o2[2][q2], o2[3][q2], o2[4][q2], o2[5][q2],
                                              o2[6][q2]);
}

template <bool ROOT>
__global__ void __launch_bounds__(128, 4) post_add3_kernel(const float* P, long long ld_in, long long cs,
                                                        long long h, long long w, float* __restrict__ out, long long ld_out,
                                                        long long out_ns, long long valid_rows, long long valid_cols,
                                                        float alpha, float beta) {
    dep_start();
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= w) return;
    const long long node = blockIdx.z;
    const float* base = P + node * 343 * cs;
    float* o = out + node * out_ns;
    for (long long r = blockIdx.y; r < h; r += gridDim.y) {
        const float* pr = base + r * ld_in + c;
        // node quadrant q0 at position s = (q1, q2)
        auto put = [&](int q0, int s, float v) {
            const int q1 = s >> 2, q2 = s & 3;
            const long long rr = (long long)(4 * (q0 >> 1) + 2 * (q1 >> 1) + (q2 >> 1)) * h + r;
            const long long cc = (long long)(4 * (q0 & 1) + 2 * (q1 & 1) + (q2 & 1)) * w + c;
            if (!ROOT) {
                o[rr * ld_out + cc] = v;
            } else if (rr < valid_rows && cc < valid_cols) {
                float* dst = o + rr * ld_out + cc;
                *dst = (beta != 0.0f) ? alpha * v + beta * *dst : alpha * v;
            }
        };
        float o1[16], a1[16], u2[16], u3[16];
        post3_child<0>(pr, cs, o1);                                  // P1
#pragma unroll
        for (int s = 0; s < 16; ++s) a1[s] = o1[s];
        post3_child<5>(pr, cs, o1);                                  // P6: U2 = P1 + P6
#pragma unroll
        for (int s = 0; s < 16; ++s) u2[s] = a1[s] + o1[s];
        post3_child<6>(pr, cs, o1);                                  // P7: U3 = U2 + P7
#pragma unroll
        for (int s = 0; s < 16; ++s) u3[s] = u2[s] + o1[s];
        post3_child<4>(pr, cs, o1);                                  // P5: U4 = U2 + P5, C22 = U7 = U3 + P5
#pragma unroll
        for (int s = 0; s < 16; ++s) {
            u2[s] = u2[s] + o1[s];
            put(3, s, u3[s] + o1[s]);
        }
        post3_child<2>(pr, cs, o1);                                  // P3: C12 = U5 = U4 + P3
#pragma unroll
        for (int s = 0; s < 16; ++s) put(1, s, u2[s] + o1[s]);
        post3_child<3>(pr, cs, o1);                                  // P4: C21 = U6 = U3 - P4
#pragma unroll
        for (int s = 0; s < 16; ++s) put(2, s, u3[s] - o1[s]);
        post3_child<1>(pr, cs, o1);                                  // P2: C11 = U1 = P1 + P2
#pragma unroll
        for (int s = 0; s < 16; ++s) put(0, s, a1[s] + o1[s]);
    }
}

// Split jobs of a batched launch: one 32 x 128 block of the source per CTA
// (jobs found by binary search on their first block).  Every thread issues all
// of its loads before its first store.  Untransposed jobs go straight from
// 16-byte loads to the planes (a warp covers 512 contiguous bytes of a row);
// transposed jobs stage the block in a 32 x 129 shared tile (conflict-free both
// ways) and leave it as 128 rows of 32 elements.
//
// KIND tf32x: jobs of both FP32 plane forms, by SplitJob::corr16.
template <int KIND>
__global__ void __launch_bounds__(256) batched_split_kernel(const SplitJob* __restrict__ jobs, int njobs) {
    __shared__ float tile[32][129];
    const long long t = blockIdx.x;
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].tile_begin <= t) lo = mid; else hi = mid - 1;
    }
    const SplitJob J = jobs[lo];
    const float sc = J.scale ? J.scale[J.transpose] : 1.0f;
    const long long local = t - J.tile_begin;
    const long long r0 = (local / J.tiles_c) * 32, c0 = (local % J.tiles_c) * 128;
    const int tid = threadIdx.y * 32 + threadIdx.x;
    if (!J.transpose) {
        const bool vec = (reinterpret_cast<uintptr_t>(J.src) & 15) == 0 && (J.lds & 3) == 0;
        float4 v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int g = tid + 256 * j;   // row g / 32 of the block, columns 4 (g % 32) .. + 3
            const long long r = r0 + (g >> 5), c = c0 + 4 * (g & 31);
            v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r >= J.rows || c >= J.cols) continue;
            const float* src = J.src + r * J.lds + c;
            if (vec && c + 3 < J.cols) {
                v[j] = __ldg(reinterpret_cast<const float4*>(src));
            } else {
                v[j].x = __ldg(src);
                if (c + 1 < J.cols) v[j].y = __ldg(src + 1);
                if (c + 2 < J.cols) v[j].z = __ldg(src + 2);
                if (c + 3 < J.cols) v[j].w = __ldg(src + 3);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int g = tid + 256 * j;
            const long long r = r0 + (g >> 5), c = c0 + 4 * (g & 31);
            // ld is a multiple of 8, so a group of 4 never crosses a row: padding columns get zeros
            if (KIND == kSplitTF32X && !J.corr16) {
                if (r < J.rows && c < J.cols) split_store<kSplitTF32>(J.dst, J.lo, r * J.ldd + c, v[j], sc);
            } else if (r < J.rows && c < plane_cols<KIND>(J.cols)) {
                split_store<KIND, true>(J.dst, J.lo, r * J.ldd + c, v[j], sc);
            }
        }
        return;
    }
    // source rows r0 + i (i = warp + 8 s), columns c0 + lane + 32 q
    const int lane = threadIdx.x, warp = threadIdx.y;
    float x[4][4];
#pragma unroll
    for (int sI = 0; sI < 4; ++sI)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const long long r = r0 + warp + 8 * sI, c = c0 + lane + 32 * q;
            x[sI][q] = (r < J.rows && c < J.cols) ? __ldg(J.src + r * J.lds + c) : 0.0f;
        }
#pragma unroll
    for (int sI = 0; sI < 4; ++sI)
#pragma unroll
        for (int q = 0; q < 4; ++q) tile[warp + 8 * sI][lane + 32 * q] = x[sI][q];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int g = tid + 256 * j;   // output row a (a source column), 4 consecutive output columns
        const int a = g >> 3, q = (g & 7) * 4;
        const long long orow = c0 + a, ocol = r0 + q;
        if (orow < J.cols && ocol < plane_cols<KIND>(J.rows)) {
            const float4 v = make_float4(tile[q][a], tile[q + 1][a], tile[q + 2][a], tile[q + 3][a]);
            if (KIND == kSplitTF32X && !J.corr16) {
                if (ocol < J.rows) split_store<kSplitTF32>(J.dst, J.lo, orow * J.ldd + ocol, v, sc);
            } else {
                split_store<KIND>(J.dst, J.lo, orow * J.ldd + ocol, v, sc);
            }
        }
    }
}

inline unsigned gy(long long rows) { return (unsigned)(rows < 65535 ? (rows > 0 ? rows : 1) : 65535); }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace

cudaError_t launch_pre_add(const View& parent, long long nodes, const Stack& out, int side_b, int full,
                           cudaStream_t stream) {
    const long long h = parent.rows / 2, w = parent.cols / 2;
    if (h <= 0 || w <= 0 || nodes <= 0) return cudaSuccess;
    const bool vec = aligned16(parent.ptr) && aligned16(out.ptr) && parent.ld % 4 == 0 && w % 4 == 0 &&
                     parent.node_stride % 4 == 0 && out.ld % 4 == 0 && out.child_stride % 4 == 0;
    dim3 grid((unsigned)((w + 4 * 128 - 1) / (4 * 128)), gy(h), (unsigned)nodes);
    // dependent on the pass before it while a row keeps two warps busy, or all blocks run at
    // once; many blocks of less work pay more for the wait than it hides (5700 x 4441 x 312,
    // TF32, depth 3, rows of 160, 80 and 40: pre-additions 74 us in plain order, 102 dependent;
    // n = 1500, depth 2, rows of 752 and 376: 31 and 26; 520 x 292 x 152, depth 2, a call 24, 20)
    const int dep = w >= 256 || (long long)grid.x * grid.y * grid.z <= 2048;
#define FMM_PRE(V, S, F)                                                                              \
    if (dep) launch_dep(pre_add_kernel<V, S, F>, grid, 128, 0, stream, parent, h, w, out, 1);           \
    else pre_add_kernel<V, S, F><<<grid, 128, 0, stream>>>(parent, h, w, out, 0)
    if (vec) {
        if (side_b) { if (full) { FMM_PRE(true, 1, true); } else { FMM_PRE(true, 1, false); } }
        else        { if (full) { FMM_PRE(true, 0, true); } else { FMM_PRE(true, 0, false); } }
    } else {
        if (side_b) { if (full) { FMM_PRE(false, 1, true); } else { FMM_PRE(false, 1, false); } }
        else        { if (full) { FMM_PRE(false, 0, true); } else { FMM_PRE(false, 0, false); } }
    }
#undef FMM_PRE
    return cudaGetLastError();
}

cudaError_t launch_pre_add_b_root(const float* B, long long ldb, long long K, long long N, long long kh,
                                  long long nh, const Stack& out, int full, cudaStream_t stream) {
    if (kh <= 0 || nh <= 0) return cudaSuccess;
    dim3 grid((unsigned)((nh + 31) / 32), (unsigned)((kh + 31) / 32));
    dim3 block(32, 8);
    if (full) launch_dep(pre_add_b_root_kernel<true>, grid, block, 0, stream, B, ldb, K, N, kh, nh, out);
    else launch_dep(pre_add_b_root_kernel<false>, grid, block, 0, stream, B, ldb, K, N, kh, nh, out);
    return cudaGetLastError();
}

cudaError_t launch_post_add(const float* P, long long ld_in, long long child_stride, long long nodes, long long h,
                            long long w, float* out, long long ld_out, long long out_node_stride,
                            long long valid_rows, long long valid_cols, float alpha, float beta,
                            cudaStream_t stream) {
    if (h <= 0 || w <= 0 || nodes <= 0) return cudaSuccess;
    const bool root = valid_rows >= 0;
    const bool vec = aligned16(P) && ld_in % 4 == 0 && child_stride % 4 == 0 && w % 4 == 0 &&
                     (root || (aligned16(out) && ld_out % 4 == 0 && out_node_stride % 4 == 0));
    dim3 grid((unsigned)((w + 4 * 128 - 1) / (4 * 128)), gy(h), (unsigned)nodes);
#define FMM_POST(V, R)                                                                                         \
    launch_dep(post_add_kernel<V, R>, grid, 128, 0, stream, P, ld_in, child_stride, h, w, out, ld_out, out_node_stride, \
                                                   valid_rows, valid_cols, alpha, beta)
    if (root) { if (vec) FMM_POST(true, true); else FMM_POST(false, true); }
    else      { if (vec) FMM_POST(true, false); else FMM_POST(false, false); }
#undef FMM_POST
    return cudaGetLastError();
}

cudaError_t launch_transpose(const float* B, long long ldb, long long K, long long N, float* Bt, long long ldt,
                             cudaStream_t stream, long long rows_out, long long cols_out) {
    if (rows_out < 0) rows_out = N;
    if (cols_out < 0) cols_out = K;
    if (rows_out <= 0 || cols_out <= 0) return cudaSuccess;
    dim3 grid((unsigned)((rows_out + 31) / 32), (unsigned)((cols_out + 127) / 128));
    launch_dep(transpose_kernel, grid, dim3(32, 8), 0, stream, B, ldb, K, N, Bt, ldt, rows_out, cols_out);
    return cudaGetLastError();
}

cudaError_t launch_copy2d(const float* A, long long lda, long long M, long long K, float* dst, long long ldd,
                          cudaStream_t stream) {
    if (M <= 0 || K <= 0) return cudaSuccess;
    dim3 grid((unsigned)((K + 255) / 256), gy(M));
    launch_dep(copy2d_kernel, grid, 256, 0, stream, A, lda, M, K, dst, ldd);
    return cudaGetLastError();
}

cudaError_t launch_batched_copy(const CopyJob* jobs, int njobs, long long total_tiles, cudaStream_t stream) {
    if (njobs <= 0 || total_tiles <= 0) return cudaSuccess;
    batched_copy_kernel<<<(unsigned)total_tiles, dim3(32, 8), 0, stream>>>(jobs, njobs);
    return cudaGetLastError();
}

cudaError_t launch_fp16_scales(const float* A, long long lda, long long M, long long K, const float* B,
                               long long ldb, long long N, float bound_mult, float* scale, unsigned* scratch,
                               cudaStream_t stream) {
    cudaError_t e = cudaMemsetAsync(scratch, 0, 2 * sizeof(unsigned), stream);
    if (e != cudaSuccess) return e;
    auto operand = [](const float* X, long long ld, long long rows, long long cols) {
        const long long tc = (cols + 127) / 128;
        return MaxOperand{X, ld, rows, cols, tc > 0 ? tc : 1, tc * ((rows + 31) / 32)};
    };
    const MaxOperand a = operand(A, lda, M, K), b = operand(B, ldb, K, N);
    const long long most = (a.tiles > b.tiles ? a.tiles : b.tiles);
    const long long grid = (most + 1) / 2 < 152 * 8 ? (most + 1) / 2 : 152 * 8;
    if (grid > 0) absmax_kernel<<<(unsigned)grid, 256, 0, stream>>>(a, b, scratch);
    launch_dep(fp16_scale_kernel, 1, 32, 0, stream, scratch, bound_mult, scale);
    return cudaGetLastError();
}

cudaError_t launch_quad_pre(const QuadPre& q, QuadSums sums, cudaStream_t stream) {
    if (q.h <= 0 || q.w <= 0) return cudaSuccess;
    dim3 grid((unsigned)((q.w + 511) / 512), gy(q.h));
    switch (sums) {
        case kQuadS123: quad_pre_kernel<kQuadS123><<<grid, 128, 0, stream>>>(q); break;
        case kQuadS4: quad_pre_kernel<kQuadS4><<<grid, 128, 0, stream>>>(q); break;
        case kQuadT1: quad_pre_kernel<kQuadT1><<<grid, 128, 0, stream>>>(q); break;
        case kQuadT23: quad_pre_kernel<kQuadT23><<<grid, 128, 0, stream>>>(q); break;
        case kQuadT4: quad_pre_kernel<kQuadT4><<<grid, 128, 0, stream>>>(q); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_quad_post(const QuadPost& q, int part, cudaStream_t stream) {
    if (q.h <= 0 || q.w <= 0) return cudaSuccess;
    dim3 grid((unsigned)((q.w + 511) / 512), gy(q.h));
    switch (part) {
        case 0: quad_post_kernel<0><<<grid, 128, 0, stream>>>(q); break;
        case 1: quad_post_kernel<1><<<grid, 128, 0, stream>>>(q); break;
        case 2: quad_post_kernel<2><<<grid, 128, 0, stream>>>(q); break;
        case 3: quad_post_kernel<3><<<grid, 128, 0, stream>>>(q); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_split16(const float* X, long long ldx, long long rows, long long cols, const Stack16& out,
                           int transpose, int kind, const float* scale, int which, cudaStream_t stream) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    // plain: 32 x 128 blocks; transposed: 128 (row) x 32 (column) blocks
    const dim3 grid = transpose ? dim3((unsigned)((cols + 31) / 32), (unsigned)((rows + 127) / 128))
                                : dim3((unsigned)((cols + 127) / 128), (unsigned)((rows + 31) / 32));
#define FMM_SPLIT(K, T) launch_dep(split16_kernel<K, T>, grid, dim3(32, 8), 0, stream, X, ldx, rows, cols, out, scale, which)
#define FMM_SPLITK(T)                                   \
    switch (kind) {                                      \
        case kSplitBF16: FMM_SPLIT(kSplitBF16, T); break; \
        case kSplitFP16: FMM_SPLIT(kSplitFP16, T); break; \
        case kSplitTF32X: FMM_SPLIT(kSplitTF32X, T); break; \
        default: FMM_SPLIT(kSplitTF32, T); break;         \
    }
    if (transpose) { FMM_SPLITK(true) } else { FMM_SPLITK(false) }
#undef FMM_SPLITK
#undef FMM_SPLIT
    return cudaGetLastError();
}

template <int D>
static cudaError_t launch_pre_root_impl(const View& a, const float* B, long long ldb, long long K, long long N,
                                        long long hb, const Stack16& sa, const Stack16& sb, int kind,
                                        const float* scale, cudaStream_t stream) {
    const long long h = a.rows >> D, w = a.cols >> D;
    if (h <= 0 || w <= 0 || hb <= 0) return cudaSuccess;
    if (w % 4 || hb % 4) return cudaErrorInvalidValue;
    const long long wp = kind == kSplitTF32X ? (w + 31) & ~31LL : w;
    const long long a_blocks = (h * (wp / 4) + 127) / 128, tiles_n = (hb + kRootN - 1) / kRootN;
    const long long blocks = a_blocks + tiles_n * ((w + kRootK - 1) / kRootK);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const RootB b{B, ldb, K, N, hb, w};
    // launched in plain stream order: resident beside the previous call's last pass its
    // blocks cost more than their launch (n = 1024, depth 2 in a row: 43.7 against 36.7 us)
#define FMM_ROOT(KIND_) \
    pre_root_kernel<D, KIND_><<<(unsigned)blocks, 128, 0, stream>>>(a, h, w, sa, b, sb, a_blocks, tiles_n, scale)
    switch (kind) {
        case kSplitBF16: FMM_ROOT(kSplitBF16); break;
        case kSplitFP16: FMM_ROOT(kSplitFP16); break;
        case kSplitTF32X: FMM_ROOT(kSplitTF32X); break;
        default: FMM_ROOT(kSplitTF32); break;
    }
#undef FMM_ROOT
    return cudaGetLastError();
}

cudaError_t launch_pre_root(int depth, const View& a, const float* B, long long ldb, long long K, long long N,
                            long long hb, const Stack16& sa, const Stack16& sb, int kind, const float* scale,
                            cudaStream_t stream) {
    if (depth == 1) return launch_pre_root_impl<1>(a, B, ldb, K, N, hb, sa, sb, kind, scale, stream);
    if (depth == 2) return launch_pre_root_impl<2>(a, B, ldb, K, N, hb, sa, sb, kind, scale, stream);
    return cudaErrorInvalidValue;
}

cudaError_t launch_pre_add3(const View& node, long long nodes, const Stack16& out, int side_b, int kind,
                            const float* scale, cudaStream_t stream) {
    const long long h = node.rows / 8, w = node.cols / 8;
    if (h <= 0 || w <= 0 || nodes <= 0) return cudaSuccess;
    dim3 grid((unsigned)((w + 255) / 256), gy(h), (unsigned)nodes);
    // in plain order, as pre_root (n = 2048, depth 3 176 -> 170 us, 269 x 277 x 3195 98 -> 82,
    // with the leaf launch's end, ptx.cuh), but for a handful of blocks (173 x 232 x 1220, 22
    // of them, 63.5 -> 61.5)
    const int dep = (long long)grid.x * grid.y * grid.z <= 24;
#define FMM_PRE3(S, K)                                                                                      \
    if (dep) launch_dep(pre_add3_kernel<S, K>, grid, 256, 0, stream, node, h, w, out, scale, 1);              \
    else pre_add3_kernel<S, K><<<grid, 256, 0, stream>>>(node, h, w, out, scale, 0)
#define FMM_PRE3K(S)                                        \
    switch (kind) {                                          \
        case kSplitBF16: FMM_PRE3(S, kSplitBF16); break;    \
        case kSplitFP16: FMM_PRE3(S, kSplitFP16); break;    \
        default: FMM_PRE3(S, kSplitTF32); break;            \
    }
    if (side_b) { FMM_PRE3K(1) } else { FMM_PRE3K(0) }
#undef FMM_PRE3K
#undef FMM_PRE3
    return cudaGetLastError();
}

template <int KIND>
static cudaError_t launch_pre_add3_bt_impl(const float* B, long long ldb, long long K, long long N, long long h,
                                           long long w, const Stack16& out, const float* scale,
                                           cudaStream_t stream) {
    // once per device and instantiation (keeps later launches free of other API calls)
    static bool attr_done[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        e = cudaFuncSetAttribute(pre_add3_bt_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBtSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    const long long tiles_n = (h + kBtN - 1) / kBtN, tiles = tiles_n * ((w + kBtK - 1) / kBtK);
    launch_dep(pre_add3_bt_kernel<KIND>, (unsigned)tiles, 256, kBtSmem, stream, B, ldb, K, N, h, w, tiles_n, out, scale);
    return cudaGetLastError();
}

cudaError_t launch_pre_add3_bt(const float* B, long long ldb, long long K, long long N, long long h, long long w,
                               const Stack16& out, int kind, const float* scale, cudaStream_t stream) {
    if (h <= 0 || w <= 0) return cudaSuccess;
    if ((h & 3) != 0) return cudaErrorInvalidValue;   // float4 staging along n
    switch (kind) {
        case kSplitBF16: return launch_pre_add3_bt_impl<kSplitBF16>(B, ldb, K, N, h, w, out, scale, stream);
        case kSplitFP16: return launch_pre_add3_bt_impl<kSplitFP16>(B, ldb, K, N, h, w, out, scale, stream);
        default: return launch_pre_add3_bt_impl<kSplitTF32>(B, ldb, K, N, h, w, out, scale, stream);
    }
}

cudaError_t launch_post_add3(const float* P, long long ld_in, long long child_stride, long long nodes, long long h,
                             long long w, float* out, long long ld_out, long long out_node_stride,
                             long long valid_rows, long long valid_cols, float alpha, float beta,
                             cudaStream_t stream) {
    if (h <= 0 || w <= 0 || nodes <= 0) return cudaSuccess;
    dim3 grid((unsigned)((w + 127) / 128), gy(h), (unsigned)nodes);
    if (valid_rows >= 0)
        launch_dep(post_add3_kernel<true>, grid, 128, 0, stream, P, ld_in, child_stride, h, w, out, ld_out, out_node_stride,
                                                         valid_rows, valid_cols, alpha, beta);
    else
        launch_dep(post_add3_kernel<false>, grid, 128, 0, stream, P, ld_in, child_stride, h, w, out, ld_out, out_node_stride,
                                                          -1, -1, 1.f, 0.f);
    return cudaGetLastError();
}

cudaError_t launch_post_add2(const float* P, long long ld_in, long long child_stride, long long nodes, long long h,
                             long long w, float* out, long long ld_out, long long out_node_stride,
                             long long valid_rows, long long valid_cols, float alpha, float beta,
                             cudaStream_t stream) {
    if (h <= 0 || w <= 0 || nodes <= 0) return cudaSuccess;
    dim3 grid((unsigned)((w + 127) / 128), gy(h), (unsigned)nodes);
    if (valid_rows >= 0)
        launch_dep(post_add2_kernel<true>, grid, 128, 0, stream, P, ld_in, child_stride, h, w, out, ld_out, out_node_stride,
                                                         valid_rows, valid_cols, alpha, beta);
    else
        launch_dep(post_add2_kernel<false>, grid, 128, 0, stream, P, ld_in, child_stride, h, w, out, ld_out, out_node_stride,
                                                          -1, -1, 1.f, 0.f);
    return cudaGetLastError();
}

cudaError_t launch_batched_split(const SplitJob* jobs, int njobs, long long total_tiles, int kind,
                                 cudaStream_t stream) {
    if (njobs <= 0 || total_tiles <= 0) return cudaSuccess;
    switch (kind) {
        case kSplitBF16: batched_split_kernel<kSplitBF16><<<(unsigned)total_tiles, dim3(32, 8), 0, stream>>>(jobs, njobs); break;
        case kSplitFP16: batched_split_kernel<kSplitFP16><<<(unsigned)total_tiles, dim3(32, 8), 0, stream>>>(jobs, njobs); break;
        case kSplitTF32X: batched_split_kernel<kSplitTF32X><<<(unsigned)total_tiles, dim3(32, 8), 0, stream>>>(jobs, njobs); break;
        default: batched_split_kernel<kSplitTF32><<<(unsigned)total_tiles, dim3(32, 8), 0, stream>>>(jobs, njobs);
    }
    return cudaGetLastError();
}

cudaError_t launch_batched_absmax(const AbsJob* jobs, int njobs, long long total_tiles, cudaStream_t stream) {
    if (njobs <= 0 || total_tiles <= 0) return cudaSuccess;
    const long long blocks = (total_tiles + 1) / 2 < 152 * 8 ? (total_tiles + 1) / 2 : 152 * 8;
    // in plain order: the memset of the slots before it lets nothing overlap
    batched_absmax_kernel<<<(unsigned)blocks, 256, 0, stream>>>(jobs, njobs, total_tiles);
    return cudaGetLastError();
}

cudaError_t launch_batched_fp16_scales(const unsigned* maxima, const float* bound, float* scales, int count,
                                       cudaStream_t stream) {
    if (count <= 0) return cudaSuccess;
    launch_dep(batched_fp16_scale_kernel, (unsigned)((2 * count + 255) / 256), 256, 0, stream, maxima, bound, scales, count);
    return cudaGetLastError();
}

cudaError_t launch_fill(float* p, size_t n, unsigned seed, cudaStream_t stream) {
    if (n == 0) return cudaSuccess;
    fill_kernel<<<1024, 256, 0, stream>>>(p, n, seed);
    return cudaGetLastError();
}

// 2-D copy of a rows x cols block between pinned host memory (through its
// device mapping) and device memory, by SM loads and stores: the host-resident
// plan's alternative to the copy engines.  float4 when both blocks allow it,
// four of them in flight per thread; otherwise a warp takes 512 floats of a row
// at a time, sixteen loads per lane in flight (one load in flight and a division
// per float: 2216 x 2112 x 6607, odd rows, 1547 us a call; 915 now, panels
// included).  Few and large blocks: what a copy beside the compute costs is the
// SMs it touches.  Calls of 8192^3, 3861 x 8164 x 6564, 4000^3 (us) with
//    8 blocks of 1024 threads: 5250, 2365, 936     64 blocks of 256: 5360, 3055, 1160
//   12 blocks of 1024:         5177, 2472, 948    152 blocks of 128: 5950, 3157, 1230
//   16 blocks of 1024:         5190, 2680, 960     32 blocks of 512: 5335, 3113, 1156
// C of odd length and row stride, in one or two panels of a depth-0 product of less than
// a tenth of the copies' time, leaves by 32 blocks of 512, a float per thread, the whole
// grid at one stretch of a row (BY_GRID): 3372 x 1683 x 136 169 us, 209 by warps of 512
// floats; 4425 x 1185 x 87 158 and 208; 3001 x 1501 x 501 185 and 229 (but 2995 x 4863 x 85 in
// four panels 512 and 440).
// Where the products, not the copies, set the pace (the second order of a root's
// products), 32 blocks of 512 are ahead, which with 48 registers a thread share an SM
// with a fused leaf CTA (256 x 160 of 65536): 16384^3 29.5 ms, 32.4 with 50 registers
// and 32.9 with 12 blocks of 1024.
constexpr int kHostCopyBlocks = 12, kHostCopyThreads = 1024, kHostCopyBlocksWide = 32, kHostCopyThreadsWide = 512;
constexpr int kHostCopyUnroll = 4;
template <bool VEC, bool BY_GRID>
__global__ void __maxnreg__(48) host_copy2d_kernel(const float* __restrict__ src, long long lds,
                                                          float* __restrict__ dst, long long ldd, long long rows,
                                                          long long cols) {
    const long long step = (long long)gridDim.x * blockDim.x;
    if constexpr (VEC) {
        const long long c4 = cols >> 2, total = rows * c4;
        long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        for (; i + (kHostCopyUnroll - 1) * step < total; i += kHostCopyUnroll * step) {
            float4 v[kHostCopyUnroll];
#pragma unroll
            for (int j = 0; j < kHostCopyUnroll; ++j) {
                const long long e = i + j * step, r = e / c4, c = e - r * c4;
                v[j] = reinterpret_cast<const float4*>(src + r * lds)[c];
            }
#pragma unroll
            for (int j = 0; j < kHostCopyUnroll; ++j) {
                const long long e = i + j * step, r = e / c4, c = e - r * c4;
                reinterpret_cast<float4*>(dst + r * ldd)[c] = v[j];
            }
        }
        for (; i < total; i += step) {
            const long long r = i / c4, c = i - r * c4;
            reinterpret_cast<float4*>(dst + r * ldd)[c] = reinterpret_cast<const float4*>(src + r * lds)[c];
        }
    } else if constexpr (BY_GRID) {
        const long long total = rows * cols;
        for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
            const long long r = i / cols, c = i - r * cols;
            dst[r * ldd + c] = src[r * lds + c];
        }
    } else {
        // a warp takes 512 consecutive floats of a row, sixteen loads per lane in flight
        const int lane = threadIdx.x & 31;
        const long long segs = (cols + 511) / 512, total = rows * segs, warps = step >> 5;
        for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < total; i += warps) {
            const long long r = i / segs, c0 = (i - r * segs) * 512 + lane;
            const float* s = src + r * lds;
            float* d = dst + r * ldd;
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (c0 + 32 * j < cols) v[j] = s[c0 + 32 * j];
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (c0 + 32 * j < cols) d[c0 + 32 * j] = v[j];
        }
    }
}

cudaError_t launch_host_copy2d(const float* src, long long lds, float* dst, long long ldd, long long rows,
                               long long cols, bool wide, bool by_grid, cudaStream_t stream) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    const int vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) == 0 &&
                    lds % 4 == 0 && ldd % 4 == 0 && cols % 4 == 0;
    const unsigned blocks = wide ? kHostCopyBlocksWide : kHostCopyBlocks;
    const unsigned threads = wide ? kHostCopyThreadsWide : kHostCopyThreads;
    if (vec) host_copy2d_kernel<true, false><<<blocks, threads, 0, stream>>>(src, lds, dst, ldd, rows, cols);
    else if (by_grid) host_copy2d_kernel<false, true><<<blocks, threads, 0, stream>>>(src, lds, dst, ldd, rows, cols);
    else host_copy2d_kernel<false, false><<<blocks, threads, 0, stream>>>(src, lds, dst, ldd, rows, cols);
    return cudaGetLastError();
}

cudaError_t launch_scale(float* C, long long ldc, long long M, long long N, float beta, cudaStream_t stream) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    dim3 grid((unsigned)((N + 255) / 256), gy(M));
    scale_kernel<<<grid, 256, 0, stream>>>(C, ldc, M, N, beta);
    return cudaGetLastError();
}

}  // namespace fmm
