// mlp.cu -- the planner's cost model: a 6 -> 64 -> 64 -> 1 ReLU network in fp32
// that predicts log(run time) of a candidate plan from
// (log2 M, log2 K, log2 N, depth, leaf tile / 128, precision), standardised.
//
// Parameter vector (flat, NPARAM floats): W1[64][6], b1[64], W2[64][64], b2[64],
// W3[1][64], b3[1]; weights row-major [out][in].
//
// Kernels: forward (one thread per sample, weights in shared memory); training
// step = forward, backward and gradient sums of each block's samples, then the
// blocks' sums added in a fixed order and Adam in place.
#include "../../include/fmm.h"
#include "fmm_internal.h"
#include "ptx.cuh"

namespace fmm {
namespace {

constexpr int IN = 6, HID = 64;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + HID * IN, OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID * HID,
              OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + HID, NPARAM = OFF_B3 + 1;
static_assert(NPARAM == FMM_MLP_NPARAM, "parameter count");

__device__ __forceinline__ void load_params(float* sp, const float* __restrict__ params) {
    for (int i = threadIdx.x; i < NPARAM; i += blockDim.x) sp[i] = params[i];
    __syncthreads();
}

__global__ void __launch_bounds__(128) mlp_forward_kernel(const float* __restrict__ params,
                                                          const float* __restrict__ X, float* __restrict__ Y,
                                                          int batch) {
    __shared__ float sp[NPARAM];
    load_params(sp, params);
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= batch) return;
    float x[IN], h1[HID];
#pragma unroll
    for (int j = 0; j < IN; ++j) x[j] = X[s * IN + j];
#pragma unroll 4
    for (int i = 0; i < HID; ++i) {
        float z = sp[OFF_B1 + i];
#pragma unroll
        for (int j = 0; j < IN; ++j) z += sp[OFF_W1 + i * IN + j] * x[j];
        h1[i] = z > 0.f ? z : 0.f;
    }
    float y = sp[OFF_B3];
    for (int i = 0; i < HID; ++i) {
        float z = sp[OFF_B2 + i];
#pragma unroll 8
        for (int j = 0; j < HID; ++j) z += sp[OFF_W2 + i * HID + j] * h1[j];
        y += sp[OFF_W3 + i] * (z > 0.f ? z : 0.f);
    }
    Y[s] = y;
}

// Training step, first kernel: forward, backward and the gradient of a block's
// share of the batch, 32 samples at a time; nothing per sample leaves the SM.
// Per tile, three 64-deep products (z2 = h1 W2^T, dh1 = dz2 W2, dW2 += dz2^T h1)
// run from shared memory with 16 or 32 outputs per thread, every read 16 bytes
// of a row.  Lanes take neighbouring rows 68 floats apart, so the eight rows of
// a quarter warp fall on different banks.  Each block adds its samples in order
// and leaves one row of NPARAM + 1 sums; the second kernel adds the rows in a
// fixed order, so a step is deterministic.
//
// Bound: latency of a few warps of fp32 arithmetic per SM (batch 20000: 0.25
// GFMA), shared-memory reads next (L1 71 %).  One thread per parameter summing the
// whole batch in series, on 37 blocks, took 1066 us a step at batch 20000; this takes
// 32.0 us (33.4 with one multiply-add per instruction; four blocks per SM, whose
// registers no longer hold a tile's outputs and gradients: 32.6).
constexpr int TS = 32, NT = 128;   // samples per tile, threads per block
constexpr int PU = HID + 4;        // row pitch (floats)
struct TrainSmem {
    float w2[HID][PU];
    float h1[TS][PU], dz2[TS][PU], dz1[TS][PU];
    float w1[HID * IN], b1[HID], b2[HID], w3[HID];
    float x[TS][8];
    float ypart[16][TS];
    float dy[TS];
    float b3;
};
constexpr int kTrainGrid = 456;    // three blocks per SM on 152 SMs
constexpr int ROW = NPARAM + 1;         // a block's sums: the gradient, then the sum of (y - t)^2

struct AdamArgs {
    float *params, *m, *v, *grad_out, *loss_out;
    int batch, step;
    float lr, beta1, beta2, eps;
};

// Entry p of the summed gradient (p == NPARAM: of the squared errors).
__device__ __forceinline__ void adam_apply(const AdamArgs& a, int p, float g) {
    if (p == NPARAM) {
        if (a.loss_out) *a.loss_out = 0.5f * g / (float)a.batch;
        return;
    }
    if (a.grad_out) a.grad_out[p] = g;
    if (a.lr != 0.f) {
        const float mi = a.beta1 * a.m[p] + (1.f - a.beta1) * g;
        const float vi = a.beta2 * a.v[p] + (1.f - a.beta2) * g * g;
        a.m[p] = mi;
        a.v[p] = vi;
        const float mhat = mi / (1.f - powf(a.beta1, (float)a.step));
        const float vhat = vi / (1.f - powf(a.beta2, (float)a.step));
        a.params[p] -= a.lr * mhat / (sqrtf(vhat) + a.eps);
    }
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float a, float b, float c, float d) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}
// Two fp32 multiply-adds in one instruction, each rounded as fmaf rounds: half the
// issue slots of the products.
struct f2 { unsigned long long v; };
__device__ __forceinline__ f2 pack2(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(f2 x, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v)); }
__device__ __forceinline__ void fma2(f2& acc, f2 a, f2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc.v) : "l"(a.v), "l"(b.v));
}
__device__ __forceinline__ float sum8(float x) {   // over the eight sample groups of a unit group
    x += __shfl_xor_sync(0xffffffffu, x, 1);
    x += __shfl_xor_sync(0xffffffffu, x, 2);
    return x + __shfl_xor_sync(0xffffffffu, x, 4);
}

// rows: one ROW per block, left to the second kernel.  ALONE: a single block,
// which updates the parameters itself (batches whose workspace holds no two rows).
// Blocks take tiles blockIdx.x * per, ... (per tiles each).
template <bool ALONE>
__global__ void __launch_bounds__(NT, 3) mlp_train_kernel(const float* X, const float* T,
                                                          int per, float* __restrict__ rows, AdamArgs a) {
    extern __shared__ float4 train_smem[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(train_smem);
    dep_start();
    const int t = threadIdx.x, sg = t & 7, ug = t >> 3;      // samples sg + 8 q; units ug + 16 u, or 4 ug + u
    const int u0 = 4 * ug;
    const int i8 = 8 * (t & 7), j4 = 4 * (t >> 3);           // dW2 rows i8 .. + 7, columns j4 .. + 3
    {
        float w[HID * HID / NT];   // every load before the first store
#pragma unroll
        for (int e = 0; e < HID * HID / NT; ++e) w[e] = a.params[OFF_W2 + t + e * NT];
#pragma unroll
        for (int e = 0; e < HID * HID / NT; ++e) S.w2[(t + e * NT) / HID][(t + e * NT) % HID] = w[e];
    }
    for (int e = t; e < HID * IN; e += NT) S.w1[e] = a.params[OFF_W1 + e];
    if (t < HID) {
        S.b1[t] = a.params[OFF_B1 + t];
        S.b2[t] = a.params[OFF_B2 + t];
        S.w3[t] = a.params[OFF_W3 + t];
    }
    if (t == 0) S.b3 = a.params[OFF_B3];
    f2 gw2[8][2] = {};
    float gb1[4] = {}, gb2[4] = {}, gw3[4] = {}, gw1[3] = {}, gb3 = 0.f, sq = 0.f;
    const int tiles = (a.batch + TS - 1) / TS;
    for (int tile = blockIdx.x * per; tile < min(tiles, (int)(blockIdx.x + 1) * per); ++tile) {
        const int base = tile * TS, valid = min(TS, a.batch - base);
        __syncthreads();   // the previous tile's arrays are read
        for (int e = t; e < TS * IN; e += NT) S.x[e / IN][e % IN] = e / IN < valid ? X[(size_t)base * IN + e] : 0.f;
        __syncthreads();
        // h1 = relu(W1 x + b1); zero beyond the batch
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int row = sg + 8 * q;
            float h[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float z = S.b1[u0 + u];
#pragma unroll
                for (int j = 0; j < IN; ++j) z += S.w1[(u0 + u) * IN + j] * S.x[row][j];
                h[u] = z > 0.f && row < valid ? z : 0.f;
            }
            st4(&S.h1[row][u0], h[0], h[1], h[2], h[3]);
        }
        __syncthreads();
        f2 z2[4][4];     // sums over even and odd j
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) z2[q][u] = pack2(S.b2[ug + 16 * u], 0.f);
#pragma unroll 2
        for (int j = 0; j < HID; j += 4) {
            float4 h[4], w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) h[q] = ld4(&S.h1[sg + 8 * q][j]);
#pragma unroll
            for (int u = 0; u < 4; ++u) w[u] = ld4(&S.w2[ug + 16 * u][j]);
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    fma2(z2[q][u], pack2(h[q].x, h[q].y), pack2(w[u].x, w[u].y));
                    fma2(z2[q][u], pack2(h[q].z, h[q].w), pack2(w[u].z, w[u].w));
                }
        }
        float z[4][4];   // [sample sg + 8 q][unit ug + 16 u]
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float a0, a1;
                unpack2(z2[q][u], a0, a1);
                z[q][u] = a0 + a1;
            }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float y = 0.f;
#pragma unroll
            for (int u = 0; u < 4; ++u) y += S.w3[ug + 16 * u] * (z[q][u] > 0.f ? z[q][u] : 0.f);
            S.ypart[ug][sg + 8 * q] = y;
        }
        __syncthreads();
        if (t < TS) {
            float y = S.b3;
#pragma unroll
            for (int g = 0; g < 16; ++g) y += S.ypart[g][t];
            const float r = t < valid ? y - T[base + t] : 0.f;
            const float d = r / (float)a.batch;   // d(0.5 mean r^2)/dy
            S.dy[t] = d;
            gb3 += d;
            sq += r * r;
        }
        __syncthreads();
        // dz2, with its share of the gradients of b2 and W3
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int row = sg + 8 * q;
            const float dy = S.dy[row];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool on = z[q][u] > 0.f && row < valid;
                const float d = on ? dy * S.w3[ug + 16 * u] : 0.f;
                S.dz2[row][ug + 16 * u] = d;
                gb2[u] += d;
                gw3[u] += dy * (z[q][u] > 0.f ? z[q][u] : 0.f);   // dy = 0 beyond the batch; a dy of NaN shows
            }
        }
        __syncthreads();
        f2 dh2[4][2] = {};     // [sample sg + 8 q][units 4 ug + 2 p, + 1]
#pragma unroll 2
        for (int i = 0; i < HID; i += 4) {
            float4 d[4], w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) d[q] = ld4(&S.dz2[sg + 8 * q][i]);
#pragma unroll
            for (int k = 0; k < 4; ++k) w[k] = ld4(&S.w2[i + k][u0]);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float dd[4] = {d[q].x, d[q].y, d[q].z, d[q].w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const f2 x = pack2(dd[k], dd[k]);
                    fma2(dh2[q][0], x, pack2(w[k].x, w[k].y));
                    fma2(dh2[q][1], x, pack2(w[k].z, w[k].w));
                }
            }
        }
        float dh[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            unpack2(dh2[q][0], dh[q][0], dh[q][1]);
            unpack2(dh2[q][1], dh[q][2], dh[q][3]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 h = ld4(&S.h1[sg + 8 * q][u0]);
            const float hh[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                dh[q][u] = hh[u] > 0.f ? dh[q][u] : 0.f;   // h1 > 0 <=> z1 > 0
                gb1[u] += dh[q][u];
            }
            st4(&S.dz1[sg + 8 * q][u0], dh[q][0], dh[q][1], dh[q][2], dh[q][3]);
        }
#pragma unroll 2
        for (int q = 0; q < TS; ++q) {   // dW2 += dz2^T h1
            const float4 d0 = ld4(&S.dz2[q][i8]), d1 = ld4(&S.dz2[q][i8 + 4]), h = ld4(&S.h1[q][j4]);
            const float dd[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
            const f2 h01 = pack2(h.x, h.y), h23 = pack2(h.z, h.w);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const f2 x = pack2(dd[i], dd[i]);
                fma2(gw2[i][0], x, h01);
                fma2(gw2[i][1], x, h23);
            }
        }
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 3; ++e) {    // dW1 += dz1^T x
            const int i = (t + e * NT) / IN, j = (t + e * NT) % IN;
#pragma unroll 8
            for (int q = 0; q < TS; ++q) gw1[e] += S.dz1[q][i] * S.x[q][j];
        }
    }
    auto emit = [&](int p, float g) {
        if constexpr (ALONE) adam_apply(a, p, g);
        else rows[(size_t)blockIdx.x * ROW + p] = g;
    };
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float g0, g1;
            unpack2(gw2[i][j], g0, g1);
            emit(OFF_W2 + (i8 + i) * HID + j4 + 2 * j, g0);
            emit(OFF_W2 + (i8 + i) * HID + j4 + 2 * j + 1, g1);
        }
#pragma unroll
    for (int e = 0; e < 3; ++e) emit(OFF_W1 + t + e * NT, gw1[e]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float g1 = sum8(gb1[u]), g2 = sum8(gb2[u]), g3 = sum8(gw3[u]);
        if (sg == 0) {
            emit(OFF_B1 + u0 + u, g1);
            emit(OFF_B2 + ug + 16 * u, g2);
            emit(OFF_W3 + ug + 16 * u, g3);
        }
    }
    if (t < 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            gb3 += __shfl_xor_sync(0xffffffffu, gb3, o);
            sq += __shfl_xor_sync(0xffffffffu, sq, o);
        }
        if (t == 0) {
            emit(OFF_B3, gb3);
            emit(NPARAM, sq);
        }
    }
}

// Second kernel: 32 parameters per block, 16 warps over the rows (warp w adds
// rows w, w + 16, ...), then the 16 sums in order, then Adam (bias-corrected) in
// place.
__global__ void __launch_bounds__(512) mlp_adam_kernel(const float* rows, int nrows, AdamArgs a) {
    __shared__ float part[16][32];
    dep_start();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
    float g = 0.f;
    if (p <= NPARAM) {
#pragma unroll 8
        for (int r = w; r < nrows; r += 16) g += rows[(size_t)r * ROW + p];
    }
    part[w][lane] = g;
    __syncthreads();
    if (w != 0 || p > NPARAM) return;
#pragma unroll
    for (int q = 1; q < 16; ++q) g += part[q][lane];
    adam_apply(a, p, g);
}

}  // namespace

cudaError_t mlp_forward(const float* params, const float* X, float* Y, int batch, cudaStream_t s) {
    if (batch <= 0) return cudaSuccess;
    mlp_forward_kernel<<<(batch + 127) / 128, 128, 0, s>>>(params, X, Y, batch);
    return cudaGetLastError();
}

}  // namespace fmm

extern "C" fmm_status_t fmm_mlp_forward(const float* params, const float* X, float* Y, int batch, fmm_stream_t s) {
    if (batch < 0 || (batch > 0 && (!params || !X || !Y))) return FMM_ERR_INVALID_ARG;
    return fmm::mlp_forward(params, X, Y, batch, (cudaStream_t)s) == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}

extern "C" fmm_status_t fmm_mlp_train_step(float* params, float* adam_m, float* adam_v, int step, float lr,
                                           const float* X, const float* T, int batch, void* workspace,
                                           size_t workspace_bytes, size_t* workspace_needed, float* grad_out,
                                           float* loss_out, fmm_stream_t stream) {
    using namespace fmm;
    if (batch < 0) return FMM_ERR_INVALID_ARG;
    const size_t per = (size_t)(batch > 0 ? batch : 1);
    const size_t need = (4 * per * HID + 2 * per) * sizeof(float) + 256;
    if (workspace_needed) *workspace_needed = need;
    if (!workspace && !params) return FMM_OK;  // size query
    if (batch == 0) return FMM_OK;
    if (!params || !adam_m || !adam_v || !X || !T || step < 1) return FMM_ERR_INVALID_ARG;
    if (!workspace || workspace_bytes < need) return FMM_ERR_WORKSPACE;
    // one row of sums per block, as many blocks as the workspace and the SMs hold
    const int tiles = (batch + TS - 1) / TS;
    const long long cap = (long long)(need / (ROW * sizeof(float)));
    int blocks = tiles < kTrainGrid ? tiles : kTrainGrid;
    if (blocks > cap) blocks = cap > 1 ? (int)cap : 1;
    const int tiles_per = (tiles + blocks - 1) / blocks;
    blocks = (tiles + tiles_per - 1) / tiles_per;
    const AdamArgs a{params, adam_m, adam_v, grad_out, loss_out, batch, step, lr, 0.9f, 0.999f, 1e-8f};
    cudaStream_t s = (cudaStream_t)stream;
    static bool attr_done[64] = {};   // once per device: later launches make no other API call
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FMM_ERR_CUDA;
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        if (cudaFuncSetAttribute(mlp_train_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(TrainSmem)) != cudaSuccess ||
            cudaFuncSetAttribute(mlp_train_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(TrainSmem)) != cudaSuccess)
            return FMM_ERR_CUDA;
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    float* rows = static_cast<float*>(workspace);
    if (blocks == 1) {
        launch_dep(mlp_train_kernel<true>, 1, NT, sizeof(TrainSmem), s, X, T, tiles_per, nullptr, a);
    } else {
        launch_dep(mlp_train_kernel<false>, blocks, NT, sizeof(TrainSmem), s, X, T, tiles_per, rows, a);
        launch_dep(mlp_adam_kernel, (ROW + 31) / 32, 512, 0, s, rows, blocks, a);
    }
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}
