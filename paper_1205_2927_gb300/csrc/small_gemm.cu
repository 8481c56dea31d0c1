// small_gemm.cu -- one-launch tensor-core GEMM for products too small to fill
// the GPU with the leaf kernels' tiles:  C = alpha A B + beta C, row-major, any
// alignment and leading dimension, no workspace.
//
// The leaf path of a small product costs three launches (A's and B's operand
// planes, then 128 x 256 tiles on a fraction of the SMs).  Here each CTA reads
// its fp32 operands itself, splits them and writes the tensor core's swizzled
// tiles in one step (B turned to K-major on the way), so that tiles can be as
// narrow as 32 columns, and a cluster of CTAs can share one tile's K range, each
// taking a chunk; their accumulators meet in shared memory and are added in a
// fixed order, every CTA storing its share of the rows.
//
// Bound: the launch, then the serial chain of K steps, each of which the L1 and
// shared-memory pipe sets (operand loads, split stores and MMA reads; 512 loader
// threads keep loads two steps ahead, 256 took 1.0 us a step): 0.60 / 0.65 / 0.80
// us per 32 columns of K at tiles of 32 / 64 / 128 columns in FP32.  Calls:
// 700 x 515 x 901 38 us by the leaf path, 13.7 this way; 768^3 30 and 11; 573 x
// 452 x 2103 55 and 22; 512^3 21 and 15.5 (16 clusters of 8, of which 15 fit at once).
//
//   warps 0..15 loaders: coalesced global reads (rows of A 128 bytes at a time,
//               B by columns), split, 16-byte swizzled shared-memory stores; after
//               the last step warps 0..3 read the accumulator and all store C
//   warp 16     TMEM allocation, MMA issue
// Every wait is bounded (ptx.cuh).
#include "fmm_internal.h"
#include "ptx.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

namespace fmm {
namespace {

// How the operands are split: SmallMode of a launch.
//   kSmall3xTF32   fp32 hi (read truncated) and lo planes, three TF32 products
//   kSmallTF32     one plane, one product
//   kSmallBF16x3 / kSmallFP16x3  16-bit hi and lo, three products
template <int MODE, int BN>
struct SmallCfg {
    static constexpr bool k16 = MODE == kSmallBF16x3 || MODE == kSmallFP16x3;
    static constexpr int kPlanes = MODE == kSmallTF32 ? 1 : 2;
    static constexpr int kKB = k16 ? 64 : 32;               // K per stage: one 128-byte row
    static constexpr int kABytes = 128 * 128, kBBytes = BN * 128;
    static constexpr int kStageBytes = kPlanes * (kABytes + kBBytes);
    static constexpr int kFit = (200 * 1024) / kStageBytes;
    static constexpr int kStages = kFit < 6 ? kFit : 6;
    static constexpr int kOutPitch = BN + 4;                // floats
    static constexpr int kLoaders = 512;                    // threads of the 16 loader warps
    static constexpr size_t kSmem = 1024 + (size_t)kStages * kStageBytes + 256;
    static_assert(kStages >= 3 && 128 * kOutPitch * 4 <= kStages * kStageBytes, "stages");
};

__device__ __forceinline__ void sts16(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
// Four consecutive values of K at 16-byte group c (0..7) of row r into the hi and
// lo planes of a 128-byte-swizzled tile (fp32 modes).
template <int MODE>
__device__ __forceinline__ void put4(uint32_t hi, uint32_t lo, int r, int c, const float (&x)[4]) {
    const uint32_t at = (uint32_t)r * 128u + (uint32_t)((c ^ (r & 7)) << 4);
    sts16(hi + at, __float_as_uint(x[0]), __float_as_uint(x[1]), __float_as_uint(x[2]), __float_as_uint(x[3]));
    if constexpr (MODE == kSmall3xTF32) {
        float l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) l[i] = tf32_round_rne(x[i] - tf32_trunc(x[i]));
        sts16(lo + at, __float_as_uint(l[0]), __float_as_uint(l[1]), __float_as_uint(l[2]), __float_as_uint(l[3]));
    }
}
// Eight consecutive values of K at group c of row r (16-bit modes).
template <int MODE>
__device__ __forceinline__ void put8(uint32_t hi, uint32_t lo, int r, int c, const float (&x)[8], float sc) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float a = x[2 * i] * sc, b = x[2 * i + 1] * sc;
        if constexpr (MODE == kSmallBF16x3) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
            const float2 f = __bfloat1622float2(p);
            const __nv_bfloat162 q = __floats2bfloat162_rn(a - f.x, b - f.y);
            h[i] = *reinterpret_cast<const uint32_t*>(&p);
            l[i] = *reinterpret_cast<const uint32_t*>(&q);
        } else {
            const __half2 p = __floats2half2_rn(a, b);
            const float2 f = __half22float2(p);
            const __half2 q = __floats2half2_rn(a - f.x, b - f.y);
            h[i] = *reinterpret_cast<const uint32_t*>(&p);
            l[i] = *reinterpret_cast<const uint32_t*>(&q);
        }
    }
    const uint32_t at = (uint32_t)r * 128u + (uint32_t)((c ^ (r & 7)) << 4);
    sts16(hi + at, h[0], h[1], h[2], h[3]);
    sts16(lo + at, l[0], l[1], l[2], l[3]);
}

__device__ __forceinline__ float4 ld_cluster4(uint32_t addr, uint32_t rank) {
    uint32_t ra;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(ra)
                 : "memory");
    return v;
}

template <int MODE, int BN>
__global__ void __launch_bounds__(544, 1) small_gemm_kernel(const SmallArgs args) {
    using Cfg = SmallCfg<MODE, BN>;
    constexpr int G = Cfg::k16 ? 8 : 4;            // K elements per 16-byte group
    constexpr int NL = Cfg::kLoaders;
    constexpr int NA = 128 * 8 / NL;               // A groups per loader
    constexpr int NB = (BN * 8 + NL - 1) / NL;     // B groups per loader (BN = 32: of half of them)
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw_addr = smem_u32(smem_raw);
    const uint32_t base = (raw_addr + 1023u) & ~1023u;
    uint8_t* base_ptr = smem_raw + (base - raw_addr);
    const uint32_t bar0 = base + Cfg::kStages * Cfg::kStageBytes;
    uint8_t* bar_ptr = base_ptr + Cfg::kStages * Cfg::kStageBytes;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (Cfg::kStages + s); };
    const uint32_t done_bar = bar0 + 8u * (2 * Cfg::kStages);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + 8 * (2 * Cfg::kStages + 1));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 8 * (2 * Cfg::kStages + 1) + 8);

    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int splits = args.splits, rank = (int)blockIdx.x % splits, tile = (int)blockIdx.x / splits;
    const int tm = tile % args.tiles_m, tn = tile / args.tiles_m;
    const int k_begin = rank * args.k_chunk, k_end = min(args.K, k_begin + args.k_chunk);
    const int nk = (k_end - k_begin + Cfg::kKB - 1) / Cfg::kKB;   // >= 1 (the launch sees to it)
    unsigned* status = args.status;

    if (t == 0) {
        for (int s = 0; s < Cfg::kStages; ++s) {
            mbar_init(full_bar(s), NL / 32);   // one arrival per loader warp
            mbar_init(empty_bar(s), 1);
        }
        mbar_init(done_bar, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == NL / 32) {
        tmem_alloc(smem_u32(tmem_slot), BN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    dep_start();
    // a call that owns its status word starts it from zero: waits run out, and
    // report, seconds after the launch's first block has passed here
    if (args.clear_status && blockIdx.x == 0 && t == 0) *status = 0u;
    bool ok = true;

    if (warp < NL / 32) {
        const int m0 = tm * 128, n0 = tn * BN;
        const float sa = args.scale ? args.scale[0] : 1.0f, sb = args.scale ? args.scale[1] : 1.0f;
        // A: group i of this thread is row t / 8 + 64 i, group t % 8; B: column
        // (t + 512 i) % BN, consecutive lanes on consecutive columns.  Rows past M and
        // columns past N read the last valid one: what they add up to is not stored.
        const int ar = t >> 3, ac = t & 7;
        const bool has_b = BN * 8 >= NL || t < BN * 8;
        const float *pa[NA], *pb[NB];
#pragma unroll
        for (int i = 0; i < NA; ++i)
            pa[i] = args.A + (long long)min(m0 + ar + NL / 8 * i, args.M - 1) * args.lda + k_begin + ac * G;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int e = t + NL * i;
            pb[i] = args.B + (long long)(k_begin + e / BN * G) * args.ldb + min(n0 + e % BN, args.N - 1);
        }
        float a[2][NA][G], b[2][NB][G];
        auto load = [&](int buf, int step) {
            const int left = k_end - k_begin - step * Cfg::kKB;   // columns of K from this step on
            const long long ao = (long long)step * Cfg::kKB, bo = ao * args.ldb;
            const bool whole = left >= Cfg::kKB;   // else the end of K: zeros beyond it in both operands
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                const float* p = pa[i] + ao;
                if (whole && args.a_vec) {
#pragma unroll
                    for (int j = 0; j < G; j += 4) {
                        const float4 v = *reinterpret_cast<const float4*>(p + j);
                        a[buf][i][j] = v.x; a[buf][i][j + 1] = v.y; a[buf][i][j + 2] = v.z; a[buf][i][j + 3] = v.w;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < G; ++j) a[buf][i][j] = whole || ac * G + j < left ? p[j] : 0.0f;
                }
            }
            if (has_b) {
#pragma unroll
                for (int i = 0; i < NB; ++i) {
                    const float* p = pb[i] + bo;
                    const int k = (t + NL * i) / BN * G;
#pragma unroll
                    for (int j = 0; j < G; ++j, p += args.ldb) b[buf][i][j] = whole || k + j < left ? *p : 0.0f;
                }
            }
        };
        int stage = 0;
        uint32_t phase = 0;
        auto step = [&](int buf, int it) {
            if (ok) ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) return;
            const uint32_t ah = base + stage * Cfg::kStageBytes;
            const uint32_t bh = ah + Cfg::kABytes;
            const uint32_t al = bh + Cfg::kBBytes, bl = al + Cfg::kABytes;   // second planes
#pragma unroll
            for (int i = 0; i < NA; ++i) {
                if constexpr (Cfg::k16) put8<MODE>(ah, al, ar + NL / 8 * i, ac, a[buf][i], sa);
                else put4<MODE>(ah, al, ar + NL / 8 * i, ac, a[buf][i]);
            }
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                const int e = t + NL * i;
                if (!has_b) break;
                if constexpr (Cfg::k16) put8<MODE>(bh, bl, e % BN, e / BN, b[buf][i], sb);
                else put4<MODE>(bh, bl, e % BN, e / BN, b[buf][i]);
            }
            if (it + 2 < nk) load(buf, it + 2);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(full_bar(stage));
            if (++stage == Cfg::kStages) { stage = 0; phase ^= 1u; }
        };
        load(0, 0);
        if (nk > 1) load(1, 1);
        for (int it = 0; it < nk && ok; it += 2) {
            step(0, it);
            if (it + 1 < nk) step(1, it + 1);
        }
    } else if (lane == 0) {
        constexpr uint32_t idesc = make_idesc(2u, 128, BN);
        constexpr uint32_t idesc16 = make_idesc(MODE == kSmallFP16x3 ? 0u : 1u, 128, BN);
        int stage = 0;
        uint32_t phase = 0;
        for (int it = 0; it < nk; ++it) {
            if (!mbar_wait(full_bar(stage), phase, abort_flag, status)) break;
            tc_fence_after();
            const uint32_t ah = base + stage * Cfg::kStageBytes;
            const uint32_t bh = ah + Cfg::kABytes;
            const uint32_t al = bh + Cfg::kBBytes, bl = al + Cfg::kABytes;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                const uint32_t first = (it == 0 && kk == 0) ? 0u : 1u;
                const uint64_t ahd = sdesc_kmajor_sw128(ah + kk * 32), bhd = sdesc_kmajor_sw128(bh + kk * 32);
                if constexpr (MODE == kSmallTF32) {
                    mma_tf32(tmem, ahd, bhd, idesc, first);
                } else {
                    const uint64_t ald = sdesc_kmajor_sw128(al + kk * 32), bld = sdesc_kmajor_sw128(bl + kk * 32);
                    if constexpr (Cfg::k16) {
                        mma_f16(tmem, ald, bhd, idesc16, first);
                        mma_f16(tmem, ahd, bld, idesc16, 1u);
                        mma_f16(tmem, ahd, bhd, idesc16, 1u);
                    } else {
                        mma_tf32(tmem, ald, bhd, idesc, first);
                        mma_tf32(tmem, ahd, bld, idesc, 1u);
                        mma_tf32(tmem, ahd, bhd, idesc, 1u);
                    }
                }
            }
            mma_commit(empty_bar(stage));
            if (++stage == Cfg::kStages) { stage = 0; phase ^= 1u; }
        }
        mma_commit(done_bar);
    }

    // accumulator -> this CTA's shared memory (the stages are free once done_bar
    // completes), rows kOutPitch floats apart
    float* out = reinterpret_cast<float*>(base_ptr);
    if (warp < 4) {
        if (ok) ok = mbar_wait(done_bar, 0u, abort_flag, status);
        if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            float* row = out + (warp * 32 + lane) * Cfg::kOutPitch;
#pragma unroll 1
            for (int c = 0; c < BN; c += 32) {
                uint32_t r[32];
                tmem_ld_32x32b_x32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c, r);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    *reinterpret_cast<float4*>(row + c + j) =
                        make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]), __uint_as_float(r[j + 2]),
                                    __uint_as_float(r[j + 3]));
            }
        }
        tc_fence_before();
    }
    __syncwarp();
    if (splits > 1) cluster_sync();
    else __syncthreads();
    // rows of the tile shared out over the cluster's CTAs; a thread takes 4 columns
    {
        const int per = 128 / splits, lo = rank * per;
        const int rows = min(per, args.M - tm * 128 - lo);
        float alpha = args.alpha;
        if (Cfg::k16 && args.scale) alpha = alpha / (args.scale[0] * args.scale[1]);   // undo the operand scaling
        const uint32_t out0 = base;
        for (int e = t; e < rows * (BN / 4); e += NL + 32) {
            const int r = lo + e / (BN / 4), c = e % (BN / 4) * 4, col = tn * BN + c;
            if (col >= args.N) continue;
            float4 v = *reinterpret_cast<const float4*>(out + r * Cfg::kOutPitch + c);
            if (splits > 1) {
                v = ld_cluster4(out0 + (uint32_t)(r * Cfg::kOutPitch + c) * 4u, 0u);
                for (int s = 1; s < splits; ++s) {
                    const float4 w = ld_cluster4(out0 + (uint32_t)(r * Cfg::kOutPitch + c) * 4u, (uint32_t)s);
                    v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
                }
            }
            v.x *= alpha; v.y *= alpha; v.z *= alpha; v.w *= alpha;
            float* p = args.C + (long long)(tm * 128 + r) * args.ldc + col;
            if (args.c_vec && col + 4 <= args.N) {
                if (args.beta != 0.0f) {
                    const float4 o = *reinterpret_cast<const float4*>(p);
                    v.x += args.beta * o.x; v.y += args.beta * o.y; v.z += args.beta * o.z; v.w += args.beta * o.w;
                }
                *reinterpret_cast<float4*>(p) = v;
            } else {
                const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (col + j < args.N) p[j] = args.beta != 0.0f ? x[j] + args.beta * p[j] : x[j];
            }
        }
    }
    __syncwarp();
    if (splits > 1) cluster_sync();   // no CTA leaves while another reads its sums
    else __syncthreads();
    if (warp == NL / 32) {
        tc_fence_after();
        tmem_dealloc(tmem, BN);
    }
}

template <int MODE, int BN>
cudaError_t launch(const SmallArgs& a, cudaStream_t stream) {
    using Cfg = SmallCfg<MODE, BN>;
    auto kern = small_gemm_kernel<MODE, BN>;
    static bool attr_done[64] = {};   // once per device: later launches make no other API call
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_done[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_done[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.splits;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_dep
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)((long long)a.tiles_m * a.tiles_n * a.splits));
    cfg.blockDim = dim3(Cfg::kLoaders + 32);
    cfg.dynamicSmemBytes = Cfg::kSmem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int MODE>
cudaError_t launch_mode(const SmallArgs& a, int bn, cudaStream_t stream) {
    switch (bn) {
        case 32: return launch<MODE, 32>(a, stream);
        case 64: return launch<MODE, 64>(a, stream);
        default: return launch<MODE, 128>(a, stream);
    }
}

}  // namespace

cudaError_t launch_small_gemm(SmallArgs a, int mode, int bn, int splits, cudaStream_t stream) {
    if (a.M <= 0 || a.N <= 0 || a.K <= 0) return cudaErrorInvalidValue;
    const int kb = mode == kSmallBF16x3 || mode == kSmallFP16x3 ? 64 : 32;
    const int steps = (a.K + kb - 1) / kb;
    while (splits > 1 && (splits - 1) * ((steps + splits - 1) / splits) >= steps) splits >>= 1;   // no empty chunk
    a.splits = splits;
    a.k_chunk = (steps + splits - 1) / splits * kb;
    a.tiles_m = (a.M + 127) / 128;
    a.tiles_n = (a.N + bn - 1) / bn;
    a.a_vec = (reinterpret_cast<uintptr_t>(a.A) & 15) == 0 && a.lda % 4 == 0;
    a.c_vec = (reinterpret_cast<uintptr_t>(a.C) & 15) == 0 && a.ldc % 4 == 0;
    switch (mode) {
        case kSmall3xTF32: return launch_mode<kSmall3xTF32>(a, bn, stream);
        case kSmallTF32: return launch_mode<kSmallTF32>(a, bn, stream);
        case kSmallBF16x3: return launch_mode<kSmallBF16x3>(a, bn, stream);
        case kSmallFP16x3: return launch_mode<kSmallFP16x3>(a, bn, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace fmm
