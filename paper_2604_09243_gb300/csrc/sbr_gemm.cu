// sbr_gemm.cu -- BF16 tensor-core GEMM on the 5th-generation tensor cores
// (tcgen05) for the learned surrogate: C = A B^T with FP32 accumulation in
// tensor memory (TMEM), for one problem or for a group of equal ones (the
// ensemble's members, and for weight gradients every layer of every member).
//
// A is [M x K] and B [N x K], each stored either K-contiguous or (for
// gradients, whose contraction runs over the stored rows) with M or N
// contiguous: the tensor core reads both forms from shared memory, so no
// operand is transposed in memory.
//
// One persistent kernel: a CTA per SM loops over 128 x BN tiles
// t = blockIdx.x, t + gridDim.x, ... (n-tile fastest, then m-tile, then group):
//   - warp 0 (one lane) streams 64-deep slices of A and B of every k-step of
//     every tile into a ring of shared-memory stages with TMA (128-byte
//     swizzle), refilling a stage once the MMAs that read it have completed;
//   - warp 1 (one lane) issues tcgen05.mma (M = 128, N = BN, K = 16 per
//     instruction) for the CTA's tile j into TMEM accumulator j % 2 once the
//     epilogue has drained it, and commits it;
//   - the other 8 or 16 warps read the accumulator (warp w: TMEM lanes 32 (w % 4)
//     .., a share of the columns), hand it back, and apply the fused epilogue 32
//     columns at a time through staging rows of their own, so that a tile's
//     read-out and stores overlap the next tile's MMAs.
// Every wait is bounded and polls the CTA's failure flag: on a timeout the CTA
// records an error flag, skips the remaining work, lets its loads and MMAs
// finish, frees its TMEM and returns.
//
// What bounds it: the GELU epilogues cost ~36 instructions per output, twice
// the MMAs' time at K = 512, and one epilogue warp per scheduler left them
// latency-bound (issue 30 %). Four per scheduler where only BF16 is stored
// (prediction: issue 72 %, 4 x 65536 x 512 x 512 in 188 us = 730 TFLOP/s; a
// member alone with one epilogue warp per scheduler 111 us), two where FP32
// staging rows take the shared memory. Training's forward and backward products
// are bound by their activations: 43 us per layer of 4 members x 8192 rows (134
// MB moved, 3.1 TB/s) forward and 44 backward. All 24 weight gradients take 122
// us (94.5 GFLOP, 775 TFLOP/s, 2.3 tiles per SM). One by one: 23 us per member
// and layer, 46 us per weight gradient.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <math.h>
#include <stdint.h>

#include "sbr_internal.h"

namespace sbr {

namespace {

constexpr int kBM = 128, kBK = 64;
constexpr int kTileA = kBM * kBK * 2;  // bytes
constexpr unsigned kSpin = 1u << 24;   // try_wait rounds before a wait gives up
// staging of one epilogue warp: 32 rows x 32 columns, FP32 (stride 36) and BF16 (stride 40)
constexpr int kLdF = 36, kLdH = 40;
constexpr int kWarpF = 32 * kLdF * 4, kWarpH = 32 * kLdH * 2;

template <int BN, int kMode>
struct Cfg {
    static constexpr bool kF32 = kMode != kEpiGelu, kH16 = kMode != kEpiF32;  // staging an epilogue warp needs
    static constexpr int kEpiWarps = kMode == kEpiGelu ? 16 : 8;
    static constexpr int kThreads = 32 * (2 + kEpiWarps);
    static constexpr int kWarpStage = (kF32 ? kWarpF : 0) + (kH16 ? kWarpH : 0);
    static constexpr int kStages = BN == 256 ? 3 : (BN == 128 ? 5 : 6);
    static constexpr int kStageBytes = kTileA + BN * kBK * 2;
    static constexpr int kPipe = kStages * kStageBytes;
    static constexpr int kSmem = kPipe + kEpiWarps * kWarpStage + 1024;
    static_assert(kSmem <= 227 * 1024, "GEMM shared memory");
    // instruction descriptor: D FP32, A and B BF16, M = 128, N = BN; bits 15 and 16: A, B with M, N contiguous
    __host__ __device__ static constexpr uint32_t idesc(bool mn_a, bool mn_b)
    {
        return (1u << 4) | (1u << 7) | (1u << 10) | (mn_a ? 1u << 15 : 0u) | (mn_b ? 1u << 16 : 0u) |
               ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
    }
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_wait(uint64_t* b, unsigned parity)
{
    const uint32_t a = smem_u32(b);
    for (unsigned i = 0; i < kSpin; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int x, int y, int z, uint64_t* bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)tm), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}
// Shared-memory matrix descriptors of a 64-deep slice, 128-byte swizzle, for
// the 16-deep step kk. K contiguous: rows of 128 bytes (64 k), 8-row groups
// 1024 bytes apart, a step 32 bytes along the row. M or N contiguous: blocks of
// 64 m by 64 k (a row of 128 bytes per k) 8192 bytes apart, 8-k groups 1024
// bytes apart, a step two groups further.
template <bool kMn>
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr, int kk)
{
    const uint32_t a = kMn ? saddr + 2048u * kk : saddr + 32u * kk;
    const uint64_t lead = kMn ? 512ull : 1ull;
    return (uint64_t)((a >> 4) & 0x3FFF) | (lead << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 accumulator columns of the warp's rows; the registers hold them after tmem_wait
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r)
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z)
{
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// a bounded wait that also gives up once another role of the CTA has failed
__device__ __forceinline__ bool pp_wait(uint64_t* b, unsigned parity, volatile int* fail)
{
    const uint32_t a = smem_u32(b);
    for (unsigned i = 0; i < kSpin; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((i & 1023u) == 1023u && *fail) return false;
    }
    return false;
}

// What a launch computes. Tile t < tiles0 belongs to the first segment: group
// t / per[0] (operands at that index of the third map dimension, A from za[0]
// on), tile rows and columns from the remainder; later tiles to the second one
// (B from tmB1). Group g = layer * n_inner + member: its outputs start at
// layer * (layer stride) + member * (member stride).
struct GemmGrid {
    int KT;                // 64-deep k-steps
    int n_tiles, tiles0;
    int tn[2], per[2];     // n-tiles per tile row, tiles per group
    int za[2];
    int n_inner;
    GemmEpi ep[2];
};

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&p);
}

template <int BN, bool kMnA, bool kMnB, int kMode>
__global__ void __launch_bounds__((Cfg<BN, kMode>::kThreads), 1) k_gemm(const __grid_constant__ CUtensorMap tmA,
                                                          const __grid_constant__ CUtensorMap tmB0,
                                                          const __grid_constant__ CUtensorMap tmB1,
                                                          const __grid_constant__ GemmGrid G, int* err)
{
    using C = Cfg<BN, kMode>;
    constexpr int kStages = C::kStages, kEpiWarps = C::kEpiWarps;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], tfull[2], tempty[2], drained;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail, s_issued, s_consumed;
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int KT = G.KT;
    const int my_tiles = (G.n_tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    volatile int* fail = &s_fail;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(2 * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int st = 0; st < kStages; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], kEpiWarps);  // one arrival per epilogue warp
        }
        mbar_init(&drained, 1);
        s_fail = 0;
        s_issued = 0;
        s_consumed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base;

    if (tid == 0) {
        // producer: global k-step g of the CTA refills stage g % kStages once the MMAs of step g - kStages have
        // completed
        int g = 0;
        for (int j = 0; j < my_tiles && !*fail; ++j) {
            const int t = (int)blockIdx.x + j * (int)gridDim.x;
            const int sg = t >= G.tiles0, tt = sg ? t - G.tiles0 : t;
            const int z = tt / G.per[sg], r = tt - z * G.per[sg];
            const int m0 = (r / G.tn[sg]) * kBM, n0 = (r % G.tn[sg]) * BN, zA = G.za[sg] + z;
            const CUtensorMap* tmB = sg ? &tmB1 : &tmB0;
            for (int kt = 0; kt < KT; ++kt, ++g) {
                const int st = g % kStages;
                if (g >= kStages && !pp_wait(&empty[st], (unsigned)(g / kStages - 1) & 1u, fail)) {
                    *fail = 1;
                    break;
                }
                unsigned char *sa = smem + st * C::kStageBytes, *sb = sa + kTileA;
                mbar_expect_tx(&full[st], C::kStageBytes);
                if (kMnA) {
                    tma_load_3d(sa, &tmA, m0, kt * kBK, zA, &full[st]);
                    tma_load_3d(sa + 8192, &tmA, m0 + 64, kt * kBK, zA, &full[st]);
                } else {
                    tma_load_3d(sa, &tmA, kt * kBK, m0, zA, &full[st]);
                }
                if (kMnB) {
#pragma unroll
                    for (int b = 0; b < BN / 64; ++b)
                        tma_load_3d(sb + 8192 * b, tmB, n0 + 64 * b, kt * kBK, z, &full[st]);
                } else {
                    tma_load_3d(sb, tmB, kt * kBK, n0, z, &full[st]);
                }
                *(volatile int*)&s_issued = g + 1;
            }
        }
    } else if (tid == 32) {
        // MMA issuer: tile j into accumulator j % 2 once the epilogue has drained tile j - 2 from it
        int g = 0;
        bool ok = true;
        for (int j = 0; j < my_tiles && ok; ++j) {
            const int b = j & 1;
            if (j >= 2 && !pp_wait(&tempty[b], (unsigned)((j >> 1) - 1) & 1u, fail)) {
                ok = false;
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + (uint32_t)(b * BN);
            for (int kt = 0; kt < KT; ++kt, ++g) {
                const int st = g % kStages;
                if (!pp_wait(&full[st], (unsigned)(g / kStages) & 1u, fail)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = smem_u32(smem + st * C::kStageBytes);
                const uint32_t sb = sa + kTileA;
#pragma unroll
                for (int kk = 0; kk < kBK / 16; ++kk)
                    mma_bf16(acc, desc_sw128<kMnA>(sa, kk), desc_sw128<kMnB>(sb, kk), C::idesc(kMnA, kMnB),
                             (kt | kk) != 0);
                mma_commit(&empty[st]);
                *(volatile int*)&s_consumed = g + 1;
            }
            if (ok) mma_commit(&tfull[b]);
        }
        if (!ok) *fail = 1;
        // every MMA issued has completed before the accumulators are freed (waited for even after a failure)
        mma_commit(&drained);
        mbar_wait(&drained, 0);
    } else if (warp >= 2) {
        // epilogue: warp w owns tile rows (TMEM lanes) 32 (w % 4) .. 32 (w % 4) + 31 and a share of the columns
        constexpr int kCols = BN / (kEpiWarps / 4) < 32 ? 32 : BN / (kEpiWarps / 4);
        constexpr int kShares = BN / kCols;  // warps beyond them (64 columns, 16 warps) only hand back
        const int q = warp & 3, share = (warp - 2) >> 2, c_off = share * kCols;
        unsigned char* stage = smem + C::kPipe + (warp - 2) * C::kWarpStage;
        float* sf = reinterpret_cast<float*>(stage);
        __nv_bfloat16* sh = reinterpret_cast<__nv_bfloat16*>(stage + (C::kF32 ? kWarpF : 0));
        const int fr = lane >> 3, fc = 4 * (lane & 7);  // FP32 staging: 16-byte piece of rows fr, fr + 4, ...
        const int hr = lane >> 2, hc = 8 * (lane & 3);  // BF16 staging: 16-byte piece of rows hr, hr + 8, ...
        for (int j = 0; j < my_tiles; ++j) {
            const int b = j & 1;
            const int t = (int)blockIdx.x + j * (int)gridDim.x;
            const int sg = t >= G.tiles0, tt = sg ? t - G.tiles0 : t;
            const int z = tt / G.per[sg], r = tt - z * G.per[sg];
            const int m0 = (r / G.tn[sg]) * kBM + 32 * q, n0 = (r % G.tn[sg]) * BN + c_off;
            const GemmEpi& ep = G.ep[sg];
            const int layer = z / G.n_inner, member = z - layer * G.n_inner;
            const long long gc = layer * ep.sl_c + member * ep.sg_c;
            float4 zr[8];  // GELU derivative: the chunk's pre-activations, coalesced, loaded ahead
            const float* zp = nullptr;
            if (kMode == kEpiGeluGrad) {
                zp = ep.z + member * ep.sg_z + (size_t)(m0 + fr) * ep.ldz + n0 + fc;
#pragma unroll
                for (int i = 0; i < 8; ++i) zr[i] = *reinterpret_cast<const float4*>(zp + (size_t)(4 * i) * ep.ldz);
            }
            // warp-uniform decision: the TMEM loads below are warp-collective
            if (!__all_sync(0xffffffffu, pp_wait(&tfull[b], (unsigned)(j >> 1) & 1u, fail))) {
                *fail = 1;
                break;
            }
            tc_fence_after();
            const uint32_t acc = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * BN + c_off);
            uint32_t vn[32];
            if (share < kShares) tmem_ld32(acc, vn);
#pragma unroll 1
            for (int c0 = 0; c0 < kCols; c0 += 32) {
                float v[32];
                tmem_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(vn[i]);
                if (c0 + 32 < kCols) {
                    tmem_ld32(acc + c0 + 32, vn);  // the next chunk's columns arrive during this one's epilogue
                } else {
                    // the accumulator is in registers: hand it back to the MMA issuer
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[b])) : "memory");
                    if (share >= kShares) break;
                }
                if (kMode == kEpiF32) {
#pragma unroll
                    for (int i = 0; i < 32; i += 4)
                        *reinterpret_cast<float4*>(sf + lane * kLdF + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
                } else if (kMode == kEpiBiasGelu || kMode == kEpiGelu) {
                    const float4* bias = reinterpret_cast<const float4*>(ep.bias + member * ep.sg_bias + n0 + c0);
#pragma unroll
                    for (int i = 0; i < 32; i += 8) {
                        uint32_t o[4];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const float4 bb = bias[i / 4 + u];
                            const float* w = v + i + 4 * u;
                            const float z0 = w[0] + bb.x, z1 = w[1] + bb.y, z2 = w[2] + bb.z, z3 = w[3] + bb.w;
                            if (C::kF32) *reinterpret_cast<float4*>(sf + lane * kLdF + i + 4 * u) = make_float4(z0, z1, z2, z3);
                            o[2 * u] = pack_bf16(gelu(z0), gelu(z1));
                            o[2 * u + 1] = pack_bf16(gelu(z2), gelu(z3));
                        }
                        *reinterpret_cast<uint4*>(sh + lane * kLdH + i) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                } else {  // kEpiGeluGrad: dz = acc * gelu'(z)
#pragma unroll
                    for (int i = 0; i < 8; ++i) *reinterpret_cast<float4*>(sf + (fr + 4 * i) * kLdF + fc) = zr[i];
                    if (c0 + 32 < kCols) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            zr[i] = *reinterpret_cast<const float4*>(zp + (size_t)(4 * i) * ep.ldz + c0 + 32);
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 32; i += 8) {
                        uint32_t o[4];
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const float4 zz = *reinterpret_cast<const float4*>(sf + lane * kLdF + i + 4 * u);
                            const float* w = v + i + 4 * u;
                            o[2 * u] = pack_bf16(w[0] * gelu_grad(zz.x), w[1] * gelu_grad(zz.y));
                            o[2 * u + 1] = pack_bf16(w[2] * gelu_grad(zz.z), w[3] * gelu_grad(zz.w));
                        }
                        *reinterpret_cast<uint4*>(sh + lane * kLdH + i) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
                }
                __syncwarp();
                if (kMode == kEpiF32 || kMode == kEpiBiasGelu) {
                    float* o = ep.c_f32 + gc + (size_t)(m0 + fr) * ep.ldc + n0 + c0 + fc;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *reinterpret_cast<float4*>(o + (size_t)(4 * i) * ep.ldc) =
                            *reinterpret_cast<const float4*>(sf + (fr + 4 * i) * kLdF + fc);
                }
                if (kMode != kEpiF32) {
                    __nv_bfloat16* o = ep.out_bf16 + member * ep.sg_o + (size_t)(m0 + hr) * ep.ldo + n0 + c0 + hc;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        *reinterpret_cast<uint4*>(o + (size_t)(8 * i) * ep.ldo) =
                            *reinterpret_cast<const uint4*>(sh + (hr + 8 * i) * kLdH + hc);
                }
                __syncwarp();  // the staging rows are rewritten by the next chunk
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*fail && tid == 0) {
        atomicExch(err, 1);
        // let the loads still in flight land before the CTA's shared memory goes away
        for (int g = s_consumed; g < s_issued; ++g) mbar_wait(&full[g % kStages], (unsigned)(g / kStages) & 1u);
    }
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN) : "memory");
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

cudaError_t get_encode()
{
    if (g_encode) return cudaSuccess;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return e != cudaSuccess ? e : cudaErrorNotSupported;
    g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    return cudaSuccess;
}

// BF16 tensor map (inner, rows, groups) over a matrix with contiguous rows of
// `inner` elements (row stride ld, group stride sg elements), box of 64 inner
// elements x box_rows rows, 128-byte swizzle
cudaError_t make_map(CUtensorMap* m, const GemmOperand& p, int inner, int rows, int box_rows)
{
    cudaError_t e = get_encode();
    if (e != cudaSuccess) return e;
    const long long sg = p.groups > 1 ? p.sg : (long long)p.ld * rows;
    cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)rows, (cuuint64_t)p.groups};
    cuuint64_t strides[2] = {(cuuint64_t)p.ld * 2, (cuuint64_t)sg * 2};
    cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(p.p), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

bool operand_ok(const GemmOperand& p)
{
    return p.p && p.groups > 0 && p.ld % 8 == 0 && ((uintptr_t)p.p & 15) == 0 && (p.groups == 1 || p.sg % 8 == 0);
}

template <int BN, bool kMnA, bool kMnB, int kMode>
cudaError_t launch_gemm(const GemmProblem& P, int sms, int dev, int* err, cudaStream_t st)
{
    static bool attr[64] = {false};  // per device
    if (!attr[dev]) {
        cudaError_t e = cudaFuncSetAttribute(k_gemm<BN, kMnA, kMnB, kMode>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (Cfg<BN, kMode>::kSmem));
        if (e != cudaSuccess) return e;
        attr[dev] = true;
    }
    CUtensorMap ta, tb[2];
    cudaError_t e = kMnA ? make_map(&ta, P.A, P.M, P.K, kBK) : make_map(&ta, P.A, P.K, P.M, kBM);
    for (int s = 0; s < 2 && e == cudaSuccess; ++s) {
        if (s == 1 && !P.n2) {
            tb[1] = tb[0];
            break;
        }
        const GemmOperand& B = s ? P.B2 : P.B;
        const int N = s ? P.n2 : P.N;
        e = kMnB ? make_map(&tb[s], B, N, P.K, kBK) : make_map(&tb[s], B, P.K, N, BN);
    }
    if (e != cudaSuccess) return e;
    GemmGrid g;
    g.KT = P.K / kBK;
    g.n_inner = P.n_inner;
    for (int s = 0; s < 2; ++s) {
        const int N = s && P.n2 ? P.n2 : P.N;
        g.tn[s] = N / BN;
        g.per[s] = (P.M / kBM) * (N / BN);
        g.za[s] = s ? P.za2 : P.za;
        g.ep[s] = s ? P.ep2 : P.ep;
    }
    g.tiles0 = P.groups * g.per[0];
    g.n_tiles = g.tiles0 + (P.n2 ? P.groups2 * g.per[1] : 0);
    k_gemm<BN, kMnA, kMnB, kMode><<<g.n_tiles < sms ? g.n_tiles : sms, Cfg<BN, kMode>::kThreads, (Cfg<BN, kMode>::kSmem), st>>>(ta, tb[0], tb[1],
                                                                                                      g, err);
    return cudaGetLastError();
}

template <bool kMnA, bool kMnB, int kMode>
cudaError_t launch_gemm_bn(const GemmProblem& P, int sms, int dev, int* err, cudaStream_t st)
{
    // 128 x 128 tiles of the whole launch
    const long long tiles = (long long)(P.M / kBM) * ((long long)P.groups * (P.N / 128) + (long long)P.groups2 * (P.n2 / 128));
    if (tiles >= (1ll << 30)) return cudaErrorInvalidValue;
    // 256 columns (three quarters of the operand reads per output) where half the tiles still make an even last
    // wave and the epilogue stores BF16 only: 300k x 4 members' prediction 6.85 against 8.3 ms with 128 columns. With
    // FP32 pre-activations stored or read the epilogue's memory traffic sets the time and smaller tiles balance
    // better: 43 against 48 us per forward layer of 4 x 8192 rows.
    if constexpr (kMode == kEpiGelu)
        if (P.N % 256 == 0 && P.n2 % 256 == 0 && tiles >= 4ll * sms)
            return launch_gemm<256, kMnA, kMnB, kMode>(P, sms, dev, err, st);
    // A wave of tiles of 64, 128 and 256 columns takes times like 344, 408 and 536 (22, 26.6 and 34.6 us at K = 4096),
    // so what counts is how many waves there are: 64 columns pay where they are one wave (128 x 8192 x 4096: 25 us,
    // 26.6 with 128), 128 where 64 would be two (512 x 4096 x 4096: 26.6, 43.9 with 64), and for the plain product,
    // whose epilogue only stores, 256 where that saves more waves than it lengthens (2048 x 1280 x 8192: 59 us, 83
    // with 128; 4096 x 4096 x 4096: 112, 143; 65536 x 512 x 512: 46, 49.5)
    auto waves = [&](long long n) { return (n + sms - 1) / sms; };
    if constexpr (kMode == kEpiF32 && !kMnA && !kMnB)
        if (P.N % 256 == 0 && !P.n2 && 2 * tiles > sms && 536 * waves((tiles + 1) / 2) < 408 * waves(tiles))
            return launch_gemm<256, kMnA, kMnB, kMode>(P, sms, dev, err, st);
    if (2 * tiles > sms) return launch_gemm<128, kMnA, kMnB, kMode>(P, sms, dev, err, st);
    return launch_gemm<64, kMnA, kMnB, kMode>(P, sms, dev, err, st);
}

}  // namespace

bool gemm_shape_ok(int M, int N, int K)
{
    return M > 0 && N > 0 && K > 0 && M % kBM == 0 && N % 128 == 0 && K % kBK == 0;
}

cudaError_t gemm_bf16(const GemmProblem& P, int* err, cudaStream_t st)
{
    if (!gemm_shape_ok(P.M, P.N, P.K) || !operand_ok(P.A) || !operand_ok(P.B) || P.groups < 1 || P.n_inner < 1)
        return cudaErrorInvalidValue;
    if (P.n2 && (!gemm_shape_ok(P.M, P.n2, P.K) || !operand_ok(P.B2) || P.groups2 < 1 || P.ep2.mode != P.ep.mode))
        return cudaErrorInvalidValue;
    for (int s = 0; s < (P.n2 ? 2 : 1); ++s) {
        const GemmEpi& ep = s ? P.ep2 : P.ep;
        if ((ep.mode == kEpiF32 || ep.mode == kEpiBiasGelu) && (!ep.c_f32 || ep.ldc % 4 || ((uintptr_t)ep.c_f32 & 15) || ep.sg_c % 4 || ep.sl_c % 4))
            return cudaErrorInvalidValue;
        if (ep.mode != kEpiF32 && (!ep.out_bf16 || ep.ldo % 8 || ((uintptr_t)ep.out_bf16 & 15) || ep.sg_o % 8))
            return cudaErrorInvalidValue;
        if ((ep.mode == kEpiBiasGelu || ep.mode == kEpiGelu) && (!ep.bias || ((uintptr_t)ep.bias & 15) || ep.sg_bias % 4))
            return cudaErrorInvalidValue;
        if (ep.mode == kEpiGeluGrad && (!ep.z || ep.ldz % 4 || ((uintptr_t)ep.z & 15) || ep.sg_z % 4))
            return cudaErrorInvalidValue;
    }
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || sms < 1) return cudaErrorInvalidDevice;
    if (P.ep.mode == kEpiBiasGelu && !P.A.mn && !P.B.mn)
        return launch_gemm_bn<false, false, kEpiBiasGelu>(P, sms, dev, err, st);
    if (P.ep.mode == kEpiGelu && !P.A.mn && !P.B.mn)
        return launch_gemm_bn<false, false, kEpiGelu>(P, sms, dev, err, st);
    if (P.ep.mode == kEpiGeluGrad && !P.A.mn && P.B.mn)
        return launch_gemm_bn<false, true, kEpiGeluGrad>(P, sms, dev, err, st);
    if (P.ep.mode == kEpiF32 && P.A.mn && P.B.mn) return launch_gemm_bn<true, true, kEpiF32>(P, sms, dev, err, st);
    if (P.ep.mode == kEpiF32 && !P.A.mn && !P.B.mn) return launch_gemm_bn<false, false, kEpiF32>(P, sms, dev, err, st);
    return cudaErrorInvalidValue;  // no other combination is used
}

}  // namespace sbr
