// sbr_surrogate.cu -- learned surrogate of the SBR field: a Fourier-feature MLP
// in BF16 with FP32 accumulation whose forward and backward products run on
// the tcgen05 tensor-core GEMM of sbr_gemm.cu.
//
// Network (per ensemble member): input (az, el, f) -> (sin az, cos az, el / 30
// deg, log-frequency mapped to [-1, 1]) -> Fourier features [sin 2 pi B x,
// cos 2 pi B x] (B fixed, N(0, sigma^2)) -> depth x (width GELU) -> 4 outputs
// (Re and Im of HH and VV, divided by a target scale). Hidden layers: BF16
// activations and weights, FP32 accumulation (tcgen05 GEMM), FP32 master weights
// with Adam. The 4-output head runs on CUDA cores.
//
// One training step on a batch of M samples (M a multiple of 128):
//   forward  h0 = FF(x); z_l = h_l W_l^T + b_l, h_{l+1} = GELU(z_l)   (GEMM, fused epilogue)
//            y = h_D W_h^T + b_h                                        (head kernel)
//   loss     mean squared error over the 4 outputs
//   backward dz_{D-1} = (dy W_h) * GELU'(z_{D-1});
//            dz_{l-1} = (dz_l W_l) * GELU'(z_{l-1})                     (GEMM, fused epilogue)
//            dW_l = dz_l^T h_l (one GEMM launch for all layers), db_l = sum_m dz_l
//   Adam on all FP32 parameters, the BF16 copies of W_l written with them.
// The members of the ensemble take each step together (grouped launches).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <mutex>
#include <random>
#include <string>
#include <thread>
#include <vector>

#include "sbr.h"
#include "sbr_internal.h"

using namespace sbr;

namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr int kMaxDepth = 16;
constexpr int kMaxMembers = 16;
constexpr int kOut = 4;
constexpr int kIn = 4;

std::mutex g_gemm_mu;
int* g_gemm_err[64] = {nullptr};

// ---------------------------------------------------------------- small kernels
// Every kernel below works on a group of members at once (a grid dimension is
// the member, its arrays a fixed stride apart): one member's arrays are too
// small to fill the GPU, and a launch costs as much as its work. Each sum keeps
// its order whatever the group, so the members' results do not depend on it.

// raw (az deg, el deg, f Hz) -> the 4 network inputs
__global__ void k_encode(const double* raw, int n, float* x4)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double az = raw[3 * i] * (kPi / 180.0), el = raw[3 * i + 1], f = raw[3 * i + 2];
    x4[4 * i + 0] = (float)sin(az);
    x4[4 * i + 1] = (float)cos(az);
    x4[4 * i + 2] = (float)(el / 30.0);
    x4[4 * i + 3] = (float)(2.0 * (log(f / 1e9) / log(12.0)) - 1.0);
}

// member blockIdx.y's batch: rows idx[member * n_idx + i], i < n
__global__ void k_gather(const float4* x4, const float4* y4, const int* idx, long long n_idx, int n, float4* xb,
                         float4* yb)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int j = idx[blockIdx.y * n_idx + i];
    const size_t o = (size_t)blockIdx.y * n + i;
    xb[o] = x4[j];
    yb[o] = y4[j];
}

// Fourier features: h0[m][j] = sin(2 pi B_j . x_m) (j < nf/2), cos(...) (j >= nf/2); two frequencies per thread.
// sx: rows between the members' inputs (0: all members read the same)
__global__ void k_fourier(const float4* x4, long long sx, const float4* B, int M, int nh, __nv_bfloat16* h0)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int half = nh / 2;
    if (i >= (long long)M * half) return;
    const int m = (int)(i / half), j = 2 * (int)(i % half);
    const float4 x = x4[blockIdx.y * sx + m];
    __nv_bfloat162 sv, cv;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float4 b = B[(size_t)blockIdx.y * nh + j + u];
        const float arg = b.x * x.x + b.y * x.y + b.z * x.z + b.w * x.w;
        float s, c;
        sincospif(2.f * arg, &s, &c);
        (u ? sv.y : sv.x) = __float2bfloat16_rn(s);
        (u ? cv.y : cv.x) = __float2bfloat16_rn(c);
    }
    __nv_bfloat16* o = h0 + ((size_t)blockIdx.y * M + m) * (2 * nh) + j;
    *reinterpret_cast<__nv_bfloat162*>(o) = sv;
    *reinterpret_cast<__nv_bfloat162*>(o + nh) = cv;
}

__device__ __forceinline__ float gelu_grad_f(float z)
{
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// head: y[m][o] = sum_k h[m][k] W[o][k] + b[o]; one warp per row, lane l the terms k = l, l + 32, ...
__global__ void k_head_fwd(const __nv_bfloat16* h, int M, int K, const float* P, long long sp, long long ow,
                           long long ob, float* y)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (warp >= M) return;
    const float* W = P + blockIdx.y * sp + ow;
    const float* b = P + blockIdx.y * sp + ob;
    const __nv_bfloat16* row = h + ((size_t)blockIdx.y * M + warp) * K;
    float acc[kOut] = {0.f, 0.f, 0.f, 0.f};
    for (int k = lane; k < K; k += 32) {
        const float v = __bfloat162float(row[k]);
#pragma unroll
        for (int o = 0; o < kOut; ++o) acc[o] = fmaf(v, W[o * K + k], acc[o]);
    }
#pragma unroll
    for (int o = 0; o < kOut; ++o)
        for (int s = 16; s > 0; s >>= 1) acc[o] += __shfl_xor_sync(0xffffffffu, acc[o], s);
    if (lane == 0)
#pragma unroll
        for (int o = 0; o < kOut; ++o) y[((size_t)blockIdx.y * M + warp) * kOut + o] = acc[o] + b[o];
}

// The same for widths up to 512 (kT terms per lane): the weights stay in registers while a warp walks its rows
// (reading them again for every row was four loads per activation), and the four sums are reduced together, each
// lane keeping the half it will finish (6 exchanges instead of 20, every sum in the order of the plain butterfly).
// Bound by loads in flight: 17 us for 4 x 8192 rows, 25 us by k_head_fwd.
template <int kT>
__global__ void __launch_bounds__(256) k_head_fwd_reg(const __nv_bfloat16* __restrict__ h, int M,
                                                      const float* __restrict__ P, long long sp, long long ow,
                                                      long long ob, float* __restrict__ y)
{
    constexpr int K = 32 * kT;
    const int lane = threadIdx.x & 31, nw = (gridDim.x * blockDim.x) >> 5;
    const float* W = P + blockIdx.y * sp + ow;
    float w[kOut][kT];
#pragma unroll
    for (int o = 0; o < kOut; ++o)
#pragma unroll
        for (int i = 0; i < kT; ++i) w[o][i] = W[o * K + 32 * i + lane];
    const bool b16 = lane & 16, b8 = lane & 8;
    const int out = (b16 ? 2 : 0) + (b8 ? 1 : 0);
    const float bias = P[blockIdx.y * sp + ob + out];
    for (int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; m < M; m += nw) {
        const __nv_bfloat16* row = h + ((size_t)blockIdx.y * M + m) * K + lane;
        float v[kT];
#pragma unroll
        for (int i = 0; i < kT; ++i) v[i] = __bfloat162float(row[32 * i]);
        float acc[kOut] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < kT; ++i)
#pragma unroll
            for (int o = 0; o < kOut; ++o) acc[o] = fmaf(v[i], w[o][i], acc[o]);
        const float r0 = __shfl_xor_sync(0xffffffffu, b16 ? acc[0] : acc[2], 16);
        const float r1 = __shfl_xor_sync(0xffffffffu, b16 ? acc[1] : acc[3], 16);
        const float a0 = (b16 ? acc[2] : acc[0]) + r0, a1 = (b16 ? acc[3] : acc[1]) + r1;
        float a = (b8 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, b8 ? a0 : a1, 8);
#pragma unroll
        for (int s = 4; s > 0; s >>= 1) a += __shfl_xor_sync(0xffffffffu, a, s);
        if ((lane & 7) == 0) y[((size_t)blockIdx.y * M + m) * kOut + out] = a + bias;
    }
}

// dy = 2 (y - t) / (M * 4); loss sum in FP64 (loss[member * sl])
__global__ void k_loss(const float* y, const float* t, int n, float* dy, double* loss, int sl)
{
    __shared__ double s_red[8];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t g = (size_t)blockIdx.y * n;
    double l = 0.0;
    if (i < n) {
        const float d = y[g + i] - t[g + i];
        dy[g + i] = 2.f * d / (float)n;
        l = (double)d * d;
    }
    for (int s = 16; s > 0; s >>= 1) l += __shfl_xor_sync(0xffffffffu, l, s);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = l;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t2 = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t2 += s_red[w];
        atomicAdd(loss + (size_t)blockIdx.y * sl, t2);
    }
}

// dz[m][k] = (sum_o dy[m][o] W[o][k]) * gelu'(z[m][k]), four k per thread
__global__ void k_head_bwd_dz(const float4* dy, const float* P, long long sp, long long ow, const float4* z, int M,
                              int K, uint2* dz)
{
    const int k4 = K / 4;
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= (long long)M * k4) return;
    const int m = (int)(i / k4), k = 4 * (int)(i % k4);
    const float* W = P + blockIdx.y * sp + ow;
    const float4 d4 = dy[(size_t)blockIdx.y * M + m];
    const float d[kOut] = {d4.x, d4.y, d4.z, d4.w};
    const size_t at = (size_t)blockIdx.y * M * k4 + i;
    const float4 zz = z[at];
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
        const float4 w = *reinterpret_cast<const float4*>(W + (size_t)o * K + k);
        s[0] = fmaf(d[o], w.x, s[0]);
        s[1] = fmaf(d[o], w.y, s[1]);
        s[2] = fmaf(d[o], w.z, s[2]);
        s[3] = fmaf(d[o], w.w, s[3]);
    }
    __nv_bfloat162 a = __floats2bfloat162_rn(s[0] * gelu_grad_f(zz.x), s[1] * gelu_grad_f(zz.y));
    __nv_bfloat162 b = __floats2bfloat162_rn(s[2] * gelu_grad_f(zz.z), s[3] * gelu_grad_f(zz.w));
    dz[at] = make_uint2(*reinterpret_cast<unsigned*>(&a), *reinterpret_cast<unsigned*>(&b));
}

// Column sums over the batch in two fixed-order stages (deterministic): stage 1
// gives one partial per kRedRows rows (block 32 columns x 8 row lanes), stage 2
// adds the partials in order.
constexpr int kRedRows = 256;

// head gradient, stage 1: part[p][o][k] = sum over rows m of chunk p of dy[m][o] h[m][k]
// (k < K) and of dy[m][o] (k = K, the bias); member blockIdx.z
__global__ void k_head_dw_part(const float* dy, const __nv_bfloat16* h, int M, int K, float* part)
{
    __shared__ float sh[8][kOut][33];
    const int k = blockIdx.x * 32 + threadIdx.x, p = blockIdx.y;
    dy += (size_t)blockIdx.z * M * kOut;
    h += (size_t)blockIdx.z * M * K;
    part += (size_t)blockIdx.z * gridDim.y * kOut * (K + 1);
    float acc[kOut] = {0.f, 0.f, 0.f, 0.f};
    if (k <= K) {
        const int r1 = min(M, (p + 1) * kRedRows);
#pragma unroll 4
        for (int m = p * kRedRows + threadIdx.y; m < r1; m += 8) {
            const float v = k < K ? __bfloat162float(h[(size_t)m * K + k]) : 1.f;
#pragma unroll
            for (int o = 0; o < kOut; ++o) acc[o] = fmaf(dy[m * kOut + o], v, acc[o]);
        }
    }
#pragma unroll
    for (int o = 0; o < kOut; ++o) sh[threadIdx.y][o][threadIdx.x] = acc[o];
    __syncthreads();
    if (threadIdx.y < kOut && k <= K) {
        const int o = threadIdx.y;
        float t = 0.f;
        for (int y = 0; y < 8; ++y) t += sh[y][o][threadIdx.x];
        part[((size_t)p * kOut + o) * (K + 1) + k] = t;
    }
}

// head gradient, stage 2: dW[o][k], db[o] = sum over the n_part partials; member blockIdx.y
__global__ void k_head_dw_fin(const float* part, int n_part, int K, float* G, long long sp, long long ow, long long ob)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= kOut * (K + 1)) return;
    part += (size_t)blockIdx.y * n_part * kOut * (K + 1);
    const int o = j / (K + 1), k = j % (K + 1);
    float t = 0.f;
    for (int q = 0; q < n_part; ++q) t += part[((size_t)q * kOut + o) * (K + 1) + k];
    if (k < K) G[blockIdx.y * sp + ow + o * K + k] = t;
    else G[blockIdx.y * sp + ob + o] = t;
}

// bias gradient, stage 1: part[p][n] = sum over rows m of chunk p of dz[m][n]; (layer, member) blockIdx.z; four
// columns per thread (8-byte loads; N is a multiple of 128)
__global__ void __launch_bounds__(256) k_colsum_part(const __nv_bfloat16* dz, int M, int N, float* part)
{
    __shared__ float4 sh[8][32];
    const int n = blockIdx.x * 128 + 4 * threadIdx.x, p = blockIdx.y;
    dz += (size_t)blockIdx.z * M * N + n;
    part += (size_t)blockIdx.z * gridDim.y * N;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const int r1 = min(M, (p + 1) * kRedRows);
#pragma unroll 8
    for (int m = p * kRedRows + threadIdx.y; m < r1; m += 8) {
        const uint2 u = *reinterpret_cast<const uint2*>(dz + (size_t)m * N);
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x)),
                     b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
        acc.x += a.x;
        acc.y += a.y;
        acc.z += b.x;
        acc.w += b.y;
    }
    sh[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y == 0) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int y = 0; y < 8; ++y) {
            const float4 v = sh[y][threadIdx.x];
            t.x += v.x;
            t.y += v.y;
            t.z += v.z;
            t.w += v.w;
        }
        *reinterpret_cast<float4*>(part + (size_t)p * N + n) = t;
    }
}

// offsets of the layers' weights and biases in a member's parameters, and of the BF16 weights (layer depth = head)
struct Layout {
    int depth;
    long long offW[kMaxDepth + 1], offb[kMaxDepth + 1], offWbf[kMaxDepth + 1];
};

// bias gradient, stage 2; blockIdx.y = layer * members + member
__global__ void k_colsum_fin(const float* part, int n_part, int N, int members, float* G, long long sp, const Layout L)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const int layer = blockIdx.y / members, e = blockIdx.y - layer * members;
    part += (size_t)blockIdx.y * n_part * N;
    float t = 0.f;
    for (int q = 0; q < n_part; ++q) t += part[(size_t)q * N + n];
    G[e * sp + L.offb[layer] + n] = t;
}

struct AdamBias {
    float c1[kMaxMembers], c2[kMaxMembers];  // bias corrections of each member of the group
};

__device__ __forceinline__ void adam1(float& p, float& m, float& v, float gi, float lr, float b1, float b2, float c1,
                                      float c2, float eps)
{
    // one rounding per product and sum as written, so that training gives the same bits however it is compiled
    const float mi = __fmaf_rn(1.f - b1, gi, __fmul_rn(b1, m));
    const float vi = __fmaf_rn(__fmul_rn(1.f - b2, gi), gi, __fmul_rn(b2, v));
    m = mi;
    v = vi;
    p -= lr * (mi * c1) / (sqrtf(vi * c2) + eps);
}

// Adam on four parameters per thread, the BF16 copies of the hidden weights written with them
__global__ void k_adam(float* p, float* m, float* v, const float* g, long long n, __nv_bfloat16* wbf, long long n_bf,
                       const Layout L, float lr, float b1, float b2, const AdamBias A, float eps)
{
    const long long i = 4 * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
    if (i >= n) return;
    const int e = blockIdx.y;
    const size_t at = (size_t)e * n + i;
    float4 pp = *reinterpret_cast<float4*>(p + at), mm = *reinterpret_cast<float4*>(m + at),
           vv = *reinterpret_cast<float4*>(v + at);
    const float4 gg = *reinterpret_cast<const float4*>(g + at);
    const float c1 = A.c1[e], c2 = A.c2[e];
    adam1(pp.x, mm.x, vv.x, gg.x, lr, b1, b2, c1, c2, eps);
    adam1(pp.y, mm.y, vv.y, gg.y, lr, b1, b2, c1, c2, eps);
    adam1(pp.z, mm.z, vv.z, gg.z, lr, b1, b2, c1, c2, eps);
    adam1(pp.w, mm.w, vv.w, gg.w, lr, b1, b2, c1, c2, eps);
    *reinterpret_cast<float4*>(p + at) = pp;
    *reinterpret_cast<float4*>(m + at) = mm;
    *reinterpret_cast<float4*>(v + at) = vv;
    for (int l = 0; l < L.depth; ++l)
        if (i >= L.offW[l] && i < L.offb[l]) {
            __nv_bfloat162 a = __floats2bfloat162_rn(pp.x, pp.y), b = __floats2bfloat162_rn(pp.z, pp.w);
            *reinterpret_cast<uint2*>(wbf + (size_t)e * n_bf + L.offWbf[l] + (i - L.offW[l])) =
                make_uint2(*reinterpret_cast<unsigned*>(&a), *reinterpret_cast<unsigned*>(&b));
        }
}

__global__ void k_to_bf16(const float* in, long long n, __nv_bfloat16* out)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) out[i] = __float2bfloat16_rn(in[i]);
}

// ensemble mean (scaled back) and spread: per point, max over HH and VV of the
// range over members of 10 log10 |E|^2
__global__ void k_ens_stats(const float* y, int n_members, long long stride, int n, float scale, double* mean,
                            float* spread)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float mu[kOut] = {0.f, 0.f, 0.f, 0.f};
    float lo[2] = {1e30f, 1e30f}, hi[2] = {-1e30f, -1e30f};
    for (int e = 0; e < n_members; ++e) {
        const float* r = y + e * stride + (size_t)i * kOut;
#pragma unroll
        for (int o = 0; o < kOut; ++o) mu[o] += r[o];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float a2 = r[2 * p] * r[2 * p] + r[2 * p + 1] * r[2 * p + 1];
            const float db = 10.f * log10f(fmaxf(a2, 1e-30f));
            lo[p] = fminf(lo[p], db);
            hi[p] = fmaxf(hi[p], db);
        }
    }
#pragma unroll
    for (int o = 0; o < kOut; ++o) mean[(size_t)i * kOut + o] = (double)(mu[o] / n_members) * scale;
    spread[i] = fmaxf(hi[0] - lo[0], hi[1] - lo[1]);
}

inline unsigned blocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr size_t kKeepBytes = (size_t)64 << 20;

struct Buf {
    void* p = nullptr;
    size_t cap = 0;
    cudaError_t ensure(size_t bytes)
    {
        if (bytes <= cap) return cudaSuccess;
        release();
        const cudaError_t e = cudaMalloc(&p, bytes);
        if (e == cudaSuccess) cap = bytes;
        else p = nullptr;
        return e;
    }
    void release()
    {
        if (p) cudaFree(p);
        p = nullptr;
        cap = 0;
    }
    template <class T>
    T* as() const { return (T*)p; }
};

}  // namespace

// ------------------------------------------------------------------ surrogate state
struct sbr_surrogate {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    sbr_surrogate_opts opt;
    std::string err;
    int nh = 0;  // Fourier frequencies (features = 2 nh)
    std::vector<int> K;  // inputs of hidden layer l (each has width outputs)
    Layout L;
    long long n_params = 0;  // per member (a multiple of 4)
    long long n_bf = 0;      // BF16 hidden weights per member
    // all members, n_params / n_bf / 4 nh apart: parameters, Adam moments, Fourier matrices, BF16 weights
    Buf P, Pm, Pv, Bf, Wbf;
    std::vector<long long> steps;
    // Workspace of a group of g members on a batch of M rows, member-major: h0 [g][M][nf], h [layer][g][M][width]
    // (h_{l+1} at l), z and dz [layer][g][M][width], outputs and targets [g][M][4], gradients [g][n_params]. Kept and
    // grown as needed.
    Buf h0, h, z, dz, y, dy, xb, yb, red, G;
    // Arrays of a call: inputs as given and encoded, targets, permutations and losses, predictions. Kept up to
    // kKeepBytes each: taken from the allocator and given back on every call they cost 0.1 to 0.2 ms whenever they
    // were alone in a mapping of it.
    Buf raw, x4, y4, perm, eloss, mean, spread;
    Buf loss, gerr;
    float target_scale = 1.f;
    bool trained = false;
};

namespace {

int sfail(sbr_surrogate* s, int code, const char* msg)
{
    if (s) s->err = msg;
    return code;
}

#define SCK(call, what)                                                                   \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess) {                                                          \
            cudaGetLastError();                                                           \
            return sfail(s, e_ == cudaErrorMemoryAllocation ? SBR_ERR_OOM : SBR_ERR_CUDA, \
                         (std::string(what) + ": " + cudaGetErrorString(e_)).c_str());    \
        }                                                                                 \
    } while (0)

// the workspace of g members on M rows: `layers` activations kept (all of them for a backward pass, two to
// alternate between for prediction), pre-activations and deltas with `train`
cudaError_t ensure_ws(sbr_surrogate* s, int M, int g, bool train)
{
    const size_t D = (size_t)s->opt.depth, W = (size_t)s->opt.width, R = (size_t)M * g;
    const size_t layers = train ? D : std::min<size_t>(D, 2);
    cudaError_t e = s->h0.ensure(sizeof(__nv_bfloat16) * R * s->opt.n_fourier);
    if (e == cudaSuccess) e = s->h.ensure(sizeof(__nv_bfloat16) * R * W * layers);
    if (e == cudaSuccess) e = s->y.ensure(sizeof(float) * R * kOut);
    if (e == cudaSuccess) e = s->xb.ensure(sizeof(float) * R * kIn);
    if (!train || e != cudaSuccess) return e;
    e = s->z.ensure(sizeof(float) * R * W * D);
    if (e == cudaSuccess) e = s->dz.ensure(sizeof(__nv_bfloat16) * R * W * D);
    if (e == cudaSuccess) e = s->dy.ensure(sizeof(float) * R * kOut);
    if (e == cudaSuccess) e = s->yb.ensure(sizeof(float) * R * kOut);
    if (e == cudaSuccess) e = s->G.ensure(sizeof(float) * (size_t)s->n_params * g);
    const size_t parts = (size_t)((M + kRedRows - 1) / kRedRows) * g;
    if (e == cudaSuccess) e = s->red.ensure(sizeof(float) * parts * std::max<size_t>(kOut * (W + 1), D * W));
    return e;
}

void release_ws(sbr_surrogate* s)
{
    for (Buf* b : {&s->h0, &s->h, &s->z, &s->dz, &s->y, &s->dy, &s->xb, &s->yb, &s->red, &s->G}) b->release();
}

// an array of the call at hand; where the GPU is full the workspace kept from earlier calls makes room
cudaError_t call_alloc(sbr_surrogate* s, Buf& b, size_t bytes)
{
    cudaError_t e = b.ensure(bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        release_ws(s);
        e = b.ensure(bytes);
    }
    return e;
}

// gives back at the end of a call what is too large to keep
struct CallArrays {
    sbr_surrogate* s;
    ~CallArrays()
    {
        for (Buf* b : {&s->raw, &s->x4, &s->y4, &s->perm, &s->eloss, &s->mean, &s->spread})
            if (b->cap > kKeepBytes) b->release();
    }
};

// Members worked on at once: all of them while their workspace (200 MB per
// member at 8192 rows of the default network) stays within kGroupBytes and can
// be had beside the group's permutations (at most kGroupPerm) and losses, else
// fewer, down to one; the call's other arrays are there already. A step of four
// members of 8192 rows takes 0.75 ms of device time together, 3.1 ms one member
// at a time.
constexpr size_t kGroupBytes = (size_t)8 << 30, kGroupPerm = (size_t)1 << 30;
int choose_group(sbr_surrogate* s, int M, long long n, int epochs, int* g_out)
{
    const size_t row = (size_t)s->opt.depth * s->opt.width * 8 + (size_t)s->opt.n_fourier * 2 + 128;
    size_t most = std::min<size_t>((size_t)s->opt.n_members, kGroupBytes / (row * (size_t)M));
    most = std::min(most, kGroupPerm / (sizeof(int) * (size_t)n));
    int g = (int)std::max<size_t>(1, most);
    for (bool last = false;;) {
        cudaError_t e = ensure_ws(s, M, g, true);
        if (e == cudaSuccess) e = s->perm.ensure(sizeof(int) * (size_t)n * g);
        if (e == cudaSuccess) e = s->eloss.ensure(sizeof(double) * (size_t)epochs * g);
        if (e == cudaSuccess) break;
        cudaGetLastError();
        release_ws(s);
        for (Buf* b : {&s->perm, &s->eloss, &s->raw, &s->mean, &s->spread}) b->release();
        if (e != cudaErrorMemoryAllocation || last) SCK(e, "alloc training workspace");
        if (g == 1) last = true;  // once more, without what earlier calls had left
        else g = (g + 1) / 2;
    }
    *g_out = g;
    return SBR_OK;
}

// refresh the BF16 copies of the hidden weights of member e
int refresh_bf16(sbr_surrogate* s, int e)
{
    for (int l = 0; l < s->opt.depth; ++l) {
        const long long n = (long long)s->opt.width * s->K[l];
        k_to_bf16<<<blocks(n, 256), 256, 0, s->stream>>>(s->P.as<float>() + e * s->n_params + s->L.offW[l], n,
                                                         s->Wbf.as<__nv_bfloat16>() + e * s->n_bf + s->L.offWbf[l]);
    }
    SCK(cudaGetLastError(), "refresh weights");
    return SBR_OK;
}

// forward pass of members e0 .. e0 + g - 1 on M rows each: fills h0, h and y. sx: rows between the members' inputs
// at xb (0: shared). keep_z: store the FP32 pre-activations and every layer's activations for a backward pass
// (prediction writes only BF16 activations, into two buffers in turn).
int forward(sbr_surrogate* s, int e0, int g, int M, const float* xb, long long sx, float* yout, bool keep_z)
{
    const int D = s->opt.depth, W = s->opt.width, nf = s->opt.n_fourier;
    const long long S = (long long)M * W;
    const float* P = s->P.as<float>() + e0 * s->n_params;
    __nv_bfloat16* h = s->h.as<__nv_bfloat16>();
    auto hl = [&](int l) { return h + (size_t)(keep_z ? l : l & 1) * g * S; };  // h_{l+1}
    k_fourier<<<dim3(blocks((long long)M * (s->nh / 2), 256), g), 256, 0, s->stream>>>(
        (const float4*)xb, sx, s->Bf.as<float4>() + (size_t)e0 * s->nh, M, s->nh, s->h0.as<__nv_bfloat16>());
    for (int l = 0; l < D; ++l) {
        GemmProblem p;
        memset(&p, 0, sizeof(p));
        if (l == 0) p.A = GemmOperand{s->h0.p, nf, false, g, (long long)M * nf};
        else p.A = GemmOperand{hl(l - 1), W, false, g, S};
        p.B = GemmOperand{s->Wbf.as<__nv_bfloat16>() + e0 * s->n_bf + s->L.offWbf[l], s->K[l], false, g, s->n_bf};
        p.M = M;
        p.N = W;
        p.K = s->K[l];
        p.groups = p.n_inner = g;
        p.ep.mode = keep_z ? kEpiBiasGelu : kEpiGelu;
        p.ep.c_f32 = keep_z ? s->z.as<float>() + (size_t)l * g * S : nullptr;
        p.ep.ldc = W;
        p.ep.sg_c = S;
        p.ep.out_bf16 = hl(l);
        p.ep.ldo = W;
        p.ep.sg_o = S;
        p.ep.bias = P + s->L.offb[l];
        p.ep.sg_bias = s->n_params;
        SCK(gemm_bf16(p, s->gerr.as<int>(), s->stream), "forward gemm");
    }
    {
        const __nv_bfloat16* hD = hl(D - 1);
        const long long np = s->n_params, ow = s->L.offW[D], ob = s->L.offb[D];
        // about eight rows per warp pay for the weight loads; no more blocks than stay resident, and fewer rows a warp
        // where the GPU would be half empty (8.5 us for 2,677 rows of one member of width 384 with eight, 3.2 with one)
        const unsigned fill = std::min<unsigned>(blocks(M, 8), 608u / (unsigned)g);
        const dim3 grid(std::min<unsigned>(std::max<unsigned>(blocks(M, 64), fill), 1216u / (unsigned)g + 1u), g);
        if (W == 512) k_head_fwd_reg<16><<<grid, 256, 0, s->stream>>>(hD, M, P, np, ow, ob, yout);
        else if (W == 384) k_head_fwd_reg<12><<<grid, 256, 0, s->stream>>>(hD, M, P, np, ow, ob, yout);
        else if (W == 256) k_head_fwd_reg<8><<<grid, 256, 0, s->stream>>>(hD, M, P, np, ow, ob, yout);
        else if (W == 128) k_head_fwd_reg<4><<<grid, 256, 0, s->stream>>>(hD, M, P, np, ow, ob, yout);
        else
            k_head_fwd<<<dim3(blocks((long long)M * 32, 256), g), 256, 0, s->stream>>>(hD, M, W, P, np, ow, ob, yout);
    }
    SCK(cudaGetLastError(), "head");
    return SBR_OK;
}

// backward pass of the group after forward with keep_z on the same batch (targets in yb): gradients in G (the
// group's first member at G). The sums of squared errors are added to lacc[member * sl].
int backward(sbr_surrogate* s, int e0, int g, int M, double* lacc, int sl)
{
    const int D = s->opt.depth, W = s->opt.width, nf = s->opt.n_fourier;
    const long long S = (long long)M * W, np = s->n_params;
    const float* P = s->P.as<float>() + e0 * np;
    float* G = s->G.as<float>();
    __nv_bfloat16 *h = s->h.as<__nv_bfloat16>(), *dz = s->dz.as<__nv_bfloat16>();
    float* z = s->z.as<float>();
    k_loss<<<dim3(blocks((long long)M * kOut, 256), g), 256, 0, s->stream>>>(s->y.as<float>(), s->yb.as<float>(),
                                                                             M * kOut, s->dy.as<float>(), lacc, sl);
    const int parts = (M + kRedRows - 1) / kRedRows;
    k_head_dw_part<<<dim3((W + 1 + 31) / 32, parts, g), dim3(32, 8), 0, s->stream>>>(
        s->dy.as<float>(), h + (size_t)(D - 1) * g * S, M, W, s->red.as<float>());
    k_head_dw_fin<<<dim3(blocks(kOut * (W + 1), 256), g), 256, 0, s->stream>>>(s->red.as<float>(), parts, W, G, np,
                                                                               s->L.offW[D], s->L.offb[D]);
    k_head_bwd_dz<<<dim3(blocks((long long)M * (W / 4), 256), g), 256, 0, s->stream>>>(
        s->dy.as<float4>(), P, np, s->L.offW[D], (const float4*)(z + (size_t)(D - 1) * g * S), M, W,
        (uint2*)(dz + (size_t)(D - 1) * g * S));
    for (int l = D - 1; l > 0; --l) {
        // dz_{l-1} = (dz_l W_l) * gelu'(z_{l-1}): W_l as stored, its inputs contiguous
        GemmProblem p;
        memset(&p, 0, sizeof(p));
        p.A = GemmOperand{dz + (size_t)l * g * S, W, false, g, S};
        p.B = GemmOperand{s->Wbf.as<__nv_bfloat16>() + e0 * s->n_bf + s->L.offWbf[l], W, true, g, s->n_bf};
        p.M = M;
        p.N = W;
        p.K = W;
        p.groups = p.n_inner = g;
        p.ep.mode = kEpiGeluGrad;
        p.ep.out_bf16 = dz + (size_t)(l - 1) * g * S;
        p.ep.ldo = W;
        p.ep.sg_o = S;
        p.ep.z = z + (size_t)(l - 1) * g * S;
        p.ep.ldz = W;
        p.ep.sg_z = S;
        SCK(gemm_bf16(p, s->gerr.as<int>(), s->stream), "input-gradient gemm");
    }
    // dW_l = dz_l^T h_l, every layer of every member in one launch: the batch is the contraction, both operands
    // as stored; the hidden-to-hidden layers first, then layer 0 on the Fourier features
    {
        GemmProblem p;
        memset(&p, 0, sizeof(p));
        p.A = GemmOperand{dz, W, true, D * g, S};
        p.M = W;
        p.K = M;
        p.n_inner = g;
        p.ep.mode = kEpiF32;
        p.ep.sg_c = np;
        GemmEpi e0p = p.ep;  // layer 0
        e0p.c_f32 = G + s->L.offW[0];
        e0p.ldc = nf;
        const GemmOperand b0{s->h0.p, nf, true, g, (long long)M * nf};
        if (D > 1) {
            p.B = GemmOperand{h, W, true, (D - 1) * g, S};
            p.N = W;
            p.groups = (D - 1) * g;
            p.za = g;
            p.ep.c_f32 = G + s->L.offW[1];
            p.ep.ldc = W;
            p.ep.sl_c = (long long)W * W + W;
            p.B2 = b0;
            p.n2 = nf;
            p.groups2 = g;
            p.ep2 = e0p;
        } else {
            p.B = b0;
            p.N = nf;
            p.groups = g;
            p.ep = e0p;
        }
        SCK(gemm_bf16(p, s->gerr.as<int>(), s->stream), "weight-gradient gemm");
    }
    k_colsum_part<<<dim3(W / 128, parts, D * g), dim3(32, 8), 0, s->stream>>>(dz, M, W, s->red.as<float>());
    k_colsum_fin<<<dim3(blocks(W, 256), D * g), 256, 0, s->stream>>>(s->red.as<float>(), parts, W, g, G, np, s->L);
    SCK(cudaGetLastError(), "backward");
    return SBR_OK;
}

int check_gemm_err(sbr_surrogate* s)
{
    int herr = 0;
    SCK(cudaMemcpyAsync(&herr, s->gerr.p, sizeof(int), cudaMemcpyDeviceToHost, s->stream), "copy error flag");
    SCK(cudaStreamSynchronize(s->stream), "sync");
    if (herr) return sfail(s, SBR_ERR_TIMEOUT, "tensor-core GEMM: a bounded wait gave up");
    return SBR_OK;
}

// the n inputs at x, encoded into s->x4
int upload_inputs(sbr_surrogate* s, const double* x, int64_t n)
{
    SCK(call_alloc(s, s->x4, sizeof(float) * kIn * (size_t)n), "alloc inputs");
    SCK(call_alloc(s, s->raw, sizeof(double) * 3 * (size_t)n), "alloc inputs");
    SCK(cudaMemcpyAsync(s->raw.p, x, sizeof(double) * 3 * (size_t)n, cudaMemcpyHostToDevice, s->stream), "copy inputs");
    k_encode<<<blocks(n, 256), 256, 0, s->stream>>>(s->raw.as<double>(), (int)n, s->x4.as<float>());
    SCK(cudaStreamSynchronize(s->stream), "encode inputs");
    if (s->raw.cap > kKeepBytes) s->raw.release();
    return SBR_OK;
}

}  // namespace

// ------------------------------------------------------------------ C ABI
namespace {
GemmProblem plain_gemm(const void* A, int lda, const void* B, int ldb, int M, int N, int K, float* C, int ldc)
{
    GemmProblem p;
    memset(&p, 0, sizeof(p));
    p.A = GemmOperand{A, lda, false, 1, 0};
    p.B = GemmOperand{B, ldb, false, 1, 0};
    p.M = M;
    p.N = N;
    p.K = K;
    p.groups = p.n_inner = 1;
    p.ep.mode = kEpiF32;
    p.ep.c_f32 = C;
    p.ep.ldc = ldc;
    return p;
}
}  // namespace

extern "C" {

int sbr_gemm_bf16_tn(const void* A, int lda, const void* B, int ldb, int M, int N, int K, float* C, int ldc,
                     void* cuda_stream)
{
    if (!A || !B || !C) return SBR_ERR_ARG;
    if (!gemm_shape_ok(M, N, K) || lda < K || ldb < K || ldc < N || lda % 8 || ldb % 8 || ldc % 4)
        return SBR_ERR_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SBR_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_gemm_mu);
    if (!g_gemm_err[dev]) {
        if (cudaMalloc(&g_gemm_err[dev], sizeof(int)) != cudaSuccess) return SBR_ERR_OOM;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    if (cudaMemsetAsync(g_gemm_err[dev], 0, sizeof(int), st) != cudaSuccess) return SBR_ERR_CUDA;
    if (gemm_bf16(plain_gemm(A, lda, B, ldb, M, N, K, C, ldc), g_gemm_err[dev], st) != cudaSuccess) return SBR_ERR_CUDA;
    int herr = 0;
    if (cudaMemcpyAsync(&herr, g_gemm_err[dev], sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return SBR_ERR_CUDA;
    return herr ? SBR_ERR_TIMEOUT : SBR_OK;
}

int sbr_gemm_bf16_tn_async(const void* A, int lda, const void* B, int ldb, int M, int N, int K, float* C, int ldc,
                           int* err_dev, void* cuda_stream)
{
    if (!A || !B || !C || !err_dev) return SBR_ERR_ARG;
    if (!gemm_shape_ok(M, N, K) || lda < K || ldb < K || ldc < N || lda % 8 || ldb % 8 || ldc % 4)
        return SBR_ERR_ARG;
    return gemm_bf16(plain_gemm(A, lda, B, ldb, M, N, K, C, ldc), err_dev, (cudaStream_t)cuda_stream) == cudaSuccess
               ? SBR_OK
               : SBR_ERR_CUDA;
}

const char* sbr_surrogate_last_error(const sbr_surrogate* s) { return s ? s->err.c_str() : ""; }

int sbr_surrogate_create(sbr_surrogate** out, int device, void* cuda_stream, const sbr_surrogate_opts* opt)
{
    if (!out) return SBR_ERR_ARG;
    *out = nullptr;
    sbr_surrogate_opts o;
    o.n_members = 4;
    o.width = 512;
    o.depth = 6;
    o.n_fourier = 256;
    o.fourier_sigma = 4.f;
    o.seed = 1;
    if (opt) o = *opt;
    if (o.n_members < 1 || o.n_members > kMaxMembers || o.width < 128 || o.width % 128 || o.depth < 1 || o.depth > kMaxDepth ||
        o.n_fourier < 128 || o.n_fourier % 128 || !(o.fourier_sigma > 0.f))
        return SBR_ERR_ARG;
    int nd = 0;
    if (cudaGetDeviceCount(&nd) != cudaSuccess || nd == 0) {
        cudaGetLastError();
        return SBR_ERR_NODEV;
    }
    if (device < 0 || device >= nd || cudaSetDevice(device) != cudaSuccess) return SBR_ERR_ARG;
    sbr_surrogate* s = new sbr_surrogate();
    s->device = device;
    s->opt = o;
    s->nh = o.n_fourier / 2;
    if (cuda_stream) {
        s->stream = (cudaStream_t)cuda_stream;
    } else {
        if (cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete s;
            return SBR_ERR_CUDA;
        }
        s->own_stream = true;
    }
    const int D = o.depth;
    s->K.resize(D);
    memset(&s->L, 0, sizeof(s->L));
    s->L.depth = D;
    long long off = 0, offbf = 0;
    for (int l = 0; l <= D; ++l) {
        if (l < D) s->K[l] = l == 0 ? o.n_fourier : o.width;
        const int Kl = l < D ? s->K[l] : o.width, Nl = l < D ? o.width : kOut;
        s->L.offW[l] = off;
        off += (long long)Nl * Kl;
        s->L.offb[l] = off;
        off += Nl;
        if (l < D) {
            s->L.offWbf[l] = offbf;
            offbf += (long long)Nl * Kl;
        }
    }
    s->n_params = off;
    s->n_bf = offbf;
    const size_t ne = (size_t)o.n_members;
    int rc = SBR_OK;
    if (s->P.ensure(sizeof(float) * off * ne) != cudaSuccess || s->Pm.ensure(sizeof(float) * off * ne) != cudaSuccess ||
        s->Pv.ensure(sizeof(float) * off * ne) != cudaSuccess ||
        s->Bf.ensure(sizeof(float) * 4 * s->nh * ne) != cudaSuccess ||
        s->Wbf.ensure(sizeof(__nv_bfloat16) * offbf * ne) != cudaSuccess ||
        s->loss.ensure(sizeof(double)) != cudaSuccess || s->gerr.ensure(sizeof(int)) != cudaSuccess)
        rc = SBR_ERR_OOM;
    // parameters: He-normal hidden layers, small head, zero biases; Fourier matrix N(0, sigma^2)
    std::mt19937_64 rng(o.seed);
    std::normal_distribution<float> nd01(0.f, 1.f);
    std::vector<float> hp((size_t)off), hb((size_t)4 * s->nh);
    for (int e = 0; e < o.n_members && rc == SBR_OK; ++e) {
        std::fill(hp.begin(), hp.end(), 0.f);
        for (int l = 0; l <= D; ++l) {
            const int Kl = l < D ? s->K[l] : o.width, Nl = l < D ? o.width : kOut;
            const float sd = l < D ? sqrtf(2.f / (float)Kl) : sqrtf(1.f / (float)Kl);
            for (long long i = 0; i < (long long)Nl * Kl; ++i) hp[(size_t)(s->L.offW[l] + i)] = sd * nd01(rng);
        }
        for (auto& v : hb) v = o.fourier_sigma * nd01(rng);
        s->steps.push_back(0);
        // on the object's stream, which nothing else orders after the default one; a pageable source is consumed
        // when the call returns
        if (cudaMemcpyAsync(s->P.as<float>() + e * off, hp.data(), sizeof(float) * off, cudaMemcpyHostToDevice,
                            s->stream) != cudaSuccess ||
            cudaMemcpyAsync(s->Bf.as<float>() + (size_t)e * 4 * s->nh, hb.data(), sizeof(float) * hb.size(),
                            cudaMemcpyHostToDevice, s->stream) != cudaSuccess)
            rc = SBR_ERR_CUDA;
        if (rc == SBR_OK) rc = refresh_bf16(s, e);
    }
    if (rc == SBR_OK && (cudaMemsetAsync(s->Pm.p, 0, s->Pm.cap, s->stream) != cudaSuccess ||
                         cudaMemsetAsync(s->Pv.p, 0, s->Pv.cap, s->stream) != cudaSuccess ||
                         cudaMemsetAsync(s->gerr.p, 0, sizeof(int), s->stream) != cudaSuccess ||
                         cudaStreamSynchronize(s->stream) != cudaSuccess))
        rc = SBR_ERR_CUDA;
    if (rc != SBR_OK) {
        sbr_surrogate_destroy(s);
        return rc;
    }
    *out = s;
    return SBR_OK;
}

void sbr_surrogate_destroy(sbr_surrogate* s)
{
    if (!s) return;
    cudaSetDevice(s->device);
    cudaStreamSynchronize(s->stream);
    release_ws(s);
    for (Buf* b : {&s->P, &s->Pm, &s->Pv, &s->Bf, &s->Wbf, &s->loss, &s->gerr, &s->raw, &s->x4, &s->y4, &s->perm, &s->eloss,
                   &s->mean, &s->spread})
        b->release();
    if (s->own_stream) cudaStreamDestroy(s->stream);
    delete s;
}

int64_t sbr_surrogate_num_params(const sbr_surrogate* s) { return s ? s->n_params : 0; }

int sbr_surrogate_params(sbr_surrogate* s, int member, float* get, const float* set)
{
    if (!s || member < 0 || member >= s->opt.n_members) return SBR_ERR_ARG;
    SCK(cudaSetDevice(s->device), "cudaSetDevice");
    const size_t b = sizeof(float) * (size_t)s->n_params;
    float* p = s->P.as<float>() + member * s->n_params;
    if (set) {
        SCK(cudaMemcpyAsync(p, set, b, cudaMemcpyHostToDevice, s->stream), "set params");
        int rc = refresh_bf16(s, member);
        if (rc != SBR_OK) return rc;
    }
    if (get) SCK(cudaMemcpyAsync(get, p, b, cudaMemcpyDeviceToHost, s->stream), "get params");
    SCK(cudaStreamSynchronize(s->stream), "sync");
    return SBR_OK;
}

int sbr_surrogate_fourier(sbr_surrogate* s, int member, float* B)
{
    if (!s || !B || member < 0 || member >= s->opt.n_members) return SBR_ERR_ARG;
    SCK(cudaSetDevice(s->device), "cudaSetDevice");
    SCK(cudaMemcpy(B, s->Bf.as<float>() + (size_t)member * 4 * s->nh, sizeof(float) * 4 * s->nh, cudaMemcpyDeviceToHost), "get Fourier matrix");
    return SBR_OK;
}

int sbr_surrogate_grads(sbr_surrogate* s, int member, const double* x, const double* y, int64_t n, double* loss,
                        float* grads)
{
    if (!s || !x || !y || n < 128 || n % 128 || member < 0 || member >= s->opt.n_members) return SBR_ERR_ARG;
    SCK(cudaSetDevice(s->device), "cudaSetDevice");
    CallArrays arrays{s};
    int rc = upload_inputs(s, x, n);
    if (rc != SBR_OK) return rc;
    cudaError_t ce = ensure_ws(s, (int)n, 1, true);
    if (ce == cudaErrorMemoryAllocation) {  // once more, without what earlier calls had left
        cudaGetLastError();
        release_ws(s);
        for (Buf* b : {&s->raw, &s->y4, &s->perm, &s->eloss, &s->mean, &s->spread}) b->release();
        ce = ensure_ws(s, (int)n, 1, true);
    }
    SCK(ce, "alloc training workspace");
    std::vector<float> yt((size_t)n * kOut);
    for (size_t i = 0; i < yt.size(); ++i) yt[i] = (float)(y[i] / s->target_scale);
    cudaMemcpyAsync(s->yb.p, yt.data(), sizeof(float) * yt.size(), cudaMemcpyHostToDevice, s->stream);
    cudaMemsetAsync(s->gerr.p, 0, sizeof(int), s->stream);
    cudaMemsetAsync(s->loss.p, 0, sizeof(double), s->stream);
    rc = forward(s, member, 1, (int)n, s->x4.as<float>(), 0, s->y.as<float>(), true);
    if (rc == SBR_OK) rc = backward(s, member, 1, (int)n, s->loss.as<double>(), 0);
    if (rc == SBR_OK) rc = check_gemm_err(s);
    if (rc != SBR_OK) return rc;
    double hl = 0.0;
    SCK(cudaMemcpy(&hl, s->loss.p, sizeof(double), cudaMemcpyDeviceToHost), "copy loss");
    if (loss) *loss = hl / (double)(n * kOut);
    if (grads) SCK(cudaMemcpy(grads, s->G.p, sizeof(float) * (size_t)s->n_params, cudaMemcpyDeviceToHost), "copy grads");
    return SBR_OK;
}

int sbr_surrogate_train(sbr_surrogate* s, const double* x, const double* y, int64_t n, int epochs, int batch,
                        float lr, float* loss_per_epoch)
{
    if (!s || !x || !y || n < 128 || epochs < 1 || batch < 128 || batch % 128 || !(lr > 0.f)) return SBR_ERR_ARG;
    if (n > (1ll << 31) - 1) return SBR_ERR_ARG;
    SCK(cudaSetDevice(s->device), "cudaSetDevice");
    const int M = (int)std::min<long long>(batch, (n / 128) * 128);
    // the call's own arrays first, then the workspace of as many members at once as fit beside them: inputs, targets,
    // and per member of the group one permutation per epoch and the per-epoch squared-error sums
    int group = 1;
    CallArrays arrays{s};
    int rc = upload_inputs(s, x, n);
    if (rc != SBR_OK) return rc;
    SCK(call_alloc(s, s->y4, sizeof(float) * kOut * (size_t)n), "alloc targets");
    rc = choose_group(s, M, n, epochs, &group);
    if (rc != SBR_OK) return rc;
    float *x4 = s->x4.as<float>(), *y4 = s->y4.as<float>();
    int* dperm = s->perm.as<int>();
    double* dloss = s->eloss.as<double>();
    // target scale: RMS of the targets
    double ss = 0.0;
    for (int64_t i = 0; i < n * kOut; ++i) ss += y[i] * y[i];
    s->target_scale = (float)std::max(sqrt(ss / (double)(n * kOut)), 1e-30);
    std::vector<float> yt((size_t)n * kOut);
    for (size_t i = 0; i < yt.size(); ++i) yt[i] = (float)(y[i] / s->target_scale);
    SCK(cudaMemcpyAsync(y4, yt.data(), sizeof(float) * yt.size(), cudaMemcpyHostToDevice, s->stream), "upload targets");
    const long long steps_per_epoch = n / M;
    std::vector<int> perm((size_t)n * group);
    std::vector<double> hloss((size_t)epochs * group);
    cudaMemsetAsync(s->gerr.p, 0, sizeof(int), s->stream);
    const double total_steps = (double)epochs * (double)steps_per_epoch;
    // the members of a group take each step together: they share no data, and one member's batch leaves most of
    // the GPU idle
    for (int e0 = 0; e0 < s->opt.n_members && rc == SBR_OK; e0 += group) {
        const int g = std::min(group, s->opt.n_members - e0);
        std::vector<std::mt19937_64> rng;
        for (int e = 0; e < g; ++e) rng.emplace_back(s->opt.seed * 7919 + (uint64_t)(e0 + e));
        cudaMemsetAsync(dloss, 0, sizeof(double) * (size_t)epochs * g, s->stream);
        long long call_step = 0;
        for (int ep = 0; ep < epochs && rc == SBR_OK; ++ep) {
            auto shuffle = [&](int e) {
                int* pe = perm.data() + (size_t)e * n;
                for (int64_t i = 0; i < n; ++i) pe[i] = (int)i;
                std::shuffle(pe, pe + n, rng[(size_t)e]);
            };
            // each member's permutation on a thread of its own (the GPU waits for the first epoch's)
            std::vector<std::thread> th;
            int started = 0;
            try {
                if (n >= 8192)
                    for (; started < g - 1; ++started) th.emplace_back(shuffle, started);
            } catch (const std::exception&) {  // no thread to be had: the rest here
            }
            for (int e = started; e < g; ++e) shuffle(e);
            for (auto& t : th) t.join();
            // pageable source: the call returns once the host buffer has been consumed
            if (cudaMemcpyAsync(dperm, perm.data(), sizeof(int) * (size_t)n * g, cudaMemcpyHostToDevice, s->stream) !=
                cudaSuccess) {
                rc = sfail(s, SBR_ERR_CUDA, "upload permutation");
                break;
            }
            for (long long st = 0; st < steps_per_epoch && rc == SBR_OK; ++st) {
                k_gather<<<dim3(blocks(M, 256), g), 256, 0, s->stream>>>((const float4*)x4, (const float4*)y4,
                                                                         dperm + st * M, n, M, s->xb.as<float4>(),
                                                                         s->yb.as<float4>());
                rc = forward(s, e0, g, M, s->xb.as<float>(), M, s->y.as<float>(), true);
                if (rc == SBR_OK) rc = backward(s, e0, g, M, dloss + ep, epochs);
                if (rc != SBR_OK) break;
                const float b1 = 0.9f, b2 = 0.999f;
                AdamBias ab;
                for (int e = 0; e < g; ++e) {
                    const long long t = ++s->steps[(size_t)(e0 + e)];
                    ab.c1[e] = 1.f / (1.f - powf(b1, (float)t));
                    ab.c2[e] = 1.f / (1.f - powf(b2, (float)t));
                }
                // cosine schedule lr -> lr / 100 over this call
                const double ph = (double)(call_step++) / std::max(1.0, total_steps - 1.0);
                const float lr_t = (float)(lr * (0.01 + 0.99 * 0.5 * (1.0 + cos(kPi * ph))));
                const size_t at = (size_t)e0 * s->n_params;
                k_adam<<<dim3(blocks(s->n_params / 4, 256), g), 256, 0, s->stream>>>(
                    s->P.as<float>() + at, s->Pm.as<float>() + at, s->Pv.as<float>() + at, s->G.as<float>(), s->n_params,
                    s->Wbf.as<__nv_bfloat16>() + (size_t)e0 * s->n_bf, s->n_bf, s->L, lr_t, b1, b2, ab, 1e-8f);
            }
        }
        if (rc == SBR_OK &&
            (cudaMemcpyAsync(hloss.data(), dloss, sizeof(double) * (size_t)epochs * g, cudaMemcpyDeviceToHost,
                             s->stream) != cudaSuccess ||
             cudaStreamSynchronize(s->stream) != cudaSuccess))
            rc = sfail(s, SBR_ERR_CUDA, "copy losses");
        if (rc == SBR_OK && loss_per_epoch)
            for (int e = 0; e < g; ++e)
                for (int ep = 0; ep < epochs; ++ep)
                    loss_per_epoch[(size_t)(e0 + e) * epochs + ep] =
                        (float)(hloss[(size_t)e * epochs + ep] / ((double)M * kOut * (double)steps_per_epoch));
    }
    if (rc == SBR_OK) rc = check_gemm_err(s);
    if (rc == SBR_OK) s->trained = true;
    return rc;
}

int sbr_surrogate_predict(sbr_surrogate* s, const double* x, int64_t n, double* y_mean, float* spread_db)
{
    if (!s || !x || n < 1 || (!y_mean && !spread_db)) return SBR_ERR_ARG;
    if (n > (1ll << 31) - 1) return SBR_ERR_ARG;
    SCK(cudaSetDevice(s->device), "cudaSetDevice");
    // all members at once, batches of about 512 MB of activations: 65536 rows of the default ensemble. Smaller ones
    // would stay in L2 but pay a pipeline fill and a last wave per launch (64 MB: 12.2, 256 MB: 8.9, 512 MB: 8.1,
    // 1 GB: 7.9 ms for 300k points). The Fourier features of a batch take no more than that either, and where the
    // workspace does not fit beside the call's own arrays the batches are halved (a point's result depends on no
    // other's).
    const int g = s->opt.n_members;
    const long long wide = std::max(4ll * s->opt.width, 2ll * s->opt.n_fourier) * g;
    const long long fit = (512ll << 20) / wide / 128 * 128;
    int M = (int)std::min<int64_t>(std::max<long long>(1024, fit), ((n + 127) / 128) * 128);
    CallArrays arrays{s};
    int rc = upload_inputs(s, x, n);
    if (rc != SBR_OK) return rc;
    SCK(call_alloc(s, s->mean, sizeof(double) * kOut * (size_t)n), "alloc outputs");
    SCK(call_alloc(s, s->spread, sizeof(float) * (size_t)n), "alloc outputs");
    for (bool last = false;;) {
        const cudaError_t e = ensure_ws(s, M, g, false);
        if (e == cudaSuccess) break;
        cudaGetLastError();
        release_ws(s);
        for (Buf* b : {&s->raw, &s->y4, &s->perm, &s->eloss}) b->release();
        if (e != cudaErrorMemoryAllocation || last) SCK(e, "alloc prediction workspace");
        if (M == 128) last = true;  // once more, without what earlier calls had left
        else M = std::max(128, M / 2 / 128 * 128);
    }
    const float* x4 = s->x4.as<float>();
    double* dmean = s->mean.as<double>();
    float* dspread = s->spread.as<float>();
    cudaMemsetAsync(s->gerr.p, 0, sizeof(int), s->stream);
    for (int64_t b0 = 0; b0 < n && rc == SBR_OK; b0 += M) {
        const int cnt = (int)std::min<int64_t>(M, n - b0);
        const int Mp = ((cnt + 127) / 128) * 128;  // padded rows are computed and ignored
        const float* xb = x4 + kIn * b0;
        if (Mp > cnt) {
            cudaMemsetAsync(s->xb.p, 0, sizeof(float) * kIn * (size_t)Mp, s->stream);
            cudaMemcpyAsync(s->xb.p, xb, sizeof(float) * kIn * (size_t)cnt, cudaMemcpyDeviceToDevice, s->stream);
            xb = s->xb.as<float>();
        }
        rc = forward(s, 0, g, Mp, xb, 0, s->y.as<float>(), false);
        if (rc == SBR_OK)
            k_ens_stats<<<blocks(cnt, 256), 256, 0, s->stream>>>(s->y.as<float>(), g, (long long)Mp * kOut, cnt,
                                                                 s->target_scale, dmean + kOut * b0, dspread + b0);
    }
    if (rc == SBR_OK) rc = check_gemm_err(s);
    if (rc == SBR_OK && y_mean)
        rc = cudaMemcpy(y_mean, dmean, sizeof(double) * kOut * (size_t)n, cudaMemcpyDeviceToHost) == cudaSuccess
                 ? SBR_OK
                 : SBR_ERR_CUDA;
    if (rc == SBR_OK && spread_db)
        rc = cudaMemcpy(spread_db, dspread, sizeof(float) * (size_t)n, cudaMemcpyDeviceToHost) == cudaSuccess
                 ? SBR_OK
                 : SBR_ERR_CUDA;
    return rc;
}

}  // extern "C"
