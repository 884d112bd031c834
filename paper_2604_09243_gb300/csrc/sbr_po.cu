// sbr_po.cu -- physical-optics ray-tube sum over the dense valid-hit records
// (Eq. po_sum of the paper; vector form from Eq. em5/em6).
//
// The records of one aspect are cut into items of up to kPoItemRecords tubes. One
// block owns an item: it loads the tubes once and, for every requested
// frequency, evaluates e^{-j k L} per tube, multiplies by the tube coefficients
// and reduces with warp shuffles and a shared-memory tree in FP32. The item
// partial is stored in FP64; a second kernel adds the partials of an aspect in
// a fixed order in FP64, applies -j k / (4 pi) and sigma = 4 pi |E|^2 (Sec. 4).
// The order of every addition is fixed, so results are bitwise reproducible
// (the paper notes run-to-run scatter of its FP32 sums, Sec. 5.1).
//
// Phase: k L is formed in cycles, kappa = f / c0, with kappa and L both held
// as unevaluated two-float sums; the integer part is dropped exactly and the
// fraction goes to sincospi. This keeps the phase error at the FP32 rounding
// of the fraction even for paths of thousands of wavelengths.
#include <math.h>

#include <algorithm>

#include "sbr_internal.h"

namespace sbr {

namespace {

constexpr int kPoThreads = 256;
constexpr int kWarps = kPoThreads / 32;

// kPhase: PoArgs::phase_mode, a kernel each: in one kernel the modes pay for each other's registers and slow paths (500
// frequencies of 12 aircraft aspects, VV, FP32 phase: 0.83 ms, 1.41 where the FP64 phase shares the kernel; four
// polarisations at 64 frequencies, FP64 phase: 3.8 and 4.1 ms)
template <int kPhase>
__device__ __forceinline__ void phase_cs(float4 fq, double kd, float lh, float ll, float& c, float& s)
{
    if (kPhase == 0) {
        const float p = __fmul_rn(fq.x, lh);
        float e = __fmaf_rn(fq.x, lh, -p);
        e = __fadd_rn(e, __fadd_rn(__fmul_rn(fq.x, ll), __fmul_rn(fq.y, lh)));
        const float n = rintf(p);
        const float r = __fadd_rn(__fsub_rn(p, n), e);
        sincospif(2.f * r, &s, &c);
    } else if (kPhase == 1) {
        sincosf(fq.z * lh, &s, &c);
    } else {
        double sd, cd;
        sincos(kd * ((double)lh + (double)ll), &sd, &cd);
        s = (float)sd;
        c = (float)cd;
    }
}

// 2 r of phase_cs's compensated form for two tubes at a frequency (x, -x and y
// twice each), every operation the same rounding on both halves: with the
// product negated, n - p = fma(rint(-p), -1, -p) and r = fma(n - p, -1, e).
__device__ __forceinline__ float2 phase_arg2(float2 fx, float2 nx, float2 fy, float2 lh, float2 ll)
{
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 np = __fmul2_rn(nx, lh);
    float2 e = __ffma2_rn(fx, lh, np);
    // (scalar additions: a packed product and the packed addition that takes it are contracted to one rounding)
    const float2 u = __fmul2_rn(fx, ll), v = __fmul2_rn(fy, lh);
    e = __fadd2_rn(e, make_float2(__fadd_rn(u.x, v.x), __fadd_rn(u.y, v.y)));
    const float2 q = __ffma2_rn(make_float2(rintf(np.x), rintf(np.y)), m1, np);
    const float2 r = __ffma2_rn(q, m1, e);
    return __fadd2_rn(r, r);
}

// Sums of kN values over a warp, every sum in the order of the plain butterfly
// (lane distance 16, 8, 4, 2, 1). As long as a lane holds several values it
// keeps one half of them and sends its partner the other, so that kN values
// take about kN exchanges instead of 5 kN; afterwards lane l holds value
// warp_sum_index<kN>(l).
template <int kN>
__device__ __forceinline__ float warp_sums(float* v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int n = kN, o = 16; o > 0; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = lane & o;
#pragma unroll
            for (int j = 0; j < kN / 2; ++j) {
                if (j >= n) break;
                const float r = __shfl_xor_sync(0xffffffffu, up ? v[j] : v[j + n], o);
                v[j] = (up ? v[j + n] : v[j]) + r;
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
    return v[0];
}
template <int kN>
__device__ __forceinline__ int warp_sum_index(int lane)
{
    return lane / (32 / kN);
}

// kPoPer records per thread (items of kPoPer * kPoThreads records) and room for
// kPol polarisations (2 or 4). A block reduction carries kSums sums: four
// frequencies at a time when kPol = 2, two when kPol = 4, one barrier each
// (the partial sums of consecutive reductions alternate between two buffers).
// Each sum is formed in the same order whatever kPol, so the results do not
// depend on it. Bound by instruction issue (~40 per tube and frequency in the
// phase, sine, cosine and products): 9 aspects of 175k tubes, 201 frequencies, 4
// polarisations in 450 us, 703 G tube-frequencies/s; 472 us with one tube at a
// time (two now share the packed FP32 instructions, and a cosine and a sine
// their products), 635 us with every sum exchanged at every step of the
// butterfly and the other phase modes' code in the loop.
constexpr int kSums = 16;
template <int kPoPer, int kPol, int kPhase>
__global__ void __launch_bounds__(kPoThreads) k_po(const PoArgs a)
{
    constexpr int kF = kSums / (2 * kPol);  // frequencies per block reduction
    __shared__ float s_red[2][kWarps][kSums];
    const int n_items = a.n_items_dev ? *a.n_items_dev : a.n_items;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int buf = 0;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const PoItem I = a.items[item];
        float2 cf[kPoPer][kPol];  // (c, -c): factors of the cosine and sine
        float2 lh[kPoPer / 2], ll[kPoPer / 2];
#pragma unroll
        for (int k = 0; k < kPoPer; ++k) {
            float xh = 0.f, xl = 0.f;
            const int idx = k * kPoThreads + tid;
            if (idx < I.count) {
                const float4* p = reinterpret_cast<const float4*>(a.rec + I.first + idx);
                const float4 x = __ldg(p), y = __ldg(p + 1);
#pragma unroll
                for (int q = 0; q < kPol; ++q) {
                    // coefficient of polarisation pol_sel[q] (a selection, not an indexed local array)
                    const int sel = a.pol_sel[q];
                    const float vec = sel == 0 ? x.x : (sel == 1 ? x.y : (sel == 2 ? x.z : x.w));
                    float v = 0.f;
                    if (q < a.n_pol) v = a.scalar ? (sel < 2 ? y.x : 0.f) : vec;
                    cf[k][q] = make_float2(v, -v);
                }
                xh = y.y;
                xl = y.z;
            } else {
#pragma unroll
                for (int q = 0; q < kPol; ++q) cf[k][q] = make_float2(0.f, 0.f);
            }
            if (k & 1) {
                lh[k / 2].y = xh;
                ll[k / 2].y = xl;
            } else {
                lh[k / 2].x = xh;
                ll[k / 2].x = xl;
            }
        }
        for (int f0 = 0; f0 < I.nf; f0 += kF, buf ^= 1) {
            float2 sum2[kSums / 2];  // (re, im)
#pragma unroll
            for (int v = 0; v < kSums / 2; ++v) sum2[v] = make_float2(0.f, 0.f);
#pragma unroll
            for (int fj = 0; fj < kF; ++fj) {
                if (f0 + fj >= I.nf) break;
                const float4 fq = a.freq[I.f0 + f0 + fj];
                const double kd = kPhase != 2 ? 0.0 : a.kfreq[I.f0 + f0 + fj];
                const float2 fx = make_float2(fq.x, fq.x), nx = make_float2(-fq.x, -fq.x), fy = make_float2(fq.y, fq.y);
#pragma unroll
                for (int k = 0; k < kPoPer; k += 2) {
                    // (a tube past the item's end adds zeros)
                    if (k * kPoThreads + tid >= I.count) break;
                    float2 e0, e1;  // (cos, sin)
                    if constexpr (kPhase == 0) {
                        const float2 t = phase_arg2(fx, nx, fy, lh[k / 2], ll[k / 2]);
                        sincospif(t.x, &e0.y, &e0.x);
                        sincospif(t.y, &e1.y, &e1.x);
                    } else {
                        phase_cs<kPhase>(fq, kd, lh[k / 2].x, ll[k / 2].x, e0.x, e0.y);
                        phase_cs<kPhase>(fq, kd, lh[k / 2].y, ll[k / 2].y, e1.x, e1.y);
                    }
#pragma unroll
                    for (int q = 0; q < kPol; ++q) {
                        float2& v = sum2[fj * kPol + q];
                        v = __ffma2_rn(cf[k][q], e0, v);
                        v = __ffma2_rn(cf[k + 1][q], e1, v);
                    }
                }
            }
            float acc[kSums];
#pragma unroll
            for (int v = 0; v < kSums / 2; ++v) {
                acc[2 * v] = sum2[v].x;
                acc[2 * v + 1] = sum2[v].y;
            }
            const float sum = warp_sums<kSums>(acc);
            if ((lane & 1) == 0) s_red[buf][w][warp_sum_index<kSums>(lane)] = sum;
            __syncthreads();
            if (tid < kSums) {
                const int fj = tid / (2 * kPol), r = tid - fj * (2 * kPol);  // r = 2 q + (0 re, 1 im)
                if (f0 + fj < I.nf && r < 2 * a.n_pol) {
                    float v = 0.f;
#pragma unroll
                    for (int k = 0; k < kWarps; ++k) v += s_red[buf][k][tid];
                    a.partial[I.part + (size_t)(f0 + fj) * (2 * a.n_pol) + r] = (double)v;
                }
            }
        }
    }
}

static_assert(kPoItemRecords == 4 * kPoThreads, "PO item size");

// ---------------------------------------------------------------- staged single-frequency sum
// With one frequency per block reduction (F <= 4 / kPol) the sum reads each
// 32-byte record once and is bound by memory. The records of the items a block
// owns are contiguous ranges; they are streamed in stages of kPoThreads records
// (8 KB) by cp.async.bulk into a ring of kBulkStages shared-memory buffers, one
// mbarrier each, issued ahead across item boundaries, so the loads of the next
// stages overlap the phases, sums and reductions of the current one. Thread t
// takes record k * kPoThreads + t of an item in stage k, in order, so every
// term and every addition is that of k_po: the sums are bit-identical. 4 GB of
// records in 632 us, 6.3 TB/s (840 us with the other phase modes' code inside).
constexpr int kBulkStages = 4;
constexpr unsigned kPoSpin = 1u << 22;  // try_wait rounds before a wait gives up

__device__ __forceinline__ uint32_t po_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool po_wait(uint64_t* bar, unsigned parity)
{
    const uint32_t b = po_smem(bar);
    for (unsigned i = 0; i < kPoSpin; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(b), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

template <int kPol, int kPhase>
__global__ void __launch_bounds__(kPoThreads) k_po_bulk(const PoArgs a)
{
    constexpr int kF = 4 / kPol;
    __shared__ __align__(128) float4 s_rec[kBulkStages][2 * kPoThreads];
    __shared__ __align__(8) uint64_t s_full[kBulkStages];
    __shared__ float s_red[kWarps][8];
    const int n_items = a.n_items_dev ? *a.n_items_dev : a.n_items;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) {
        for (int s = 0; s < kBulkStages; ++s)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(po_smem(&s_full[s])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // producer (thread 0): the next stage to load, as (item, stage of the item), and the stages issued
    int p_item = blockIdx.x, p_k = 0;
    unsigned issued = 0;
    auto produce = [&]() {
        if (p_item >= n_items) return;
        const PoItem I = a.items[p_item];
        const int cnt = min(kPoThreads, I.count - p_k * kPoThreads);
        const int s = (int)(issued % kBulkStages);
        const unsigned bytes = (unsigned)cnt * (unsigned)sizeof(Record);
        // the block's reads of this buffer (generic proxy) come before the copy that overwrites it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(po_smem(&s_full[s])), "r"(bytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                po_smem(&s_rec[s][0])),
            "l"(a.rec + I.first + (long long)p_k * kPoThreads), "r"(bytes), "r"(po_smem(&s_full[s]))
            : "memory");
        ++issued;
        if (++p_k * kPoThreads >= I.count) {
            p_k = 0;
            p_item += gridDim.x;
        }
    };
    if (tid == 0)
        for (int s = 0; s < kBulkStages; ++s) produce();
    unsigned used = 0;  // stages consumed
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const PoItem I = a.items[item];
        float acc[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[v] = 0.f;
        const int n_st = (I.count + kPoThreads - 1) / kPoThreads;
        for (int k = 0; k < n_st; ++k, ++used) {
            const int s = (int)(used % kBulkStages);
            const bool ok = po_wait(&s_full[s], (used / kBulkStages) & 1u);
            if (__syncthreads_or(!ok)) {
                // a stage did not arrive: flag it, poison this item's sums, and leave only once the copies
                // still in flight into this block's buffers have landed (each wait bounded again)
                if (tid == 0) {
                    atomicOr(a.err, 1);
                    for (int r = 0; r < I.nf * 2 * a.n_pol; ++r) a.partial[I.part + r] = __longlong_as_double(-1ll);
                    for (unsigned u = used; u < issued; ++u)
                        po_wait(&s_full[u % kBulkStages], (u / kBulkStages) & 1u);
                }
                return;
            }
            const int idx = k * kPoThreads + tid;
            const bool valid = idx < I.count;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
            if (valid) {
                x = s_rec[s][2 * tid];
                y = s_rec[s][2 * tid + 1];
            }
            __syncthreads();  // every thread has read stage s: it can be refilled
            if (tid == 0) produce();
            if (!valid) continue;
            float cf[kPol];
#pragma unroll
            for (int q = 0; q < kPol; ++q) {
                const int sel = a.pol_sel[q];
                const float vec = sel == 0 ? x.x : (sel == 1 ? x.y : (sel == 2 ? x.z : x.w));
                float v = 0.f;
                if (q < a.n_pol) v = a.scalar ? (sel < 2 ? y.x : 0.f) : vec;
                cf[q] = v;
            }
#pragma unroll
            for (int fj = 0; fj < kF; ++fj) {
                if (fj >= I.nf) break;
                const float4 fq = a.freq[I.f0 + fj];
                const double kd = kPhase != 2 ? 0.0 : a.kfreq[I.f0 + fj];
                float c, sn;
                phase_cs<kPhase>(fq, kd, y.y, y.z, c, sn);
#pragma unroll
                for (int q = 0; q < kPol; ++q) {
                    acc[(fj * kPol + q) * 2] = fmaf(cf[q], c, acc[(fj * kPol + q) * 2]);
                    acc[(fj * kPol + q) * 2 + 1] = fmaf(-cf[q], sn, acc[(fj * kPol + q) * 2 + 1]);
                }
            }
        }
        const float sum = warp_sums<8>(acc);
        if ((lane & 3) == 0) s_red[w][warp_sum_index<8>(lane)] = sum;
        __syncthreads();
        if (tid < 8) {
            const int fj = tid / (2 * kPol), r = tid - fj * (2 * kPol);
            if (fj < I.nf && r < 2 * a.n_pol) {
                float v = 0.f;
#pragma unroll
                for (int k = 0; k < kWarps; ++k) v += s_red[k][tid];
                a.partial[I.part + (size_t)fj * (2 * a.n_pol) + r] = (double)v;
            }
        }
        __syncthreads();
    }
}

// Work list, stage 1 (one block): 64-bit exclusive scans over the aspects of
// their item counts and partial sizes, in tiles of the block size.
__global__ void k_po_items_scan(const unsigned* recoff, PoAngle* angles, int na, int n_pol, int item_records,
                                int* n_items, long long* valid)
{
    __shared__ long long s_ni[32], s_np[32];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
    long long base_i = 0, base_p = 0;
    for (int t0 = 0; t0 < na; t0 += blockDim.x) {
        const int a = t0 + tid;
        long long ni = 0, np = 0;
        if (a < na) {
            const unsigned rc = recoff[a + 1] - recoff[a];
            ni = (rc + item_records - 1) / item_records;
            np = ni * (long long)angles[a].nf * 2 * n_pol;
        }
        // inclusive warp scans, then across warps
        long long xi = ni, xp = np;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long yi = __shfl_up_sync(0xffffffffu, xi, o), yp = __shfl_up_sync(0xffffffffu, xp, o);
            if (lane >= o) {
                xi += yi;
                xp += yp;
            }
        }
        if (lane == 31) {
            s_ni[w] = xi;
            s_np[w] = xp;
        }
        __syncthreads();
        long long wi = 0, wp = 0, ti = 0, tp = 0;
        for (int k = 0; k < nw; ++k) {
            if (k < w) {
                wi += s_ni[k];
                wp += s_np[k];
            }
            ti += s_ni[k];
            tp += s_np[k];
        }
        if (a < na) {
            PoAngle& A = angles[a];
            A.item_begin = (int)(base_i + wi + xi - ni);
            A.item_end = (int)(base_i + wi + xi);
            A.part = base_p + wp + xp - np;
        }
        base_i += ti;
        base_p += tp;
        __syncthreads();
    }
    if (tid == 0) {
        *n_items = (int)base_i;
        if (valid) *valid = recoff[na];
    }
}

// Work list, stage 2: the warps of row blockIdx.y's grid share the aspect's
// items. recoff: the record offsets of the aspects (32-bit within a chunk, or
// 64-bit over a whole trace).
template <typename Off>
__global__ void k_po_items_fill(const Off* recoff, const PoAngle* angles, int n_pol, int item_records, PoItem* items)
{
    const int a = blockIdx.x;
    const PoAngle A = angles[a];
    const long long r0 = (long long)recoff[a], rc = (long long)recoff[a + 1] - r0;
    for (int r = blockIdx.y * blockDim.x + threadIdx.x; r < A.item_end - A.item_begin; r += gridDim.y * blockDim.x) {
        PoItem it;
        it.angle = a;
        it.count = (int)min((long long)item_records, rc - (long long)r * item_records);
        it.first = r0 + (long long)r * item_records;
        it.f0 = A.f0;
        it.nf = A.nf;
        it.part = A.part + (long long)r * A.nf * 2 * n_pol;
        items[A.item_begin + r] = it;
    }
}

// Blocks of 8 outputs (frequency, polarisation; re and im each) x kSlices item
// slices per aspect: slice s adds the partials of items s, s + kSlices, ... in
// item order, then the slices are added in a fixed tree, so a sum's order
// depends on its aspect's item count alone. One thread adding an aspect's items
// one after another was a chain of up to thousands of dependent FP64 additions
// (3,300 items per aspect of the aircraft at 10 GHz, 37 aspects: 967 us, now 68).
constexpr int kSlices = 32, kOutB = 8;
__global__ void __launch_bounds__(kSlices* kOutB) k_po_final(const double* partial, const PoItem* items,
                                                            const PoAngle* angles, const double* kfreq, int n_pol,
                                                            double* E, double* rcs)
{
    __shared__ double2 s_sum[kSlices][kOutB];
    const PoAngle A = angles[blockIdx.x];
    const int n_out = A.nf * n_pol, oi = threadIdx.x % kOutB, slice = threadIdx.x / kOutB;
    const int n = A.item_end - A.item_begin;
    // an aspect's items are consecutive and so are their partials, nf x n_pol x (re, im) each
    const double2* p0 = n > 0 ? reinterpret_cast<const double2*>(partial + items[A.item_begin].part) : nullptr;
    for (int o0 = blockIdx.y * kOutB; o0 < n_out; o0 += gridDim.y * kOutB) {
        const int o = o0 + oi;
        double sr = 0.0, si = 0.0;
        if (o < n_out) {
            // the loads of 8 items are issued before their additions
            for (int it = slice; it < n; it += 8 * kSlices) {
                double2 v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int k = it + u * kSlices;
                    v[u] = k < n ? __ldg(p0 + (size_t)k * n_out + o) : make_double2(0.0, 0.0);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (it + u * kSlices < n) {
                        sr += v[u].x;
                        si += v[u].y;
                    }
            }
        }
        s_sum[slice][oi] = make_double2(sr, si);
#pragma unroll
        for (int h = kSlices / 2; h > 0; h >>= 1) {
            __syncthreads();
            if (slice < h) {
                sr += s_sum[slice + h][oi].x;
                si += s_sum[slice + h][oi].y;
                s_sum[slice][oi] = make_double2(sr, si);
            }
        }
        if (slice == 0 && o < n_out) {
            // E = (-j k / 4 pi) (sr + j si)
            const int q = o / n_pol, p = o - q * n_pol;
            const double pre = kfreq[A.f0 + q] / (4.0 * 3.14159265358979323846);
            const double er = pre * si, ei = -pre * sr;
            const long long i = (A.out_row + q) * n_pol + p;
            if (E) {
                E[2 * i] = er;
                E[2 * i + 1] = ei;
            }
            if (rcs) rcs[i] = 10.0 * log10(4.0 * 3.14159265358979323846 * (er * er + ei * ei));
        }
        __syncthreads();  // the next outputs' sums reuse the shared rows
    }
}

}  // namespace

namespace {

template <int kPhase>
cudaError_t launch_po_mode(const PoArgs& a, cudaStream_t st, int n_blocks)
{
    const int grid = n_blocks > 0 ? n_blocks : a.n_items;
    if (grid <= 0) return cudaSuccess;
    const int per = (a.item_records > 0 ? a.item_records : kPoItemRecords) / kPoThreads;
    const bool two = a.n_pol <= 2;
    if (a.err && n_blocks == 0 && a.n_freq <= (two ? 2 : 1) && (per == 2 || per == 4 || per == 8)) {
        // one block reduction per item: the staged kernel, one persistent wave
        int dev = 0, sms = 0, occ = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = two ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_po_bulk<2, kPhase>, kPoThreads, 0)
                    : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_po_bulk<4, kPhase>, kPoThreads, 0);
        if (e != cudaSuccess) return e;
        const int g = (int)std::min<long long>(a.n_items, (long long)sms * std::max(occ, 1));
        if (two) k_po_bulk<2, kPhase><<<g, kPoThreads, 0, st>>>(a);
        else k_po_bulk<4, kPhase><<<g, kPoThreads, 0, st>>>(a);
        return cudaGetLastError();
    }
    if (per == 2) {
        if (two) k_po<2, 2, kPhase><<<grid, kPoThreads, 0, st>>>(a);
        else k_po<2, 4, kPhase><<<grid, kPoThreads, 0, st>>>(a);
    } else if (per == 8) {
        if (two) k_po<8, 2, kPhase><<<grid, kPoThreads, 0, st>>>(a);
        else k_po<8, 4, kPhase><<<grid, kPoThreads, 0, st>>>(a);
    } else if (per == 4) {
        if (two) k_po<4, 2, kPhase><<<grid, kPoThreads, 0, st>>>(a);
        else k_po<4, 4, kPhase><<<grid, kPoThreads, 0, st>>>(a);
    } else {
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_po(const PoArgs& a, cudaStream_t st, int n_blocks)
{
    if (a.phase_mode == 0) return launch_po_mode<0>(a, st, n_blocks);
    return a.phase_mode == 1 ? launch_po_mode<1>(a, st, n_blocks) : launch_po_mode<2>(a, st, n_blocks);
}

namespace {
// a block row per aspect, more of them where few aspects hold many items
dim3 fill_grid(int n_angles) { return dim3((unsigned)n_angles, (unsigned)std::max(1, std::min(16, 1024 / n_angles))); }
}  // namespace

cudaError_t launch_po_items(const unsigned* recoff, PoAngle* angles, int n_angles, int n_pol, int item_records,
                            PoItem* items, int* n_items, long long* valid, cudaStream_t st)
{
    if (n_angles <= 0 || item_records <= 0) return cudaErrorInvalidValue;
    k_po_items_scan<<<1, 1024, 0, st>>>(recoff, angles, n_angles, n_pol, item_records, n_items, valid);
    k_po_items_fill<unsigned><<<fill_grid(n_angles), 128, 0, st>>>(recoff, angles, n_pol, item_records, items);
    return cudaGetLastError();
}

cudaError_t launch_po_items_fill(const long long* recoff, const PoAngle* angles, int n_angles, int n_pol,
                                 int item_records, PoItem* items, cudaStream_t st)
{
    if (n_angles <= 0 || item_records <= 0) return cudaErrorInvalidValue;
    k_po_items_fill<long long><<<fill_grid(n_angles), 128, 0, st>>>(recoff, angles, n_pol, item_records, items);
    return cudaGetLastError();
}

cudaError_t launch_po_final(const double* partial, const PoItem* items, const PoAngle* angles, int n_angles,
                            int max_freq, const double* kfreq, int n_pol, double* E, double* rcs, cudaStream_t st)
{
    if (n_angles <= 0) return cudaSuccess;
    const long long blocks = ((long long)max_freq * n_pol + kOutB - 1) / kOutB;
    k_po_final<<<dim3((unsigned)n_angles, (unsigned)std::max(1ll, std::min(blocks, 1024ll))), kSlices * kOutB, 0, st>>>(
        partial, items, angles, kfreq, n_pol, E, rcs);
    return cudaGetLastError();
}

}  // namespace sbr
