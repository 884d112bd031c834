// sbr_trace.cu -- multi-bounce ray transport (Algorithm 2 of the paper) as a
// wavefront of persistent kernels:
//   pass 0        primary rays generated from their index on the aperture grid
//                 (Eq. L1-L3), closest hit, one 32-bit hit mask per 32 rays
//   scan          exclusive popcount prefix of the masks = dense record slots
//   pass b >= 1   the live rays of the previous pass, compacted into a queue,
//                 take their next closest-hit query (skipping the triangle just
//                 left); rays that miss or reach B_max write their record
// Each hit applies the specular reflection d - 2 (d.n) n, the PEC field update
// E' = 2 (n.E) n - E and the origin offset eps along the normal (Sec. 4), and
// stores the ray-tube coefficients the PO sum needs if this hit is the last one.
//
// Warps fetch 32 rays at a time from a global counter, so the grid stays full
// while rays finish at different depths; the traversal keeps a per-thread
// stack of node references, visits the nearer child first and tests the
// triangles of a leaf in FP32 Moller-Trumbore form.
#include <float.h>
#include <limits.h>
#include <stddef.h>

#include <algorithm>

#include "sbr_internal.h"

namespace sbr {

namespace {

constexpr int kTraceThreads = 256;
// conservative slab test: exit distance scaled by 1 + 2*gamma_3 (robust traversal)
constexpr float kBoxGrow = 1.0000008f;
constexpr unsigned kFull = 0xffffffffu;

// trace flag bits (mirror of SBR_TRACE_* in sbr.h)
constexpr int kFlagLiteral = 1;
constexpr int kFlagEscape = 2;

// The closest candidate of a query. During the traversal its exact distance is
// known to lie in [lo, t]; its stored distance t32 (key) is computed only when
// another candidate's interval overlaps, and at the end (key_closest), which
// sets t = t32.
struct Hit {
    float t;    // upper bound of the closest candidate's exact distance (box culling); t32 after key_closest
    float lo;   // lower bound of its exact distance
    float key;  // its t32 once computed, else -1
    int k;      // its position in the reordered triangles (-1: none)
    int orig;   // its original index
};

__device__ __forceinline__ float safe_rcp(float x)
{
    const float tiny = 1e-20f;
    return __frcp_rn(fabsf(x) > tiny ? x : copysignf(tiny, x));
}

// Two fused multiply-adds in one packed FP32 instruction: (a.x b.x + c.x,
// a.y b.y + c.y), each lane rounded once as fmaf rounds it.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pc, pr;\n\t"
        "mov.b64 pa, {%2, %3};\n\tmov.b64 pb, {%4, %5};\n\tmov.b64 pc, {%6, %7};\n\t"
        "fma.rn.f32x2 pr, pa, pb, pc;\n\tmov.b64 {%0, %1}, pr;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}

// ---------------------------------------------------------------- two-float helpers
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e)
{
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ void tf_add(float& hi, float& lo, float x)
{
    float s, e;
    two_sum(hi, x, s, e);
    e = __fadd_rn(e, lo);
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}
__device__ __forceinline__ void tf_add_tf(float& hi, float& lo, float xh, float xl)
{
    float s, e;
    two_sum(hi, xh, s, e);
    e = __fadd_rn(e, __fadd_rn(lo, xl));
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}
// a . b as an unevaluated two-float sum (exact products, compensated sum)
__device__ __forceinline__ void tf_dot(const float* a, float3 b, float& hi, float& lo)
{
    float p0 = __fmul_rn(a[0], b.x), e0 = __fmaf_rn(a[0], b.x, -p0);
    float p1 = __fmul_rn(a[1], b.y), e1 = __fmaf_rn(a[1], b.y, -p1);
    float p2 = __fmul_rn(a[2], b.z), e2 = __fmaf_rn(a[2], b.z, -p2);
    float s, e, s2, f;
    two_sum(p0, p1, s, e);
    two_sum(s, p2, s2, f);
    float lo_ = __fadd_rn(__fadd_rn(e, f), __fadd_rn(__fadd_rn(e0, e1), e2));
    hi = __fadd_rn(s2, lo_);
    lo = __fsub_rn(lo_, __fsub_rn(hi, s2));
}

// ---------------------------------------------------------------- FP32 cross and dot products
// cross(a, b) = (fma(a.y, b.z, -(a.z b.y)), ...) and dot(a, b) = fma(a.x, b.x, fma(a.y, b.y, a.z b.z)):
// each fma one rounding, every other operation one IEEE round-to-nearest operation
__device__ __forceinline__ float3 cross_s(float3 a, float3 b)
{
    return make_float3(__fmaf_rn(a.y, b.z, -__fmul_rn(a.z, b.y)), __fmaf_rn(a.z, b.x, -__fmul_rn(a.x, b.z)),
                       __fmaf_rn(a.x, b.y, -__fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float dot_s(float3 a, float3 b)
{
    return __fmaf_rn(a.x, b.x, __fmaf_rn(a.y, b.y, __fmul_rn(a.z, b.z)));
}

// ---------------------------------------------------------------- exact triangle test
// Which triangle a ray hits is decided exactly: the ray o + t d (its FP32
// values) against the closed triangle of the FP32 vertices, t > 0. With the
// exact E1 = v1 - v0, E2 = v2 - v0 and S = o - v0,
//   det = E1.(d x E2), U = S.(d x E2), V = d.(S x E1), T = E2.(S x E1),
// the ray hits when det != 0 and, taken with the sign of det, U >= 0, V >= 0,
// W = det - U - V >= 0 and T > 0 (Moller-Trumbore form, inclusive edges).
// They are evaluated in FP32 on the record's rounded edges; a forward error
// bound (gamma_n analysis of the rounded inputs, cross and dot products,
// folded into the per-triangle constants bUV, bD and the ray's largest
// |S| component) says when every sign is certain. Tests left open are taken
// again with the origin moved along the ray next to the triangle (U and V do
// not change, and their bounds shrink to the triangle's own size), and what is
// still open in FP64 from the exact vertices.
constexpr float kU = 0x1p-24f;  // FP32 unit roundoff

// 0: certain miss; 1: certain hit, tc ~ T / det with |tc - t| <= et;
// 2: the sign of U, V or W is open (det and T certain); 3: det or T open.
// U0, V0, T0, det: the FP32 values; bU, bV, bD, bT: bounds of their errors.
__device__ __forceinline__ int filter_core(float U0, float V0, float T0, float det, float bU, float bV, float bD,
                                           float bT, float& tc, float& et)
{
    const bool neg = det < 0.f;
    const float U = neg ? -U0 : U0, V = neg ? -V0 : V0, T = neg ? -T0 : T0;
    const float ad = fabsf(det);
    if (!(ad > bD)) return 3;  // det's sign open
    const float W = __fsub_rn(__fsub_rn(ad, U), V);
    const float bW = __fmaf_rn(0x1.1p-23f, __fadd_rn(__fadd_rn(ad, fabsf(U)), fabsf(V)), __fadd_rn(__fadd_rn(bU, bV), bD));
    if (U < -bU || V < -bV || W < -bW || T < -bT) return 0;
    if (!(T > bT)) return 3;
    if (!(U > bU && V > bV && W > bW)) return 2;
    tc = __fdividef(T, ad);
    et = __fmaf_rn(5.f * kU, tc, 1.01f * __fdividef(__fmaf_rn(tc, bD, bT), __fsub_rn(ad, bD)));
    return 1;
}

__device__ __forceinline__ float3 abs3(float3 a) { return make_float3(fabsf(a.x), fabsf(a.y), fabsf(a.z)); }
// |a| x |b| with absolute values: (|a.y||b.z| + |a.z||b.y|, ...), non-negative
__device__ __forceinline__ float3 cross_abs(float3 a, float3 b)
{
    a = abs3(a);
    b = abs3(b);
    return make_float3(__fmaf_rn(a.y, b.z, __fmul_rn(a.z, b.y)), __fmaf_rn(a.z, b.x, __fmul_rn(a.x, b.z)),
                       __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}

// Forward error bounds (Higham's gamma_n analysis: each rounded input, cross
// and dot product adds at most u of the absolute values it combines):
//   |U - U*| <= 8.1 u |S|.(|d| x |e2|),  |V - V*| <= 8.1 u |d|.(|S| x |e1|),
//   |det - det*| <= 8.1 u |e1|.(|d| x |e2|),  |T - T*| <= 9.1 u |e2|.(|S| x |e1|),
// with the 0.1 u covering the rounding of the bounds themselves. The record's
// bUV and bD bound them through norms (24 u L |S|_max, 14 u L^2, and
// 28 u L^2 |S|_max for T): three operations instead of some twenty, tried first.
__device__ __forceinline__ int tri_filter(float4 A, float4 B, float4 C, float3 o, float3 d, float& tc, float& et)
{
    const float3 e1 = make_float3(B.x, B.y, B.z), e2 = make_float3(C.x, C.y, C.z);
    const float3 p = cross_s(d, e2);
    const float det = dot_s(e1, p);
    const float3 s = make_float3(__fsub_rn(o.x, A.x), __fsub_rn(o.y, A.y), __fsub_rn(o.z, A.z));
    const float3 qv = cross_s(s, e1);
    const float U0 = dot_s(s, p), V0 = dot_s(d, qv), T0 = dot_s(e2, qv);
    const float smax = fmaxf(fmaxf(fabsf(s.x), fabsf(s.y)), fabsf(s.z));
    const float bUV = __fmul_rn(smax, B.w);
    if (!(B.w > 0.f)) return 0;
    return filter_core(U0, V0, T0, det, bUV, bUV, C.w, __fmul_rn(2.f * smax, C.w), tc, et);
}

// the per-component bounds of a test the norm bounds left open
__device__ __forceinline__ int tri_filter_tight(float4 A, float4 B, float4 C, float3 o, float3 d, float& tc, float& et)
{
    const float3 e1 = make_float3(B.x, B.y, B.z), e2 = make_float3(C.x, C.y, C.z);
    const float3 p = cross_s(d, e2);
    const float det = dot_s(e1, p);
    const float3 s = make_float3(__fsub_rn(o.x, A.x), __fsub_rn(o.y, A.y), __fsub_rn(o.z, A.z));
    const float3 qv = cross_s(s, e1);
    const float U0 = dot_s(s, p), V0 = dot_s(d, qv), T0 = dot_s(e2, qv);
    const float3 pa = cross_abs(d, e2), qa = cross_abs(s, e1);
    const float3 as = abs3(s), ad3 = abs3(d), a1 = abs3(e1), a2 = abs3(e2);
    return filter_core(U0, V0, T0, det, 0x1.03p-21f * dot_s(as, pa), 0x1.03p-21f * dot_s(ad3, qa),
                       0x1.03p-21f * dot_s(a1, pa), 0x1.23p-21f * dot_s(a2, qa), tc, et);
}

// o + lam d - v of one component as sc, with |sc - exact| <= 3 u sa, sa = |sc| + |z|
// (lam d and o + lam d as exact two-float sums; only the last two additions round)
__device__ __forceinline__ void shift1(float o, float d, float v, float lam, float& sc, float& sa)
{
    const float P = __fmul_rn(lam, d), Pe = __fmaf_rn(lam, d, -P);
    float X, Xe;
    two_sum(o, P, X, Xe);
    const float Y = __fsub_rn(X, v), Z = __fadd_rn(Xe, Pe);
    sc = __fadd_rn(Y, Z);
    sa = __fadd_rn(fabsf(sc), fabsf(Z));
}

// The decision left open by tri_filter (code 2 or 3): bit 0 of the result is
// set on a hit (then tc = T / det in FP32), bit 1 when FP64 decided.
__device__ __noinline__ int tri_refine(const float4* __restrict__ rec, const float4* __restrict__ v12, int k, float3 o,
                                        float3 d, int code, float& tc)
{
    const float4 A = __ldg(rec + 3 * (size_t)k), B = __ldg(rec + 3 * (size_t)k + 1), C = __ldg(rec + 3 * (size_t)k + 2);
    if (code >= 4) {  // from the norm bounds: try the per-component ones first
        float et;
        code = tri_filter_tight(A, B, C, o, d, tc, et);
        if (code < 2) return code;
    }
    const float3 e1 = make_float3(B.x, B.y, B.z), e2 = make_float3(C.x, C.y, C.z);
    const float3 p = cross_s(d, e2);
    const float det = dot_s(e1, p);
    const float3 s0 = make_float3(__fsub_rn(o.x, A.x), __fsub_rn(o.y, A.y), __fsub_rn(o.z, A.z));
    const float T0 = dot_s(e2, cross_s(s0, e1));
    tc = __fdiv_rn(T0, det);
    const float lam = __fdividef(T0, det);  // any finite value keeps U and V; near t it makes S small
    if (code == 2 && isfinite(lam)) {
        float3 sc, sa;
        shift1(o.x, d.x, A.x, lam, sc.x, sa.x);
        shift1(o.y, d.y, A.y, lam, sc.y, sa.y);
        shift1(o.z, d.z, A.z, lam, sc.z, sa.z);
        const float3 q1 = cross_s(sc, e1);
        const float U0 = dot_s(sc, p), V0 = dot_s(d, q1);
        // |d| x |e2| and sa x |e1|, then bounds of det (8 u), U and V (9.5 u each)
        const float3 ad3 = make_float3(fabsf(d.x), fabsf(d.y), fabsf(d.z));
        const float3 a1 = make_float3(fabsf(e1.x), fabsf(e1.y), fabsf(e1.z));
        const float3 a2 = make_float3(fabsf(e2.x), fabsf(e2.y), fabsf(e2.z));
        const float3 pa = make_float3(__fmaf_rn(ad3.y, a2.z, __fmul_rn(ad3.z, a2.y)),
                                      __fmaf_rn(ad3.z, a2.x, __fmul_rn(ad3.x, a2.z)),
                                      __fmaf_rn(ad3.x, a2.y, __fmul_rn(ad3.y, a2.x)));
        const float3 qa = make_float3(__fmaf_rn(sa.y, a1.z, __fmul_rn(sa.z, a1.y)),
                                      __fmaf_rn(sa.z, a1.x, __fmul_rn(sa.x, a1.z)),
                                      __fmaf_rn(sa.x, a1.y, __fmul_rn(sa.y, a1.x)));
        const float bD = 0x1.02p-21f * dot_s(a1, pa);
        const float bU = 0x1.3p-21f * dot_s(sa, pa);
        const float bV = 0x1.3p-21f * dot_s(ad3, qa);
        const float ad = fabsf(det);
        if (ad > bD) {
            const bool neg = det < 0.f;
            const float U = neg ? -U0 : U0, V = neg ? -V0 : V0;
            const float W = __fsub_rn(__fsub_rn(ad, U), V);
            const float bW = __fmaf_rn(0x1.1p-23f, __fadd_rn(__fadd_rn(ad, fabsf(U)), fabsf(V)), bD + bU + bV);
            if (U < -bU || V < -bV || W < -bW) return 0;
            if (U > bU && V > bV && W > bW) return 1;
        }
    }
    // FP64 from the exact vertices: differences of FP32 values are exact, the
    // products and sums round at 2^-53, far inside the 1e-6 edge band
    const float4 P1 = __ldg(v12 + 2 * (size_t)k), P2 = __ldg(v12 + 2 * (size_t)k + 1);
    const double x0 = A.x, y0 = A.y, z0 = A.z;
    const double E1x = (double)P1.x - x0, E1y = (double)P1.y - y0, E1z = (double)P1.z - z0;
    const double E2x = (double)P2.x - x0, E2y = (double)P2.y - y0, E2z = (double)P2.z - z0;
    const double Sx = (double)o.x - x0, Sy = (double)o.y - y0, Sz = (double)o.z - z0;
    const double Dx = d.x, Dy = d.y, Dz = d.z;
    const double Px = Dy * E2z - Dz * E2y, Py = Dz * E2x - Dx * E2z, Pz = Dx * E2y - Dy * E2x;
    double dt = E1x * Px + E1y * Py + E1z * Pz;
    if (dt == 0.0) return 2;
    const double Qx = Sy * E1z - Sz * E1y, Qy = Sz * E1x - Sx * E1z, Qz = Sx * E1y - Sy * E1x;
    double U = Sx * Px + Sy * Py + Sz * Pz, V = Dx * Qx + Dy * Qy + Dz * Qz, T = E2x * Qx + E2y * Qy + E2z * Qz;
    tc = (float)(T / dt);
    if (dt < 0.0) {
        dt = -dt;
        U = -U;
        V = -V;
        T = -T;
    }
    return (U >= 0.0 && V >= 0.0 && (dt - U) - V >= 0.0 && T > 0.0) ? 3 : 2;
}

// a . b as an unevaluated two-float sum hi + lo (exact products, compensated sum)
__device__ __forceinline__ void tf_dot3(float3 a, float3 b, float& hi, float& lo)
{
    const float v[3] = {a.x, a.y, a.z};
    tf_dot(v, b, hi, lo);
}

// Hit distance stored with a hit: t32 = fl32(((v0 - o) . n) / (d . n)), the
// distance along the ray to the plane of the FP32 unit normal n through v0,
// rounded once. d.n as a two-float sum (exact products, compensated sum) and
// its reciprocal are taken once per (direction, triangle) -- once per (aspect,
// triangle) for the parallel primary rays; per origin o, v0 - o exactly as a
// two-float vector (TwoSum), the numerator (v0 - o).n as a two-float sum (its
// error relative to |v0 - o|, so short hops keep their precision), a quotient
// within a few units of the last place, its remainder and one correction.
struct PlaneKey {
    float3 n;
    float dh, dl, rd;
};

__device__ __forceinline__ PlaneKey plane_key(const float4* __restrict__ nrm, int k, float3 d)
{
    PlaneKey K;
    const float4 N = __ldg(nrm + k);
    K.n = make_float3(N.x, N.y, N.z);
    tf_dot3(d, K.n, K.dh, K.dl);
    K.rd = __frcp_rn(K.dh);
    return K;
}

// t32 for origin o and triangle vertex v0 (tfb when d.n is exactly 0)
__device__ __forceinline__ float plane_key_t(const PlaneKey& K, float3 v0, float3 o, float tfb)
{
    if (K.dh == 0.f) return tfb;
    float3 a, b;
    two_sum(v0.x, -o.x, a.x, b.x);
    two_sum(v0.y, -o.y, a.y, b.y);
    two_sum(v0.z, -o.z, a.z, b.z);
    float nh, nl;
    tf_dot3(a, K.n, nh, nl);
    nl = __fmaf_rn(b.x, K.n.x, __fmaf_rn(b.y, K.n.y, __fmaf_rn(b.z, K.n.z, nl)));
    const float q = __fmul_rn(nh, K.rd);
    const float r = __fadd_rn(__fmaf_rn(-q, K.dh, nh), __fmaf_rn(-q, K.dl, nl));
    return __fmaf_rn(r, K.rd, q);
}

// The triangle data a query reads (records, normals, exact vertices, counters)
// are those of the kernel's TraceArgs, read from its parameter space where
// needed rather than held in registers through the traversal.
using TriRefs = TraceArgs;

__device__ __forceinline__ const TraceArgs& tri_refs(const TraceArgs& a) { return a; }

// counting runs: one test left open by the filter, decided in FP64 or not
__device__ __forceinline__ void count_open(unsigned long long* stats, int r)
{
    atomicAdd(stats + kStatOpen, 1ull);
    if (r & 2) atomicAdd(stats + kStatFp64, 1ull);
}

// t32 of reordered triangle k and its error bound: |t32 - exact t| <= u t32
// (rounding) + u L / |d.n| (plane of n32 against the triangle's own), u L <= bUV / 24
__device__ __noinline__ float key_of(const TriRefs& tr, int k, float3 o, float3 d, float tfb, float& slack)
{
    const float4 A = __ldg(tr.tris + 3 * (size_t)k), B = __ldg(tr.tris + 3 * (size_t)k + 1);
    const PlaneKey K = plane_key(tr.tri_nrm, k, d);
    const float t = plane_key_t(K, make_float3(A.x, A.y, A.z), o, tfb);
    slack = __fmaf_rn(2.f * kU, fabsf(t), __fdividef(0.08f * B.w, fabsf(K.dh)));
    return t;
}

// Two candidates whose distance intervals overlap: their stored distances are
// computed and compared (rare; kept out of the traversal loop's registers).
__device__ __noinline__ void resolve_overlap(const TriRefs& tr, int k, int orig, float tc, float3 o, float3 d, Hit& h)
{
    float sl;
    if (h.key < 0.f) {
        h.key = key_of(tr, h.k, o, d, h.t, sl);
        h.t = __fadd_rn(h.key, sl);
        h.lo = __fsub_rn(h.key, sl);
    }
    const float t = key_of(tr, k, o, d, tc, sl);
    if (t < h.key || (t == h.key && orig < h.orig)) {
        h.key = t;
        h.t = __fadd_rn(t, sl);
        h.lo = __fsub_rn(t, sl);
        h.k = k;
        h.orig = orig;
    }
}

// The closest hit is the smallest (t32, original triangle index). A certain
// hit whose distance interval lies beyond the closest candidate's is dropped,
// one whose interval lies before it replaces it, and only when the two overlap
// are their stored distances computed and compared.
__device__ __forceinline__ void consider_hit(const TriRefs& tr, int k, int orig, float tc, float et, float3 o,
                                             float3 d, Hit& h)
{
    const float lo = __fsub_rn(tc, et), hi = __fadd_rn(tc, et);
    if (lo > h.t) return;
    if (h.k < 0 || hi < h.lo) {
        h.t = hi;
        h.lo = lo;
        h.key = -1.f;
        h.k = k;
        h.orig = orig;
        return;
    }
    resolve_overlap(tr, k, orig, tc, o, d, h);
}

// after the traversal: the closest hit's t32 in h.t
__device__ __forceinline__ void key_closest(const TriRefs& tr, float3 o, float3 d, Hit& h)
{
    if (h.k < 0) return;
    if (h.key < 0.f) {
        float sl;
        h.key = key_of(tr, h.k, o, d, 0.5f * (h.t + h.lo), sl);
    }
    h.t = h.key;
}

// The triangles of leaf `ref`
template <bool kCount>
__device__ __forceinline__ void leaf_test(const TriRefs& tr, int ref, float3 o, float3 d, int skip, Hit& h,
                                          unsigned& ntri)
{
    const int first = leaf_first(ref), cnt = leaf_count(ref);
    for (int q = 0; q < cnt; ++q) {
        const int k = first + q;
        if (kCount) ++ntri;
        if (k == skip) continue;
        const float4* tp = tr.tris + 3 * (size_t)k;
        const float4 A = __ldg(tp), B = __ldg(tp + 1), C = __ldg(tp + 2);
        float tc = 0.f, et = FLT_MAX;
        const int f = tri_filter(A, B, C, o, d, tc, et);
        if (f == 0) continue;
        if (f >= 2) {
            const int r = tri_refine(tr.tris, tr.tri_v12, k, o, d, f + 2, tc);
            if (kCount) count_open(tr.stats, r);
            if (!(r & 1)) continue;
            et = FLT_MAX;
        }
        consider_hit(tr, k, __float_as_int(A.w), tc, et, o, d, h);
    }
}

template <bool kCount, int kStack>
__device__ __forceinline__ void closest_hit(const float4* __restrict__ nodes, const TriRefs& tris, float3 o,
                                            float3 d, int skip, int limit, Hit& h, unsigned& nvis, unsigned& ntri,
                                            bool& overflow)
{
    int stack[kStack];
    const float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    const float3 oi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    // the slab distances of a box coordinate pair (lo, hi) of one axis: one packed fma
    const float2 ix = make_float2(inv.x, inv.x), iy = make_float2(inv.y, inv.y), iz = make_float2(inv.z, inv.z);
    const float2 mx = make_float2(-oi.x, -oi.x), my = make_float2(-oi.y, -oi.y), mz = make_float2(-oi.z, -oi.z);
    h.t = FLT_MAX;
    h.k = -1;
    h.orig = INT_MAX;
    h.lo = FLT_MAX;
    h.key = -1.f;
    int sp = 0;
    int ref = 0;
    // a query visits every node and leaf at most once; the bound guards against
    // a malformed hierarchy (reported like a stack overflow)
    for (int it = 0;; ++it) {
        if (it >= limit) {
            overflow = true;
            break;
        }
        if (ref >= 0) {
            const float4* nd = nodes + 4 * (size_t)ref;
            const float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
            if (kCount) ++nvis;
            const float tmax = h.t;
            const float2 ax = fma2(make_float2(n0.x, n0.y), ix, mx), ay = fma2(make_float2(n0.z, n0.w), iy, my);
            const float2 az = fma2(make_float2(n2.x, n2.y), iz, mz), bx = fma2(make_float2(n1.x, n1.y), ix, mx);
            const float2 by = fma2(make_float2(n1.z, n1.w), iy, my), bz = fma2(make_float2(n2.z, n2.w), iz, mz);
            float an = fmaxf(fmaxf(fminf(ax.x, ax.y), fminf(ay.x, ay.y)), fmaxf(fminf(az.x, az.y), 0.f));
            float af = fminf(fminf(fmaxf(ax.x, ax.y), fmaxf(ay.x, ay.y)), fminf(fmaxf(az.x, az.y), tmax));
            float bn = fmaxf(fmaxf(fminf(bx.x, bx.y), fminf(by.x, by.y)), fmaxf(fminf(bz.x, bz.y), 0.f));
            float bf = fminf(fminf(fmaxf(bx.x, bx.y), fmaxf(by.x, by.y)), fminf(fmaxf(bz.x, bz.y), tmax));
            const int lref = __float_as_int(n3.x), rref = __float_as_int(n3.y);
            const bool hl = an <= af * kBoxGrow;
            const bool hr = (bn <= bf * kBoxGrow) && (rref != kEmptyRef);
            if (hl && hr) {
                const bool lnear = an <= bn;
                if (sp < kStack) stack[sp++] = lnear ? rref : lref;
                else overflow = true;
                ref = lnear ? lref : rref;
                continue;
            }
            if (hl) { ref = lref; continue; }
            if (hr) { ref = rref; continue; }
        } else {
            leaf_test<kCount>(tris, ref, o, d, skip, h, ntri);
        }
        if (sp == 0) break;
        ref = stack[--sp];
    }
}

// Binary traversal over the octant copies of the nodes: the ray's direction
// signs pick the copy whose near and far slabs are already chosen, so a child
// test is 6 FMA and 6 min/max instead of 6 FMA and 12 min/max. The FMA is
// monotone in the box coordinate, so every slab value, accepted box and visit
// order equals the min/max form of closest_hit.
template <bool kCount, int kStack>
__device__ __forceinline__ void closest_hit_oct(const float4* __restrict__ octant_nodes, long long n_nodes,
                                                const TriRefs& tris, float3 o, float3 d, int skip,
                                                int limit, Hit& h, unsigned& nvis, unsigned& ntri, bool& overflow)
{
    int stack[kStack];
    const float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    const float3 oi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    const int oct = (inv.x < 0.f ? 1 : 0) | (inv.y < 0.f ? 2 : 0) | (inv.z < 0.f ? 4 : 0);
    const float4* nodes = octant_nodes + 4 * (size_t)oct * (size_t)n_nodes;
    h.t = FLT_MAX;
    h.k = -1;
    h.orig = INT_MAX;
    h.lo = FLT_MAX;
    h.key = -1.f;
    int sp = 0;
    int ref = 0;
    for (int it = 0;; ++it) {
        if (it >= limit) {
            overflow = true;
            break;
        }
        if (ref >= 0) {
            const float4* nd = nodes + 4 * (size_t)ref;
            const float4 f0 = __ldg(nd), f1 = __ldg(nd + 1), f2 = __ldg(nd + 2), f3 = __ldg(nd + 3);
            if (kCount) ++nvis;
            const float tmax = h.t;
            const float an = fmaxf(fmaxf(fmaf(f0.x, inv.x, -oi.x), fmaf(f0.y, inv.y, -oi.y)),
                                   fmaxf(fmaf(f0.z, inv.z, -oi.z), 0.f));
            const float af = fminf(fminf(fmaf(f1.z, inv.x, -oi.x), fmaf(f1.w, inv.y, -oi.y)),
                                   fminf(fmaf(f2.x, inv.z, -oi.z), tmax));
            const float bn = fmaxf(fmaxf(fmaf(f0.w, inv.x, -oi.x), fmaf(f1.x, inv.y, -oi.y)),
                                   fmaxf(fmaf(f1.y, inv.z, -oi.z), 0.f));
            const float bf = fminf(fminf(fmaf(f2.y, inv.x, -oi.x), fmaf(f2.z, inv.y, -oi.y)),
                                   fminf(fmaf(f2.w, inv.z, -oi.z), tmax));
            const int lref = __float_as_int(f3.x), rref = __float_as_int(f3.y);
            const bool hl = an <= af * kBoxGrow;
            const bool hr = bn <= bf * kBoxGrow;
            if (hl && hr) {
                const bool lnear = an <= bn;
                if (sp < kStack) stack[sp++] = lnear ? rref : lref;
                else overflow = true;
                ref = lnear ? lref : rref;
                continue;
            }
            if (hl) { ref = lref; continue; }
            if (hr) { ref = rref; continue; }
        } else {
            leaf_test<kCount>(tris, ref, o, d, skip, h, ntri);
        }
        if (sp == 0) break;
        ref = stack[--sp];
    }
}

// 4-wide variant: the near and far slab of each axis are chosen once per ray
// from the sign of its direction, which gives the same FP32 values as the
// per-axis min / max of the binary test (the fused product is monotone in the
// box coordinate), so both trees accept exactly the same child boxes. Hit
// children are ordered near to far by a 5-exchange sorting network; the far
// ones go on the stack with their entry distance and are skipped when popped
// behind the closest hit so far.
__device__ __forceinline__ void cswap(float& ka, int& ra, float& kb, int& rb)
{
    const bool sw = kb < ka;
    const float k = sw ? kb : ka, k2 = sw ? ka : kb;
    const int r = sw ? rb : ra, r2 = sw ? ra : rb;
    ka = k;
    kb = k2;
    ra = r;
    rb = r2;
}

template <bool kCount, int kStack>
__device__ __forceinline__ void closest_hit4(const float4* __restrict__ nodes, const TriRefs& tris,
                                             float3 o, float3 d, int skip, int limit, Hit& h, unsigned& nvis,
                                             unsigned& ntri, bool& overflow)
{
    int stack[kStack];
    float stack_t[kStack];
    const float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    const float3 oi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    // float4 index of the near slab of each axis inside a node (lo: even, hi: odd)
    const int sx = inv.x >= 0.f ? 0 : 1, sy = inv.y >= 0.f ? 2 : 3, sz = inv.z >= 0.f ? 4 : 5;
    h.t = FLT_MAX;
    h.k = -1;
    h.orig = INT_MAX;
    h.lo = FLT_MAX;
    h.key = -1.f;
    int sp = 0;
    int ref = 0;
    for (int it = 0;; ++it) {
        if (it >= limit) {
            overflow = true;
            break;
        }
        if (ref >= 0) {
            const float4* nd = nodes + (size_t)kNode4Float4 * ref;
            const float4 nx = __ldg(nd + sx), fx = __ldg(nd + (sx ^ 1)), ny = __ldg(nd + sy), fy = __ldg(nd + (sy ^ 1));
            const float4 nz = __ldg(nd + sz), fz = __ldg(nd + (sz ^ 1));
            const float4 rr = __ldg(nd + 6);
            if (kCount) ++nvis;
            const float tmax = h.t;
#define SBR_SLAB(c, tn, tf)                                                                                  \
    const float tn = fmaxf(fmaxf(fmaf(nx.c, inv.x, -oi.x), fmaf(ny.c, inv.y, -oi.y)),                       \
                           fmaxf(fmaf(nz.c, inv.z, -oi.z), 0.f));                                           \
    const float tf = fminf(fminf(fmaf(fx.c, inv.x, -oi.x), fmaf(fy.c, inv.y, -oi.y)),                       \
                           fminf(fmaf(fz.c, inv.z, -oi.z), tmax));
            SBR_SLAB(x, tn0, tf0)
            SBR_SLAB(y, tn1, tf1)
            SBR_SLAB(z, tn2, tf2)
            SBR_SLAB(w, tn3, tf3)
#undef SBR_SLAB
            int r0 = __float_as_int(rr.x), r1 = __float_as_int(rr.y), r2 = __float_as_int(rr.z),
                r3 = __float_as_int(rr.w);
            float k0 = (tn0 <= tf0 * kBoxGrow && r0 != kEmptyRef) ? tn0 : FLT_MAX;
            float k1 = (tn1 <= tf1 * kBoxGrow && r1 != kEmptyRef) ? tn1 : FLT_MAX;
            float k2 = (tn2 <= tf2 * kBoxGrow && r2 != kEmptyRef) ? tn2 : FLT_MAX;
            float k3 = (tn3 <= tf3 * kBoxGrow && r3 != kEmptyRef) ? tn3 : FLT_MAX;
            cswap(k0, r0, k1, r1);
            cswap(k2, r2, k3, r3);
            cswap(k0, r0, k2, r2);
            cswap(k1, r1, k3, r3);
            cswap(k1, r1, k2, r2);
            if (k0 == FLT_MAX) {
                ref = kEmptyRef;  // no child hit: pop
            } else {
                // push hits far to near (the nearest is visited now)
                if (k3 != FLT_MAX) {
                    if (sp < kStack) {
                        stack[sp] = r3;
                        stack_t[sp++] = k3;
                    } else {
                        overflow = true;
                    }
                }
                if (k2 != FLT_MAX) {
                    if (sp < kStack) {
                        stack[sp] = r2;
                        stack_t[sp++] = k2;
                    } else {
                        overflow = true;
                    }
                }
                if (k1 != FLT_MAX) {
                    if (sp < kStack) {
                        stack[sp] = r1;
                        stack_t[sp++] = k1;
                    } else {
                        overflow = true;
                    }
                }
                ref = r0;
                continue;
            }
        } else {
            leaf_test<kCount>(tris, ref, o, d, skip, h, ntri);
        }
        // pop, skipping entries that start behind the closest hit so far
        ref = kEmptyRef;
        while (sp > 0) {
            --sp;
            if (stack_t[sp] <= h.t * kBoxGrow) {
                ref = stack[sp];
                break;
            }
        }
        if (ref == kEmptyRef) break;
    }
}

// Warp-cooperative (packet) traversal of the binary tree: the 32 lanes walk
// one path together, so every node and leaf fetch is a single broadcast and
// the loop never diverges. Each lane carries a "wants" flag per node (and one
// bit per stack entry): it wants a node when its own ray enters the node's box,
// and it tests boxes and leaf triangles only for nodes it wants, so its
// result and its visit counts are those of its own ray. The warp descends into
// a child when any lane wants it; when both children are wanted, the one that
// most lanes reach first goes first. Must be called by all 32 lanes together.
template <bool kCount, int kStack>
__device__ __forceinline__ void closest_hit_packet(const float4* __restrict__ nodes, const TriRefs& tris,
                                                   bool active, float3 o, float3 d, int skip, int limit, Hit& h,
                                                   unsigned& nvis, unsigned& ntri, bool& overflow)
{
    static_assert(kStack <= 64, "packet stack flags are one 64-bit word");
    int stack[kStack];
    unsigned long long wb = 0;  // lane wants stack entry k: bit k
    const float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    const float3 oi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    h.t = FLT_MAX;
    h.k = -1;
    h.orig = INT_MAX;
    h.lo = FLT_MAX;
    h.key = -1.f;
    int sp = 0;
    int ref = 0;
    bool want = active;
    bool ovf = false;
    for (int it = 0;; ++it) {
        if (it >= limit) {
            ovf = true;
            break;
        }
        if (ref >= 0) {
            const float4* nd = nodes + 4 * (size_t)ref;
            const float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
            if (kCount && want) ++nvis;
            const float tmax = h.t;
            float ax0 = fmaf(n0.x, inv.x, -oi.x), ax1 = fmaf(n0.y, inv.x, -oi.x);
            float ay0 = fmaf(n0.z, inv.y, -oi.y), ay1 = fmaf(n0.w, inv.y, -oi.y);
            float az0 = fmaf(n2.x, inv.z, -oi.z), az1 = fmaf(n2.y, inv.z, -oi.z);
            float bx0 = fmaf(n1.x, inv.x, -oi.x), bx1 = fmaf(n1.y, inv.x, -oi.x);
            float by0 = fmaf(n1.z, inv.y, -oi.y), by1 = fmaf(n1.w, inv.y, -oi.y);
            float bz0 = fmaf(n2.z, inv.z, -oi.z), bz1 = fmaf(n2.w, inv.z, -oi.z);
            float an = fmaxf(fmaxf(fminf(ax0, ax1), fminf(ay0, ay1)), fmaxf(fminf(az0, az1), 0.f));
            float af = fminf(fminf(fmaxf(ax0, ax1), fmaxf(ay0, ay1)), fminf(fmaxf(az0, az1), tmax));
            float bn = fmaxf(fmaxf(fminf(bx0, bx1), fminf(by0, by1)), fmaxf(fminf(bz0, bz1), 0.f));
            float bf = fminf(fminf(fmaxf(bx0, bx1), fmaxf(by0, by1)), fminf(fmaxf(bz0, bz1), tmax));
            const int lref = __float_as_int(n3.x), rref = __float_as_int(n3.y);
            const bool hl = want && an <= af * kBoxGrow;
            const bool hr = want && (bn <= bf * kBoxGrow) && (rref != kEmptyRef);
            const unsigned ml = __ballot_sync(kFull, hl), mr = __ballot_sync(kFull, hr);
            if (ml && mr) {
                const unsigned both = ml & mr, lfirst = __ballot_sync(kFull, hl && hr && an <= bn);
                const bool goleft = both ? 2 * __popc(lfirst) >= __popc(both) : __popc(ml) >= __popc(mr);
                const int fref = goleft ? rref : lref;
                const bool wfar = goleft ? hr : hl;
                if (sp < kStack) {
                    stack[sp] = fref;
                    wb = wfar ? (wb | (1ull << sp)) : (wb & ~(1ull << sp));
                    ++sp;
                } else {
                    ovf = true;
                }
                ref = goleft ? lref : rref;
                want = goleft ? hl : hr;
                continue;
            }
            if (ml) {
                ref = lref;
                want = hl;
                continue;
            }
            if (mr) {
                ref = rref;
                want = hr;
                continue;
            }
        } else if (want) {
            leaf_test<kCount>(tris, ref, o, d, skip, h, ntri);
        }
        if (sp == 0) break;
        --sp;
        ref = stack[sp];
        want = (wb >> sp) & 1ull;
    }
    if (active && ovf) overflow = true;
}

// ---------------------------------------------------------------- per-ray state in registers
struct Ray {
    float3 o, d, ev;
    float lacc_hi, lacc_lo, cos0;
    float c[5];
    float lc_hi, lc_lo, nfs;
    int angle, local, last, nb;
};

// The live-ray queues, the records and the raster keys are each written once
// and read once: their loads and stores are marked evict-first (__ldcs /
// __stcs) so that they do not push the tree and the triangles out of L1 and L2.
__device__ __forceinline__ void load_state(const RayState* __restrict__ q, unsigned i, Ray& r)
{
    const float4* p = reinterpret_cast<const float4*>(q + i);
    float4 a = __ldcs(p), b = __ldcs(p + 1), c = __ldcs(p + 2), e = __ldcs(p + 3), f = __ldcs(p + 4);
    int4 g = __ldcs(reinterpret_cast<const int4*>(p) + 5);
    r.o = make_float3(a.x, a.y, a.z);
    r.d = make_float3(a.w, b.x, b.y);
    r.ev = make_float3(b.z, b.w, c.x);
    r.lacc_hi = c.y;
    r.lacc_lo = c.z;
    r.cos0 = c.w;
    r.c[0] = e.x; r.c[1] = e.y; r.c[2] = e.z; r.c[3] = e.w;
    r.c[4] = f.x;
    r.lc_hi = f.y;
    r.lc_lo = f.z;
    r.nfs = f.w;
    r.angle = g.x; r.local = g.y; r.last = g.z; r.nb = g.w;
}

// The traversal needs only the origin, the direction and the triangle to
// skip: load those first and the rest of the state after the query, so the
// payload does not occupy registers during the traversal.
__device__ __forceinline__ void load_geom(const RayState* __restrict__ q, unsigned i, Ray& r)
{
    const float4* p = reinterpret_cast<const float4*>(q + i);
    const float4 a = __ldcs(p), b = __ldcs(p + 1);
    r.o = make_float3(a.x, a.y, a.z);
    r.d = make_float3(a.w, b.x, b.y);
    r.last = __ldcs(reinterpret_cast<const int4*>(p) + 5).z;
}

__device__ __forceinline__ void load_payload(const RayState* __restrict__ q, unsigned i, Ray& r)
{
    const float4* p = reinterpret_cast<const float4*>(q + i);
    const float4 b = __ldcs(p + 1), c = __ldcs(p + 2), e = __ldcs(p + 3), f = __ldcs(p + 4);
    const int4 g = __ldcs(reinterpret_cast<const int4*>(p) + 5);
    r.ev = make_float3(b.z, b.w, c.x);
    r.lacc_hi = c.y;
    r.lacc_lo = c.z;
    r.cos0 = c.w;
    r.c[0] = e.x; r.c[1] = e.y; r.c[2] = e.z; r.c[3] = e.w;
    r.c[4] = f.x;
    r.lc_hi = f.y;
    r.lc_lo = f.z;
    r.nfs = f.w;
    r.angle = g.x; r.local = g.y; r.nb = g.w;
}

__device__ __forceinline__ void store_state(RayState* __restrict__ q, unsigned i, const Ray& r)
{
    float4* p = reinterpret_cast<float4*>(q + i);
    __stcs(p + 0, make_float4(r.o.x, r.o.y, r.o.z, r.d.x));
    __stcs(p + 1, make_float4(r.d.y, r.d.z, r.ev.x, r.ev.y));
    __stcs(p + 2, make_float4(r.ev.z, r.lacc_hi, r.lacc_lo, r.cos0));
    __stcs(p + 3, make_float4(r.c[0], r.c[1], r.c[2], r.c[3]));
    __stcs(p + 4, make_float4(r.c[4], r.lc_hi, r.lc_lo, r.nfs));
    __stcs(reinterpret_cast<int4*>(p) + 5, make_int4(r.angle, r.local, r.last, r.nb));
}

__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }

// Update the ray at its closest hit: path, bounce count, candidate PO
// coefficients of this hit (used if it turns out to be the last), reflection,
// PEC field update and the new origin. The stored state is FP32, each value
// the rounding of its formula: x = fl32(o + t32 d), dn = fl32(d . n32),
// d' = fl32(d - 2 dn n32), o' = fl32(x + eps nf) (one fma each; dn from a
// compensated dot product).
__device__ __forceinline__ void apply_hit(const AngleDev& A, const float4* __restrict__ nrm, const Hit& h, int flags,
                                          Ray& r)
{
    const float3 x = make_float3(__fmaf_rn(h.t, r.d.x, r.o.x), __fmaf_rn(h.t, r.d.y, r.o.y),
                                 __fmaf_rn(h.t, r.d.z, r.o.z));
    tf_add(r.lacc_hi, r.lacc_lo, h.t);
    const int nb_before = r.nb;
    r.nb = nb_before + 1;
    const float4 N4 = __ldg(nrm + h.k);
    const float3 n = make_float3(N4.x, N4.y, N4.z);
    float dn, dnl;
    tf_dot3(r.d, n, dn, dnl);
    const float3 nf = dn < 0.f ? n : make_float3(-n.x, -n.y, -n.z);
    r.nfs = dn < 0.f ? 1.f : -1.f;
    const float adn = fabsf(dn);
    const float3 rh = make_float3(A.rhat[0], A.rhat[1], A.rhat[2]);
    if (r.nb == 1) r.cos0 = dot3(nf, rh);
    // candidate path L = k.o0 + sum t - r_rx.x (monostatic: r_rx = -k)
    float kh, kl;
    tf_dot(A.rxdir, x, kh, kl);
    r.lc_hi = r.lacc_hi;
    r.lc_lo = r.lacc_lo;
    tf_add_tf(r.lc_hi, r.lc_lo, kh, kl);
    // H-transmit field from the V one: E_H = s (d x E_V), s = +1 after an odd number of reflections
    const float sH = (nb_before & 1) ? 1.f : -1.f;
    const float3 eh = make_float3(sH * (r.d.y * r.ev.z - r.d.z * r.ev.y), sH * (r.d.z * r.ev.x - r.d.x * r.ev.z),
                                  sH * (r.d.x * r.ev.y - r.d.y * r.ev.x));
    const float dS = adn > 0.f ? __fdiv_rn(A.dA, adn) : 0.f;
    const float nfd = dot3(nf, r.d);
    // radiation toward the receiver, projected on its basis
    const float3 rr = make_float3(A.rxr[0], A.rxr[1], A.rxr[2]);
    const float3 vh = make_float3(A.rxv[0], A.rxv[1], A.rxv[2]);
    const float3 hh = make_float3(A.rxh[0], A.rxh[1], A.rxh[2]);
    float3 W[2];
    const float3 Eq[2] = {eh, r.ev};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float ne = dot3(nf, Eq[q]);
        // J = 2 nf x (d x E) = 2 (d (nf.E) - E (nf.d))
        const float3 J = make_float3(2.f * (r.d.x * ne - Eq[q].x * nfd), 2.f * (r.d.y * ne - Eq[q].y * nfd),
                                     2.f * (r.d.z * ne - Eq[q].z * nfd));
        const float jr = dot3(J, rr);
        W[q] = make_float3(dS * (J.x - jr * rr.x), dS * (J.y - jr * rr.y), dS * (J.z - jr * rr.z));
    }
    r.c[0] = dot3(W[0], hh);  // HH
    r.c[1] = dot3(W[1], vh);  // VV
    r.c[2] = dot3(W[1], hh);  // HV
    r.c[3] = dot3(W[0], vh);  // VH
    const float gam = (r.nb & 1) ? -1.f : 1.f;  // Gamma^N, Gamma = -1
    r.c[4] = -2.f * A.dA * r.cos0 * gam;
    if (flags & kFlagLiteral) {
        // scalar form with e^{-j 2 k R}: L = 2 (k.o0 + R), stored in the candidate path
        r.lc_hi = 2.f * r.lacc_hi;
        r.lc_lo = 2.f * r.lacc_lo;
    }
    // PEC field update (FP32), then the stored reflection and offset origin
    const float nev = dot3(n, r.ev);
    r.ev = make_float3(fmaf(2.f * nev, n.x, -r.ev.x), fmaf(2.f * nev, n.y, -r.ev.y), fmaf(2.f * nev, n.z, -r.ev.z));
    const float m2 = -2.f * dn;
    r.d = make_float3(__fmaf_rn(m2, n.x, r.d.x), __fmaf_rn(m2, n.y, r.d.y), __fmaf_rn(m2, n.z, r.d.z));
    r.o = make_float3(__fmaf_rn(A.eps, nf.x, x.x), __fmaf_rn(A.eps, nf.y, x.y), __fmaf_rn(A.eps, nf.z, x.z));
    r.last = h.k;
}

__device__ __forceinline__ long long ray_global(const TraceArgs& a, const Ray& r)
{
    return a.ray_off[r.angle] + r.local;
}

// Rays are processed in tiles of W x H = 32 grid points (W = 2^tw_log2, 8 x 4
// by default): processing index p of an aspect maps to grid point
// (i, j) = (W bu + p % W, H bv + (p % 32) / W), tile p / 32 = bv * nbu + bu,
// so the 32 lanes of a warp trace a compact patch of the aperture.
__device__ __forceinline__ void tile_ij(const AngleDev& A, int p, int& i, int& j)
{
    const int blk = p >> 5, l = p & 31, tw = A.tw_log2;
    const int bv = blk / A.nbu, bu = blk - bv * A.nbu;
    i = (bu << tw) + (l & ((1 << tw) - 1));
    j = bv * (32 >> tw) + (l >> tw);
}

// Whether a query meets any triangle: binary traversal, near child first, that
// ends at the first certain hit (whether one exists depends on no order). Out of
// line, so that its registers do not burden the bounce kernel, which asks it at
// one place (33 bistatic aspects of a 250k-triangle aircraft at 3 GHz: with the
// first hits listed instead of stored, 6.51 ms per trace and PO sum; 6.82 with a
// closest-hit query and stored states).
__device__ __noinline__ bool any_hit(const TraceArgs& a, float3 o, float3 d, int skip, bool& overflow)
{
    constexpr int kStack = 64;
    int stack[kStack];
    const float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    const float3 oi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    const float2 ix = make_float2(inv.x, inv.x), iy = make_float2(inv.y, inv.y), iz = make_float2(inv.z, inv.z);
    const float2 mx = make_float2(-oi.x, -oi.x), my = make_float2(-oi.y, -oi.y), mz = make_float2(-oi.z, -oi.z);
    int sp = 0, ref = 0;
    for (int it = 0;; ++it) {
        if (it >= a.visit_limit) {
            overflow = true;
            return true;
        }
        if (ref >= 0) {
            const float4* nd = a.nodes2 + 4 * (size_t)ref;
            const float4 n0 = __ldg(nd), n1 = __ldg(nd + 1), n2 = __ldg(nd + 2), n3 = __ldg(nd + 3);
            const float2 ax = fma2(make_float2(n0.x, n0.y), ix, mx), ay = fma2(make_float2(n0.z, n0.w), iy, my);
            const float2 az = fma2(make_float2(n2.x, n2.y), iz, mz), bx = fma2(make_float2(n1.x, n1.y), ix, mx);
            const float2 by = fma2(make_float2(n1.z, n1.w), iy, my), bz = fma2(make_float2(n2.z, n2.w), iz, mz);
            const float an = fmaxf(fmaxf(fminf(ax.x, ax.y), fminf(ay.x, ay.y)), fmaxf(fminf(az.x, az.y), 0.f));
            const float af = fminf(fminf(fmaxf(ax.x, ax.y), fmaxf(ay.x, ay.y)), fmaxf(az.x, az.y));
            const float bn = fmaxf(fmaxf(fminf(bx.x, bx.y), fminf(by.x, by.y)), fmaxf(fminf(bz.x, bz.y), 0.f));
            const float bf = fminf(fminf(fmaxf(bx.x, bx.y), fmaxf(by.x, by.y)), fmaxf(bz.x, bz.y));
            const int lref = __float_as_int(n3.x), rref = __float_as_int(n3.y);
            const bool hl = an <= af * kBoxGrow;
            const bool hr = (bn <= bf * kBoxGrow) && (rref != kEmptyRef);
            if (hl && hr) {
                const bool lnear = an <= bn;
                if (sp < kStack) stack[sp++] = lnear ? rref : lref;
                else overflow = true;
                ref = lnear ? lref : rref;
                continue;
            }
            if (hl) { ref = lref; continue; }
            if (hr) { ref = rref; continue; }
        } else {
            const int first = leaf_first(ref), cnt = leaf_count(ref);
            for (int k = first; k < first + cnt; ++k) {
                if (k == skip) continue;
                const float4* tp = a.tris + 3 * (size_t)k;
                float tc, et;
                const int f = tri_filter(__ldg(tp), __ldg(tp + 1), __ldg(tp + 2), o, d, tc, et);
                if (f == 1 || (f >= 2 && (tri_refine(a.tris, a.tri_v12, k, o, d, f + 2, tc) & 1))) return true;
            }
        }
        if (sp == 0) return false;
        ref = stack[--sp];
    }
}

// Bistatic: the last hit contributes only if the receiver lies on the side of
// its oriented FP32 normal (the sign of the exact dot product) and a query from
// the offset origin toward the receiver meets no triangle (the one just hit is
// skipped).
__device__ __forceinline__ bool rx_visible(const TraceArgs& a, const AngleDev& A, const Ray& r, unsigned& nq,
                                           bool& ovf)
{
    const float4 N4 = __ldg(a.tri_nrm + r.last);
    const float3 n = make_float3(N4.x * r.nfs, N4.y * r.nfs, N4.z * r.nfs);
    const float3 rx = make_float3(A.rxr[0], A.rxr[1], A.rxr[2]);
    float sh, sl;
    tf_dot3(n, rx, sh, sl);  // the sign of the exact dot product
    if (!(sh > 0.f)) return false;
    ++nq;
    bool over = false;
    const bool hit = any_hit(a, r.o, rx, r.last, over);
    ovf = ovf || over;
    return !hit;
}

__device__ __forceinline__ void emit(const TraceArgs& a, const Ray& r, bool zero)
{
    const long long g = ray_global(a, r);
    int i, j;
    const AngleDev& A = a.angles[r.angle];
    tile_ij(A, r.local, i, j);
    const int ray_id = j * A.nu + i;
    const long long tile = g >> 5;
    const unsigned bit = (unsigned)(g & 31);
    const unsigned slot = a.tile_base[tile] + __popc(a.mask[tile] & ((1u << bit) - 1u));
    Record* rec = a.rec_of ? a.rec + a.rec_of[r.angle] : a.rec;
    float4* p = reinterpret_cast<float4*>(rec + slot);
    if (zero) {
        __stcs(p + 0, make_float4(0.f, 0.f, 0.f, 0.f));
        __stcs(p + 1, make_float4(0.f, 0.f, 0.f, __int_as_float(ray_id)));
    } else {
        __stcs(p + 0, make_float4(r.c[0], r.c[1], r.c[2], r.c[3]));
        __stcs(p + 1, make_float4(r.c[4], r.lc_hi, r.lc_lo, __int_as_float(ray_id)));
    }
    if (a.hit_nb) a.hit_nb[g] = r.nb;
}

__device__ __forceinline__ void record_hit(const TraceArgs& a, const Ray& r, const Hit& h)
{
    if (!a.hit_tri) return;
    const long long g = ray_global(a, r);
    a.hit_tri[g * a.max_bounces + (r.nb - 1)] = h.orig;
    a.hit_t[g * a.max_bounces + (r.nb - 1)] = h.t;
}

__device__ __forceinline__ int find_angle(const long long* __restrict__ off, int n, long long g)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// the same by a whole warp (converged), 32 candidates a step
__device__ __forceinline__ int find_angle_warp(const long long* __restrict__ off, int n, long long g)
{
    const int lane = threadIdx.x & 31;
    int lo = 0;
    while (n > 1) {  // off[lo] <= g, and off[lo + n] > g or lo + n is the end
        const int step = (n + 31) >> 5, i = lane * step;
        const unsigned m = __ballot_sync(kFull, i < n && off[lo + i] <= g);
        const int k = max(31 - __clz(m), 0) * step;
        lo += k;
        n = min(step, n - k);
    }
    return lo;
}

// warp-aggregated append of the lanes of m to queue q; every lane of the warp must call it
__device__ __forceinline__ void append(RayState* q, unsigned* count, unsigned m, const Ray& r)
{
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(count, (unsigned)__popc(m));
    base = __shfl_sync(kFull, base, leader);
    if ((m >> lane) & 1u) store_state(q, base + __popc(m & ((1u << lane) - 1u)), r);
}

// the rays that go on: to the live-ray queue, or to the ray pool while it has room
__device__ __forceinline__ void push(const TraceArgs& a, bool want, Ray& r)
{
    const unsigned m = __ballot_sync(kFull, want);
    if (!m) return;
    if (!a.pool) {
        append(a.q_out, a.q_out_count, m, r);
        return;
    }
    r.angle += a.angle_shift;  // the pool indexes the trace's aspects
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    unsigned base = 0;
    if (lane == leader) base = atomicAdd(a.pool_count, (unsigned)__popc(m));
    base = __shfl_sync(kFull, base, leader);
    const unsigned idx = base + __popc(m & ((1u << lane) - 1u));
    const bool fit = want && idx < a.pool_cap;
    if (fit) store_state(a.pool, idx, r);
    const unsigned over = __ballot_sync(kFull, want && !fit);
    if (over) append(a.q_out, a.q_out_count, over, r);  // kept until the pool has been traced
}

template <bool kCount>
__device__ __forceinline__ void flush_stats(const TraceArgs& a, unsigned q, unsigned nvis, unsigned ntri, bool ovf,
                                            unsigned nhit = 0, unsigned nlist = 0, unsigned long long wvis = 0)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        q += __shfl_xor_sync(kFull, q, o);
        if (kCount) {
            nvis += __shfl_xor_sync(kFull, nvis, o);
            ntri += __shfl_xor_sync(kFull, ntri, o);
            nhit += __shfl_xor_sync(kFull, nhit, o);
            nlist += __shfl_xor_sync(kFull, nlist, o);
        }
    }
    const unsigned ov = __ballot_sync(kFull, ovf);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(a.stats + kStatQueries, (unsigned long long)q);
        if (kCount) {
            atomicAdd(a.stats + kStatNodes, (unsigned long long)nvis);
            atomicAdd(a.stats + kStatTris, (unsigned long long)ntri);
            if (nhit) atomicAdd(a.stats + kStatHits, (unsigned long long)nhit);
            if (nlist) atomicAdd(a.stats + kStatListed, (unsigned long long)nlist);
            if (wvis) atomicAdd(a.stats + kStatWarpNodes, wvis);
        }
        if (ov) atomicAdd(a.stats + kStatOverflow, (unsigned long long)__popc(ov));
    }
}

// One closest-hit query per lane. kMode 0: per-lane binary traversal; 1: per-lane
// 4-wide traversal; 2: warp-cooperative binary traversal (all 32 lanes call it);
// 3: per-lane binary traversal over the octant node copies.
template <bool kCount, int kStack, int kMode>
__device__ __forceinline__ void query(const TraceArgs& a, bool active, float3 o, float3 d, int skip, Hit& h,
                                      unsigned& nvis, unsigned& ntri, bool& ovf)
{
    if (kMode == 2) {
        closest_hit_packet<kCount, (kStack < 64 ? kStack : 64)>(a.nodes, tri_refs(a), active, o, d, skip, a.visit_limit, h,
                                                                nvis, ntri, ovf);
    } else if (active) {
        if (kMode == 1) closest_hit4<kCount, kStack>(a.nodes, tri_refs(a), o, d, skip, a.visit_limit, h, nvis, ntri, ovf);
        else if (kMode == 3)
            closest_hit_oct<kCount, kStack>(a.nodes, a.n_nodes, tri_refs(a), o, d, skip, a.visit_limit, h, nvis, ntri, ovf);
        else closest_hit<kCount, kStack>(a.nodes, tri_refs(a), o, d, skip, a.visit_limit, h, nvis, ntri, ovf);
    }
    if (active) key_closest(tri_refs(a), o, d, h);
}

// ---------------------------------------------------------------- silhouette mask
// Ray (i, j) of an aspect travels along k through the aperture point
// u = u0 + i ds, v = v0 + j ds (u, v along H and V; u0, v0 those of P0). It can
// only hit a triangle whose projection contains (u, v); the FP32 ray origin,
// the intersection slack (2^-12 of the determinant) and the FP32 projection
// below all stay within the margin of 0.01 cell + 2^-10 of the triangle's
// projected extent + 2^-18 of its distance from P0 + 2^-22 of |P0|_1 (in cells).
// The last covers the roundings that grow with the coordinates, not with the
// target: u |v_k| of a vertex v0 + e and 2 u |o_k| of a ray origin per component,
// 3 u |P0|_1 along an axis beyond what the distance covers (a target of 10 m at
// 10 km from the origin on an 8 mm grid: 0.4 cells). One thread
// projects one triangle for one aspect and ORs its cells into the tile words.
// A triangle whose widened box spans more than 2^16 cells sets the aspect's
// "all rays" flag (word total_tiles + aspect) instead.
// The grid cells (i0..i1, j0..j1) of aspect A whose rays the FP32 test could
// accept on triangle (a: v0, b: e1, c: e2); false if none.
// ids = 1 / sqrt(A.dA), the inverse grid spacing (FP32, set with the aspect table)
__device__ __forceinline__ float cell_scale(const AngleDev& A) { return A.ids; }

// The triangle's vertices projected onto the aspect's grid (in cells from P0),
// their ranges and their largest distance from P0 (in cells)
struct TriProj {
    float u[3], v[3], umin, umax, vmin, vmax, mag, m0;  // m0: AngleDev::r_m0
};

__device__ __forceinline__ void tri_project(const AngleDev& A, float ids, float4 a, float4 b, float4 c, TriProj& pr)
{
    const float px[3] = {a.x, a.x + b.x, a.x + c.x}, py[3] = {a.y, a.y + b.y, a.y + c.y},
                pz[3] = {a.z, a.z + b.z, a.z + c.z};
    pr.umin = FLT_MAX;
    pr.umax = -FLT_MAX;
    pr.vmin = FLT_MAX;
    pr.vmax = -FLT_MAX;
    pr.mag = 0.f;
    pr.m0 = A.r_m0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float dx = px[k] - A.p0[0], dy = py[k] - A.p0[1], dz = pz[k] - A.p0[2];
        const float u = (dx * A.hhat[0] + dy * A.hhat[1] + dz * A.hhat[2]) * ids;
        const float v = (dx * A.vhat[0] + dy * A.vhat[1] + dz * A.vhat[2]) * ids;
        pr.u[k] = u;
        pr.v[k] = v;
        pr.umin = fminf(pr.umin, u);
        pr.umax = fmaxf(pr.umax, u);
        pr.vmin = fminf(pr.vmin, v);
        pr.vmax = fmaxf(pr.vmax, v);
        pr.mag = fmaxf(pr.mag, (fabsf(dx) + fabsf(dy) + fabsf(dz)) * ids);
    }
}

__device__ __forceinline__ bool tri_cells_p(const AngleDev& A, const TriProj& pr, int& i0, int& i1, int& j0, int& j1)
{
    const float umin = pr.umin, umax = pr.umax, vmin = pr.vmin, vmax = pr.vmax;
    if (!(umin <= umax) || !(vmin <= vmax)) return false;  // NaN vertices: no ray can hit it
    const float m = pr.m0 + (umax - umin + vmax - vmin) * (1.f / 1024.f) + pr.mag * (1.f / 262144.f);
    const float fi0 = ceilf(umin - m), fi1 = floorf(umax + m), fj0 = ceilf(vmin - m), fj1 = floorf(vmax + m);
    if (fi1 < 0.f || fj1 < 0.f || fi0 > (float)(A.nu - 1) || fj0 > (float)(A.nv - 1)) return false;
    i0 = max(0, (int)fi0);
    i1 = min(A.nu - 1, (int)fi1);
    j0 = max(0, (int)fj0);
    j1 = min(A.nv - 1, (int)fj1);
    return true;
}

__device__ __forceinline__ bool tri_cells(const AngleDev& A, float ids, float4 a, float4 b, float4 c, int& i0, int& i1,
                                          int& j0, int& j1)
{
    TriProj pr;
    tri_project(A, ids, a, b, c, pr);
    return tri_cells_p(A, pr, i0, i1, j0, j1);
}

// The projected triangle as three edge half-planes in the cell coordinates of
// an item's range (origin at its first cell i0, j0): cell (i, j) passes when
// nx (i - i0) + ny (j - j0) + c <= 0 for every edge. Each half-plane is moved
// outward by the margin m of tri_cells (the vertices' and ray origins' FP32
// errors) plus 0.002 cells (the local shift) and 1e-5 of the range per unit of
// |n| (the evaluation), so every cell of the conservative range whose ray the
// exact test can accept passes: the moved half-planes contain the projection
// widened by m in u and v. A projection of (nearly) zero area keeps every
// cell of the range.
struct CellEdges {
    float nx[3], ny[3], c[3];
};

__device__ __forceinline__ void tri_cell_edges_p(const TriProj& pr, int i0, int i1, int j0, int j1, CellEdges& E)
{
    float u[3], v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        u[k] = pr.u[k] - (float)i0;
        v[k] = pr.v[k] - (float)j0;
    }
    const float m =
        pr.m0 + (pr.umax - pr.umin + pr.vmax - pr.vmin) * (1.f / 1024.f) + pr.mag * (1.f / 262144.f) + 0.002f;
    const float a2 = (u[1] - u[0]) * (v[2] - v[0]) - (v[1] - v[0]) * (u[2] - u[0]);
    const float sg = a2 > 0.f ? 1.f : -1.f;
    const bool flat = !(fabsf(a2) > 1e-2f);
    const float ext = 1e-5f * (float)(i1 - i0 + j1 - j0 + 2);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int k1 = k == 2 ? 0 : k + 1;
        // outward normal of edge k -> k1 (counter-clockwise after the sign sg)
        const float nx = sg * (v[k1] - v[k]), ny = -sg * (u[k1] - u[k]);
        const float w = (fabsf(nx) + fabsf(ny)) * (m + ext);
        E.nx[k] = flat ? 0.f : nx;
        E.ny[k] = flat ? 0.f : ny;
        E.c[k] = flat ? -1.f : -(nx * u[k] + ny * v[k]) - w;
    }
}

__device__ __forceinline__ void tri_cell_edges(const AngleDev& A, float ids, float4 a, float4 b, float4 c, int i0,
                                               int i1, int j0, int j1, CellEdges& E)
{
    TriProj pr;
    tri_project(A, ids, a, b, c, pr);
    tri_cell_edges_p(pr, i0, i1, j0, j1, E);
}

__global__ void __launch_bounds__(256) k_silhouette(const float4* __restrict__ tris, int n_tri,
                                                    const AngleDev* __restrict__ angles,
                                                    const long long* __restrict__ ray_off, int n_angles,
                                                    long long total_tiles, unsigned* cover)
{
    for (int ang = blockIdx.y; ang < n_angles; ang += gridDim.y) {
        const AngleDev& A = angles[ang];
        const int tw = A.tw_log2, W = 1 << tw, H = 32 >> tw;
        const float ids = cell_scale(A);
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n_tri; t += gridDim.x * blockDim.x) {
            const float4 a = __ldg(tris + 3 * (size_t)t), b = __ldg(tris + 3 * (size_t)t + 1),
                         c = __ldg(tris + 3 * (size_t)t + 2);
            int i0, i1, j0, j1;
            if (!tri_cells(A, ids, a, b, c, i0, i1, j0, j1)) continue;
            if ((long long)(i1 - i0 + 1) * (j1 - j0 + 1) > 65536) {
                atomicOr(cover + total_tiles + ang, 1u);
                continue;
            }
            const long long base = ray_off[ang];
            for (int j = j0; j <= j1; ++j) {
                const int bv = j / H, jl = j - bv * H;
                for (int i = i0; i <= i1;) {
                    const int bu = i >> tw, ie = min(i1, (bu << tw) + W - 1);
                    // bits (jl W + i % W) .. (jl W + ie % W) of tile (bv nbu + bu)
                    const int lo = jl * W + (i & (W - 1)), hi = jl * W + (ie & (W - 1));
                    const unsigned bits = (hi - lo == 31) ? 0xFFFFFFFFu : (((1u << (hi - lo + 1)) - 1u) << lo);
                    atomicOr(cover + ((base >> 5) + (long long)bv * A.nbu + bu), bits);
                    i = ie + 1;
                }
            }
        }
    }
}

// origin of primary ray (i, j) of aspect A (Eq. L1-L3 grid), in FP32
__device__ __forceinline__ float3 primary_origin(const AngleDev& A, int i, int j)
{
    const float fi = (float)i, fj = (float)j;
    return make_float3(__fadd_rn(__fadd_rn(A.p0[0], __fmul_rn(fi, A.du[0])), __fmul_rn(fj, A.dv[0])),
                       __fadd_rn(__fadd_rn(A.p0[1], __fmul_rn(fi, A.du[1])), __fmul_rn(fj, A.dv[1])),
                       __fadd_rn(__fadd_rn(A.p0[2], __fmul_rn(fi, A.du[2])), __fmul_rn(fj, A.dv[2])));
}

// ---------------------------------------------------------------- primary hits by rasterisation
// All primary rays of an aspect are parallel, so the closest hit of every ray
// can be found triangle by triangle: the FP32 test of a triangle runs for every
// grid ray in its conservative cell range (the silhouette range, which
// contains every ray the test accepts), and each ray keeps the smallest key
// (t bits << 32 | original index) by a 64-bit atomic minimum. t > 0, so the
// key order is (t, index): the closest hit and the tie rule of the traversal,
// whose t is <= FLT_MAX. A triangle spanning more than kRasterMaxCells cells
// (or of an aperture row or column of more than 65,535 rays) flags its aspect
// instead, whose primary rays then traverse the tree.

// An aspect's ray grid held in registers for the cell loops: the loops' atomics
// could alias the aspect table as far as the compiler knows, so fields read
// through it would be loaded again after every atomic.
struct RasterGrid {
    float3 p0, du, dv, d;
    int nbu, tw;
};

__device__ __forceinline__ RasterGrid raster_grid(const AngleDev& A)
{
    RasterGrid G;
    G.p0 = make_float3(A.p0[0], A.p0[1], A.p0[2]);
    G.du = make_float3(A.du[0], A.du[1], A.du[2]);
    G.dv = make_float3(A.dv[0], A.dv[1], A.dv[2]);
    G.d = make_float3(A.dir[0], A.dir[1], A.dir[2]);
    G.nbu = A.nbu;
    G.tw = A.tw_log2;
    return G;
}

// the origin of grid ray (i, j): primary_origin's operations in its order
__device__ __forceinline__ float3 grid_origin(const RasterGrid& G, int i, int j)
{
    const float fi = (float)i, fj = (float)j;
    return make_float3(__fadd_rn(__fadd_rn(G.p0.x, __fmul_rn(fi, G.du.x)), __fmul_rn(fj, G.dv.x)),
                       __fadd_rn(__fadd_rn(G.p0.y, __fmul_rn(fi, G.du.y)), __fmul_rn(fj, G.dv.y)),
                       __fadd_rn(__fadd_rn(G.p0.z, __fmul_rn(fi, G.du.z)), __fmul_rn(fj, G.dv.z)));
}

// A triangle seen by the parallel rays of an aspect (direction d): the cross
// products of the triangle test depend on d and the triangle only, so with
// S = o - v0, U = S.(d x e2), V = S.(e1 x d) and T = S.(e1 x e2) (the same triple
// products) are three dot products per ray. Their error bounds are those of
// tri_filter (each below 8 u sum|S_i| of the absolute cross products).
struct RasterTri {
    float3 v0, p, p2, nn;  // vertex 0, d x e2, e1 x d, e1 x e2
    float det, bd;         // e1 . (d x e2) and its error bound (-1: degenerate, no hits)
    float bU, bV, bT;      // error bounds of U, V and T for every cell of the range
};

// The per-cell bounds 8.1 u |S|.(|d| x |e2|), 8.1 u |S|.(|e1| x |d|) and
// 9.1 u |S|.(|e1| x |e2|) taken once for the cell range i0..i1, j0..j1: each
// |S_c| is at most its largest value at the range's corner rays (|o - v0| is
// convex in (i, j) for the exact grid points) plus 8 u of the largest |o_c|
// (the FP32 rounding of the ray origins and of S).
__device__ __forceinline__ RasterTri raster_tri(const RasterGrid& G, float4 P, float4 B, float4 C, int i0, int i1,
                                                int j0, int j1)
{
    RasterTri R;
    const float3 e1 = make_float3(B.x, B.y, B.z), e2 = make_float3(C.x, C.y, C.z), d = G.d;
    R.v0 = make_float3(P.x, P.y, P.z);
    R.p = cross_s(d, e2);
    R.p2 = cross_s(e1, d);
    R.nn = cross_s(e1, e2);
    R.det = dot_s(e1, R.p);
    const float3 pa = cross_abs(d, e2);
    R.bd = B.w > 0.f ? 0x1.03p-21f * dot_s(abs3(e1), pa) : -1.f;
    float3 sm = make_float3(0.f, 0.f, 0.f), om = make_float3(0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float3 o = grid_origin(G, (c & 1) ? i1 : i0, (c & 2) ? j1 : j0);
        sm = make_float3(fmaxf(sm.x, fabsf(o.x - R.v0.x)), fmaxf(sm.y, fabsf(o.y - R.v0.y)),
                         fmaxf(sm.z, fabsf(o.z - R.v0.z)));
        om = make_float3(fmaxf(om.x, fabsf(o.x)), fmaxf(om.y, fabsf(o.y)), fmaxf(om.z, fabsf(o.z)));
    }
    const float g = 8.f * kU;
    sm = make_float3(__fmaf_rn(g, om.x + fabsf(R.v0.x), sm.x), __fmaf_rn(g, om.y + fabsf(R.v0.y), sm.y),
                     __fmaf_rn(g, om.z + fabsf(R.v0.z), sm.z));
    R.bU = 0x1.03p-21f * dot_s(sm, pa);
    R.bV = 0x1.03p-21f * dot_s(sm, cross_abs(e1, d));
    R.bT = 0x1.23p-21f * dot_s(sm, cross_abs(e1, e2));
    return R;
}

__device__ __forceinline__ void raster_cell(const RasterGrid& G, const TraceArgs& a, const RasterTri& R,
                                            const PlaneKey& K, int k, unsigned orig, int i, int j,
                                            unsigned long long* vrow, int count)
{
    const float3 o = grid_origin(G, i, j);
    const float3 s = make_float3(__fsub_rn(o.x, R.v0.x), __fsub_rn(o.y, R.v0.y), __fsub_rn(o.z, R.v0.z));
    float tc, et;
    // V = S.(e1 x d) and T = S.(e1 x e2) are the triple products of tri_filter, with the same bounds
    const int f = filter_core(dot_s(s, R.p), dot_s(s, R.p2), dot_s(s, R.nn), R.det, R.bU, R.bV, R.bd, R.bT, tc, et);
    if (f == 0) return;
    if (f >= 2) {
        const int r = tri_refine(a.tris, a.tri_v12, k, o, G.d, f, tc);
        if (count) count_open(a.stats, r);
        if (!(r & 1)) return;
    }
    const float th = plane_key_t(K, R.v0, o, tc);
    if (th >= 0.f && th <= FLT_MAX) {
        const int tw = G.tw, sh = 5 - tw;  // tile of W = 2^tw by H = 2^sh rays
        const int bu = i >> tw, bv = j >> sh;
        const long long pidx = ((long long)(bv * G.nbu + bu) << 5) + ((j & ((1 << sh) - 1)) << tw) + (i & ((1 << tw) - 1));
        atomicMin(vrow + pidx, ((unsigned long long)__float_as_uint(th) << 32) | orig);
    }
}

// Below the smallest stored distance that a ray of the grid (origin p0,
// direction d) can have on a triangle: the distances along d of the vertices
// from the grid plane (the ray origins lie in it to within micrometres and a few
// roundings of the coordinates, 2^-21 |p0|_1 with those of the vertices); the
// stored distance of any hit is at least their minimum less the key's plane
// slack (0.08 bUV / |d.n|, as in key_of), 1e-4 of it and 1 mm.
__device__ __forceinline__ float raster_tnear(float4 P, float4 B, float4 C, float3 p0, float3 d, const PlaneKey& K)
{
    const float3 q0 = make_float3(P.x - p0.x, P.y - p0.y, P.z - p0.z);
    const float z0 = dot_s(q0, d), z1 = z0 + dot_s(make_float3(B.x, B.y, B.z), d),
                z2 = z0 + dot_s(make_float3(C.x, C.y, C.z), d);
    const float zm = fminf(z0, fminf(z1, z2));
    const float slack = K.dh != 0.f ? 0.32f * B.w / fabsf(K.dh) : FLT_MAX;
    const float at = (fabsf(p0.x) + fabsf(p0.y) + fabsf(p0.z)) * 0x1p-21f;
    const float tnear = zm - (1e-4f * fabsf(zm) + 1e-3f + at + slack);
    return isfinite(tnear) ? tnear : -FLT_MAX;
}

// A triangle of the flattened rasterisation and everything its cells need,
// one per lane in shared memory as 13 16-byte words (a stride of 52 words: the
// 16-byte accesses of 8 lanes to different triangles fall in distinct banks,
// and lanes reading one triangle's fields share a broadcast):
//   g0 = (p0.x, p0.y, p0.z, du.x)   g1 = (du.y, du.z, dv.x, dv.y)   g2 = (dv.z, v0.x, v0.y, v0.z)
//   r0 = (p.x, p.y, p.z, p2.x)      r1 = (p2.y, p2.z, nn.x, nn.y)   r2 = (nn.z, det, bd, bU)
//   r3 = (bV, bT, n.x, n.y)         r4 = (n.z, dh, dl, rd)           [plane key K]
//   e0 = (nx0, ny0, c0, nx1)        e1 = (ny1, c1, nx2, ny2)         e2 = (c2, -, tnear, ray_off)
//   m0 = (i0, j0, w, orig)          m1 = (aspect, triangle, nbu, tw)
// tnear: below the smallest stored distance any cell of the range can give
// this triangle (a cell whose ray already holds a closer hit is skipped).
struct __align__(16) RasterItem {
    float4 g0, g1, g2, r0, r1, r2, r3, r4, e0, e1, e2;
    int4 m0, m1;
};
static_assert(sizeof(RasterItem) == 52 * 4, "RasterItem layout");
constexpr int kRasterWarps = 8;    // warps of a k_raster block
constexpr int kRasterFlat = 512;   // cells of a triangle the warps flatten; larger ones go to k_raster_big
constexpr size_t kRasterSmem = sizeof(RasterItem) * 32 * kRasterWarps;

// Appends the large triangles of the warp's lanes (want; cell ranges i0..i1,
// j0..j1 of aspect ang) to the list of k_raster_big, cut into bands of rows of
// about kRasterBand cells: a warp of k_raster_big takes a band at a time, so a
// plate of millions of cells is shared by all of them (traversing all rays of
// an aspect for its triangles above 2^14 cells: 4.0 of 41 ms for 23 aircraft
// aspects at 7 to 12 GHz). The aspects of entries that find the list full
// traverse, and so do those whose triangles above kRasterBanded cells cover
// more than 20 box cells per ray: every layer is a test of every ray, while the
// traversal stops at the first (4 aspects of 3000 x 3000 rays on stacked
// plates of two triangles, B = 2, banded against traversed: 1 plate 1.5 / 4.1 ms,
// 10: 4.0 / 4.4, 30: 9.0 / 4.7, 300: 73 / 8.2). Every lane of the warp calls it.
constexpr int kRasterBand = 4096, kRasterBanded = 1 << 14;
__device__ __forceinline__ void append_big(const TraceArgs& a, unsigned* full, bool want, int t, int ang, int i0, int i1,
                                           int j0, int j1)
{
    if (!__any_sync(kFull, want)) return;
    if (want) {
        const unsigned cells = (unsigned)((i1 - i0 + 1) * (j1 - j0 + 1));
        if (cells > kRasterBanded) {
            // the aspect's sum of such triangles' cells, in units of 1024 (its last value, and so whether the aspect
            // traverses, does not depend on the order; left alone above the limit, so that it cannot wrap)
            unsigned* sum = full + a.n_angles + 1 + ang;
            const unsigned most = (unsigned)(20 * (a.ray_off[ang + 1] - a.ray_off[ang]) >> 10), n = (cells + 1023u) >> 10;
            if (__ldcg(sum) > most || atomicAdd(sum, n) + n > most) {
                want = false;
                atomicOr(full + ang, 1u);
                atomicOr(full + a.n_angles, 1u);  // some aspect of the chunk traverses
            }
        }
    }
    const int lane = threadIdx.x & 31;
    const int rows = want ? max(1, kRasterBand / (i1 - i0 + 1)) : 1;
    const unsigned n = want ? (unsigned)((j1 - j0 + rows) / rows) : 0u;  // bands
    unsigned incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    unsigned base = 0xFFFFFFFFu;
    // (a full list is left alone, so that its counter cannot wrap)
    if (lane == 31 && __ldcg(a.big_ctr) < a.big_cap) base = atomicAdd(a.big_ctr, incl);
    base = __shfl_sync(kFull, base, 31);
    if (!want) return;
    bool fit = base != 0xFFFFFFFFu;
    if (fit) {
        const unsigned slot = base + incl - n;
        for (unsigned k = 0; k < n; ++k) {
            const int jb = j0 + (int)k * rows;
            if (slot + k < a.big_cap)
                a.big[slot + k] = make_int4(t, ang, i0 | (jb << 16), (i1 - i0) | ((min(j1, jb + rows - 1) - jb) << 16));
            else fit = false;
        }
    }
    if (!fit) {
        atomicOr(full + ang, 1u);
        atomicOr(full + a.n_angles, 1u);  // some aspect of the chunk traverses
    }
}

// the same out of line, for warps with any (k_raster_sparse, whose projection it would burden; inline a band takes 37 ns
// of a lane, out of line 91)
__device__ __noinline__ void append_some(const TraceArgs& a, unsigned* full, bool want, int t, int ang, int i0, int i1,
                                         int j0, int j1)
{
    append_big(a, full, want, t, ang, i0, i1, j0, j1);
}

// The cells of row y inside an item's moved edges: columns [lo, lo + cnt) of
// w <= 65536, found on the values of a cell's pretest (nx x + g <= 0 is
// x <= -g / nx) and widened by more than the quotient's error, so that no cell
// the pretest passes is left out. Each triangle's box holds about three times
// the cells of the triangle itself (29M and 9M for an aircraft aspect at
// 10 GHz); testing them one by one left two lanes of three idle in the exact
// test that follows: k_raster 8.2 ms for 37 such aspects, 4.7 with spans.
__device__ __forceinline__ void row_span(const float* nx, const float* ny, const float* c, float y, int w, int& lo, int& cnt)
{
    float x0 = 0.f, x1 = (float)(w - 1);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float g = fmaf(ny[k], y, c[k]), q = __fdividef(-g, nx[k]);
        if (nx[k] >= 1e-20f) x1 = fminf(x1, q);
        else if (nx[k] <= -1e-20f) x0 = fmaxf(x0, q);
        else if (g > 1e-15f) x1 = -1.f;  // along the row (either zero): all of its cells or none
    }
    // (a quotient may be infinite or none: 0 <= lo <= w + 1, -1 <= the last column < w)
    const float tol = fmaf((float)w, 1e-6f, 0.01f);
    lo = __float2int_ru(fminf(x0, (float)(w + 1)) - tol);
    lo = max(lo, 0);
    cnt = max(min(__float2int_rd(fmaxf(x1, -1.f) + tol), w - 1) - lo + 1, 0);
}

// Calls cell(k, row, column) for the cells of the lanes' rows (row `row` of
// triangle k < 32, columns [lo, lo + cnt)), 32 cells at a time, one per lane.
// A warp's rows hold fewer than 65,536 cells before the last one. spans: the
// warp's 32 entries; every lane calls it.
template <class Cell>
__device__ __forceinline__ void each_cell(uint2* spans, int k, int row, int lo, int cnt, Cell cell)
{
    const int lane = threadIdx.x & 31;
    const unsigned le = 0xFFFFFFFFu >> (31 - lane);
    int end = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, end, o);
        if (lane >= o) end += y;
    }
    const int start = end - cnt, cells = __shfl_sync(kFull, end, 31);
    const unsigned some = __ballot_sync(kFull, cnt > 0);
    // the rows with cells, in order: first cell number | triangle, row | first column
    if (cnt > 0) spans[__popc(some & (le >> 1))] = make_uint2(start | (k << 16), row | (lo << 16));
    __syncwarp();
    for (int cb = 0; cb < cells; cb += 32) {
        // lane l's row: the last one that starts at cell cb + l or before
        const unsigned at = (unsigned)(start - cb);
        const unsigned starts = __reduce_or_sync(kFull, cnt > 0 && at < 32u ? 1u << at : 0u);
        const int earlier = __popc(__ballot_sync(kFull, cnt > 0 && start < cb));
        if (cb + lane < cells) {
            const uint2 s = spans[earlier + __popc(starts & le) - 1];
            cell((int)(s.x >> 16), (int)(s.y & 0xFFFFu), (int)(s.y >> 16) + cb + lane - (int)(s.x & 0xFFFFu));
        }
    }
    __syncwarp();  // spans[] may be rewritten
}

// Items q = aspect * n_tri + triangle, one per lane in grid-stride order
// (aspect-major: neighbouring lanes take neighbouring triangles of one
// aspect). Each lane projects its triangle and, for a range of at most
// kRasterFlat cells, writes the triangle's constants to shared memory; the
// warp then walks the rows of its 32 triangles, 32 at a time, a row per lane,
// and the cells of these rows' spans, a cell per lane (each_cell), so every
// lane works until the warp's cells run out. A triangle with a larger range is
// appended to the list `big` (warp-aggregated) for k_raster_big. Bound by
// instruction issue (66 %, 25.5 lanes; 17.5 lanes and 1.8 times the
// instructions when every cell of a box was a lane's).
__global__ void __launch_bounds__(256, 4) k_raster(const TraceArgs a, int n_tri, unsigned long long* vis, unsigned* full,
                                                   int count)
{
    extern __shared__ RasterItem s_items[];
    __shared__ int s_off[kRasterWarps][33];
    __shared__ uint2 s_span[kRasterWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    RasterItem* my = s_items + warp * 32;
    int* off = s_off[warp];
    const unsigned long long n_items = (unsigned long long)a.n_angles * (unsigned long long)n_tri;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long q0 = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    int ang = (int)(q0 / (unsigned long long)n_tri), t = (int)(q0 % (unsigned long long)n_tri);
    const int step_a = (int)(stride / (unsigned long long)n_tri), step_t = (int)(stride % (unsigned long long)n_tri);
    unsigned long long ntri = 0;
    // the rounds depend on the warp only: every lane reaches the ballots and shuffles
    for (unsigned long long base = q0 - lane; base < n_items; base += stride) {
        bool want_big = false;
        int4 rng = make_int4(0, 0, 0, 0);
        int nr = 0;  // rows of the lane's triangle
        if (base + lane < n_items) {
            const AngleDev& A = a.angles[ang];
            const float4* tp = a.tris + 3 * (size_t)t;
            const float4 P = __ldg(tp), B = __ldg(tp + 1), C = __ldg(tp + 2);
            int i0, i1, j0, j1;
            TriProj pr;
            tri_project(A, cell_scale(A), P, B, C, pr);
            if (tri_cells_p(A, pr, i0, i1, j0, j1)) {
                const long long ncell = (long long)(i1 - i0 + 1) * (j1 - j0 + 1);
                if (ncell > kRasterMaxCells || A.nu > 65535 || A.nv > 65535) {
                    atomicOr(full + ang, 1u);
                    atomicOr(full + a.n_angles, 1u);  // some aspect of the chunk traverses
                } else if (ncell > kRasterFlat) {
                    want_big = true;
                    rng = make_int4(i0, i1, j0, j1);
                } else {
                    // each group of constants goes to shared memory as soon as it is formed
                    RasterItem& it = my[lane];
                    float c2;
                    {
                        CellEdges E;
                        tri_cell_edges_p(pr, i0, i1, j0, j1, E);
                        it.e0 = make_float4(E.nx[0], E.ny[0], E.c[0], E.nx[1]);
                        it.e1 = make_float4(E.ny[1], E.c[1], E.nx[2], E.ny[2]);
                        c2 = E.c[2];
                    }
                    const RasterGrid G = raster_grid(A);
                    float bd;
                    {
                        const RasterTri R = raster_tri(G, P, B, C, i0, i1, j0, j1);
                        it.g2 = make_float4(G.dv.z, R.v0.x, R.v0.y, R.v0.z);
                        it.r0 = make_float4(R.p.x, R.p.y, R.p.z, R.p2.x);
                        it.r1 = make_float4(R.p2.y, R.p2.z, R.nn.x, R.nn.y);
                        it.r2 = make_float4(R.nn.z, R.det, R.bd, R.bU);
                        it.r3 = make_float4(R.bV, R.bT, 0.f, 0.f);
                        bd = R.bd;
                    }
                    if (bd >= 0.f) {
                        const PlaneKey K = plane_key(a.tri_nrm, t, G.d);
                        it.r3.z = K.n.x;
                        it.r3.w = K.n.y;
                        it.r4 = make_float4(K.n.z, K.dh, K.dl, K.rd);
                        it.e2 = make_float4(c2, 0.f, raster_tnear(P, B, C, G.p0, G.d, K),
                                            __int_as_float((int)a.ray_off[ang]));
                        it.g0 = make_float4(G.p0.x, G.p0.y, G.p0.z, G.du.x);
                        it.g1 = make_float4(G.du.y, G.du.z, G.dv.x, G.dv.y);
                        it.m0 = make_int4(i0, j0, i1 - i0 + 1, __float_as_int(P.w));
                        it.m1 = make_int4(ang, t, G.nbu, G.tw);
                        nr = j1 - j0 + 1;
                    }
                }
            }
        }
        append_big(a, full, want_big, t, ang, rng.x, rng.y, rng.z, rng.w);
        // inclusive scan of the rows: off[k] = first row of lane k's triangle
        int incl = nr;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += y;
        }
        off[lane + 1] = incl;
        if (lane == 0) off[0] = 0;
        __syncwarp();
        const int total = __shfl_sync(kFull, incl, 31);
        int k = 0;
        for (int rb = 0; rb < total; rb += 32) {
            int cnt = 0, lo = 0, row = 0;
            if (rb + lane < total) {
                while (off[k + 1] <= rb + lane) ++k;
                const RasterItem& it = my[k];
                const float4 e0 = it.e0, e1 = it.e1, e2 = it.e2;
                const float nx[3] = {e0.x, e0.w, e1.z}, ny[3] = {e0.y, e1.x, e1.w}, c[3] = {e0.z, e1.y, e2.x};
                row = rb + lane - off[k];
                row_span(nx, ny, c, (float)row, it.m0.z, lo, cnt);
            }
            each_cell(s_span[warp], k, row, lo, cnt, [&](int tri, int dj, int di) {
                const RasterItem& it = my[tri];
                const int4 m0 = it.m0;
                const float4 e2 = it.e2;
                const int i = m0.x + di, j = m0.y + dj;
                const int4 m1 = it.m1;
                const int tw = m1.w, sh = 5 - tw;  // tile of W = 2^tw by H = 2^sh rays
                const long long pidx = (long long)__float_as_int(e2.w) + ((long long)((j >> sh) * m1.z + (i >> tw)) << 5) +
                                       ((j & ((1 << sh) - 1)) << tw) + (i & ((1 << tw) - 1));
                // the ray's closest hit so far (keys only decrease; a stale value is larger): nearer than any
                // distance this triangle can give, the cell is decided
                if (__uint_as_float((unsigned)(__ldcg(vis + pidx) >> 32)) < e2.z) return;
                ++ntri;
                const float4 g0 = it.g0, g1 = it.g1, g2 = it.g2;
                const float fi = (float)i, fj = (float)j;
                const float3 o = make_float3(__fadd_rn(__fadd_rn(g0.x, __fmul_rn(fi, g0.w)), __fmul_rn(fj, g1.z)),
                                             __fadd_rn(__fadd_rn(g0.y, __fmul_rn(fi, g1.x)), __fmul_rn(fj, g1.w)),
                                             __fadd_rn(__fadd_rn(g0.z, __fmul_rn(fi, g1.y)), __fmul_rn(fj, g2.x)));
                const float3 v0 = make_float3(g2.y, g2.z, g2.w);
                const float3 sv = make_float3(__fsub_rn(o.x, v0.x), __fsub_rn(o.y, v0.y), __fsub_rn(o.z, v0.z));
                const float4 r0 = it.r0, r1 = it.r1, r2 = it.r2, r3 = it.r3;
                float tc, et;
                const int f = filter_core(dot_s(sv, make_float3(r0.x, r0.y, r0.z)), dot_s(sv, make_float3(r0.w, r1.x, r1.y)),
                                          dot_s(sv, make_float3(r1.z, r1.w, r2.x)), r2.y, r2.w, r3.x, r2.z, r3.y, tc, et);
                if (f == 0) return;
                if (f >= 2) {
                    const AngleDev& A = a.angles[m1.x];
                    const int r = tri_refine(a.tris, a.tri_v12, m1.y, o, make_float3(A.dir[0], A.dir[1], A.dir[2]), f, tc);
                    if (count) count_open(a.stats, r);
                    if (!(r & 1)) return;
                }
                const float4 r4 = it.r4;
                PlaneKey K;
                K.n = make_float3(r3.z, r3.w, r4.x);
                K.dh = r4.y;
                K.dl = r4.z;
                K.rd = r4.w;
                const float th = plane_key_t(K, v0, o, tc);
                if (th >= 0.f && th <= FLT_MAX)
                    atomicMin(vis + pidx, ((unsigned long long)__float_as_uint(th) << 32) | (unsigned)m0.w);
            });
        }
        __syncwarp();  // the next round rewrites my[] and off[]
        t += step_t;
        ang += step_a;
        if (t >= n_tri) {
            t -= n_tri;
            ++ang;
        }
    }
    if (count) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ntri += __shfl_xor_sync(kFull, ntri, o);
        if (lane == 0 && ntri) {
            atomicAdd(a.stats + kStatTris, ntri);
            atomicAdd(a.stats + kStatRaster, ntri);
        }
    }
}

// One (triangle, cell) pair: the traversal's test of primary ray (i, j) against triangle t, a hit's key kept. A ray
// whose hit so far is nearer than tnear (raster_tnear; kNear) needs none; returns the tests made.
template <bool kNear = false>
__device__ __forceinline__ unsigned sparse_pair(const TraceArgs& a, unsigned long long* vis, int t, int ang, int ij,
                                                int count, float tnear = 0.f)
{
    const AngleDev& A = a.angles[ang];
    const int i = ij & 0xFFFF, j = (int)((unsigned)ij >> 16);
    auto at = [&]() {
        const int tw = A.tw_log2, sh = 5 - tw;
        return a.ray_off[ang] + ((long long)((j >> sh) * A.nbu + (i >> tw)) << 5) + ((j & ((1 << sh) - 1)) << tw) +
               (i & ((1 << tw) - 1));
    };
    if (kNear && __uint_as_float((unsigned)(__ldcg(vis + at()) >> 32)) < tnear) return 0u;
    const float3 o = primary_origin(A, i, j), d = make_float3(A.dir[0], A.dir[1], A.dir[2]);
    const float4* tp = a.tris + 3 * (size_t)t;
    const float4 P = __ldg(tp), B = __ldg(tp + 1), C = __ldg(tp + 2);
    float tc, et;
    const int f = tri_filter(P, B, C, o, d, tc, et);
    if (f == 0) return 1u;
    if (f >= 2) {
        const int r = tri_refine(a.tris, a.tri_v12, t, o, d, f + 2, tc);
        if (count) count_open(a.stats, r);
        if (!(r & 1)) return 1u;
    }
    const PlaneKey K = plane_key(a.tri_nrm, t, d);
    const float th = plane_key_t(K, make_float3(P.x, P.y, P.z), o, tc);
    if (th >= 0.f && th <= FLT_MAX)
        atomicMin(vis + at(), ((unsigned long long)__float_as_uint(th) << 32) | (unsigned)__float_as_int(P.w));
    return 1u;
}

// The cells of up to 32 triangles of a sparse grid, lane l's triangle t of
// aspect ang (t < 0: none): their edges in shared memory, their rows' spans a
// row per lane, the spans' cells a cell per lane. Returns the lane's tests.
__host__ __device__ __forceinline__ unsigned sparse_list_cap(const TraceArgs& a)
{
    const long long n = a.total_rays * (long long)(sizeof(RayState) / sizeof(int2));
    return (unsigned)(n < (1ll << 30) ? n : 1ll << 30);
}
struct __align__(16) SparseItem {
    float4 e0, e1;  // the edges of RasterItem
    float c2, tnear;
    int w, ij, t, ang;
    int pad[2];
};
__device__ __forceinline__ unsigned sparse_walk(const TraceArgs& a, unsigned long long* vis, int t, int ang, uint2* spans,
                                                int count)
{
    __shared__ SparseItem s_items[kRasterWarps][32];
    __shared__ int s_off[kRasterWarps][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SparseItem* my = s_items[warp];
    int* off = s_off[warp];
    int nr = 0;
    if (t >= 0) {
        const AngleDev& A = a.angles[ang];
        const float4* tp = a.tris + 3 * (size_t)t;
        int i0, i1, j0, j1;
        TriProj pr;
        const float4 P = __ldg(tp), B = __ldg(tp + 1), C = __ldg(tp + 2);
        tri_project(A, cell_scale(A), P, B, C, pr);
        if (tri_cells_p(A, pr, i0, i1, j0, j1)) {
            const float3 d = make_float3(A.dir[0], A.dir[1], A.dir[2]);
            const PlaneKey K = plane_key(a.tri_nrm, t, d);
            CellEdges E;
            tri_cell_edges_p(pr, i0, i1, j0, j1, E);
            SparseItem& it = my[lane];
            it.e0 = make_float4(E.nx[0], E.ny[0], E.c[0], E.nx[1]);
            it.e1 = make_float4(E.ny[1], E.c[1], E.nx[2], E.ny[2]);
            it.c2 = E.c[2];
            it.tnear = raster_tnear(P, B, C, make_float3(A.p0[0], A.p0[1], A.p0[2]), d, K);
            it.w = i1 - i0 + 1;
            it.ij = i0 | (j0 << 16);
            it.t = t;
            it.ang = ang;
            nr = j1 - j0 + 1;
        }
    }
    int incl = nr;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    off[lane + 1] = incl;
    if (lane == 0) off[0] = 0;
    __syncwarp();
    const int total = __shfl_sync(kFull, incl, 31);
    unsigned n = 0;
    int k = 0;
    for (int rb = 0; rb < total; rb += 32) {
        int cnt = 0, lo = 0, row = 0;
        if (rb + lane < total) {
            while (off[k + 1] <= rb + lane) ++k;
            const SparseItem& it = my[k];
            const float4 e0 = it.e0, e1 = it.e1;
            const float nx[3] = {e0.x, e0.w, e1.z}, ny[3] = {e0.y, e1.x, e1.w}, c[3] = {e0.z, e1.y, it.c2};
            row = rb + lane - off[k];
            row_span(nx, ny, c, (float)row, it.w, lo, cnt);
        }
        each_cell(spans, k, row, lo, cnt, [&](int tri, int dj, int di) {
            const SparseItem& it = my[tri];
            n += sparse_pair<true>(a, vis, it.t, it.ang, it.ij + (di | (dj << 16)), count, it.tnear);
        });
    }
    __syncwarp();  // my[] and off[] may be rewritten
    return n;
}

// One entry of the list of large triangles by a warp: the cells of its rows'
// spans 32 at a time, their tests added to the lane's ntri.
__device__ __forceinline__ void raster_entry(const TraceArgs& a, unsigned long long* vis, int lane, unsigned it,
                                             uint2* spans, int count, unsigned long long& ntri)
{
    const int4 b = a.big[it];
    const int td = b.x, ad = b.y;
    if (a.vis_full[ad]) return;  // traverses
    const int i0 = b.z & 0xFFFF, j0 = (unsigned)b.z >> 16, w = (b.w & 0xFFFF) + 1, h = ((unsigned)b.w >> 16) + 1;
    const int i1 = i0 + w - 1, j1 = j0 + h - 1;
    const AngleDev& A = a.angles[ad];
    const RasterGrid G = raster_grid(A);
    const float4* tp = a.tris + 3 * (size_t)td;
    const float4 P = __ldg(tp), B = __ldg(tp + 1), C = __ldg(tp + 2);
    const RasterTri R = raster_tri(G, P, B, C, i0, i1, j0, j1);
    if (!(R.bd >= 0.f)) return;  // warp-uniform
    const unsigned orig = (unsigned)__float_as_int(P.w);
    unsigned long long* vrow = vis + a.ray_off[ad];
    const PlaneKey K = plane_key(a.tri_nrm, td, G.d);
    CellEdges E;
    tri_cell_edges(A, cell_scale(A), P, B, C, i0, i1, j0, j1, E);
    for (int rb = 0; rb < h; rb += 32) {
        int lo = 0, cnt = 0;
        if (rb + lane < h) row_span(E.nx, E.ny, E.c, (float)(rb + lane), w, lo, cnt);
        each_cell(spans, 0, rb + lane, lo, cnt, [&](int, int dj, int di) {
            raster_cell(G, a, R, K, td, orig, i0 + di, j0 + dj, vrow, count);
            ++ntri;
        });
    }
}

// The listed large triangles, warp w taking entries w, w + warps, ... (every
// warp has hundreds of entries, so the few very large triangles average out;
// 0.16 ms for 37 aircraft aspects at 10 GHz, 0.70 with every cell of the box a
// lane's). kSparse: and then the middling triangles that k_raster_sparse has
// listed (a.q_out), 32 at a time or as many as keep every warp busy; mostly there
// are none of either, so the grid is what stays resident (launch and return in
// 1.9 us, 4.3 with the dense grid's) and the warps take the work by a counter.
template <bool kSparse>
__global__ void __launch_bounds__(256, 3) k_raster_big(const TraceArgs a, unsigned long long* vis, int count)
{
    __shared__ uint2 s_span[8][32];
    const int lane = threadIdx.x & 31;
    uint2* spans = s_span[threadIdx.x >> 5];
    const unsigned n_big = min(a.big_ctr[0], a.big_cap);
    const unsigned nw = (gridDim.x * blockDim.x) >> 5;
    unsigned long long ntri = 0;
    if (kSparse) {
        const unsigned n = min(a.big_ctr[1], sparse_list_cap(a)), per = max(1u, min(32u, (n + nw - 1) / nw));
        const unsigned work = n_big + (n + per - 1) / per;
        const int2* list = reinterpret_cast<const int2*>(a.q_out);
        while (work > 0) {
            unsigned it = 0;
            if (lane == 0) it = atomicAdd(a.big_ctr + 2, 1u);
            it = __shfl_sync(kFull, it, 0);
            if (it >= work) break;
            if (it < n_big) {
                raster_entry(a, vis, lane, it, spans, count, ntri);
            } else {
                it = (it - n_big) * per;
                const int2 e = (unsigned)lane < per && it + lane < n ? list[it + lane] : make_int2(-1, 0);
                ntri += sparse_walk(a, vis, e.x, e.y, spans, count);
            }
        }
    } else {
        for (unsigned it = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < n_big; it += nw)
            raster_entry(a, vis, lane, it, spans, count, ntri);
    }
    if (count) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ntri += __shfl_xor_sync(kFull, ntri, o);
        if (lane == 0 && ntri) {
            atomicAdd(a.stats + kStatTris, ntri);
            atomicAdd(a.stats + kStatRaster, ntri);
        }
    }
}

// ---------------------------------------------------------------- rasterisation of sparse grids
// Where a chunk's aspects have fewer than three grid rays (padding included, on
// the mean) for two triangles (the aircraft at 1 GHz: 0.14 rays per triangle),
// most triangles cover no cell and the others one or a few: the set-up of
// k_raster for a warp walk costs more than the tests. Here a lane keeps one triangle and projects it for up to 16 aspects in
// turn (the triangle is read once for all of them, an aspect in three broadcast
// loads); the (triangle, cell) pairs of triangles of at most kSparseCells cells
// collect in a queue of the warp, and 32 of them at a time take the traversal's
// triangle test. Triangles of at most kSparseFlat cells are listed in queue 0,
// idle until the first states are written, and k_raster_big walks the rows'
// spans of 32 of them at a time (those that find no room are queued cell by
// cell); larger ones go to its list of large triangles. 6 aspects of 800 x 800
// rays over sheets whose triangles span 5 x 5 cells, beside a fine sphere, B = 2:
// 4, 16 and 64 sheets in 1.3, 2.1 and 5.0 ms, with a warp each for triangles of
// more than 16 cells 2.0, 5.8 and 15.5 (the list full from 8 sheets on). Bound by
// instruction issue: ~235 instructions per 32 (triangle, aspect) items at 1 GHz
// against ~820 of k_raster, 354 M items in 3.2 against 10.0 ms.
constexpr int kSparseCells = 16, kSparseFlat = 256, kSparseAspects = 16;

// The aspect's fields that the projection reads
struct AspectView {
    float4 a, b, c;  // (p0, nu), (hs, nv), (vs, ids)
    float m0;
};
__device__ __forceinline__ AspectView aspect_view(const AngleDev* p)
{
    static_assert(offsetof(AngleDev, r_p0) % 16 == 0 && offsetof(AngleDev, r_ids) == offsetof(AngleDev, r_p0) + 44,
                  "AspectView reads three 16-byte words");
    const float4* w = reinterpret_cast<const float4*>(p->r_p0);
    return AspectView{__ldg(w), __ldg(w + 1), __ldg(w + 2), __ldg(&p->r_m0)};
}

// The cell range of a triangle (vertices x, y, z; size L = max(|e1|_1, |e2|_1)):
// that of tri_project and tri_cells, with the two dot products of a vertex as
// one chain of packed FP32 fused multiply-adds on the scaled axes (one more
// rounding of 2^-24, far inside the margin's 2^-18 of the distance from P0) and
// the largest distance from P0 bounded by vertex 0's plus L. Conversions
// saturate, so a range beyond the grid comes out empty.
__device__ __forceinline__ bool sparse_cells(const AspectView& A, const float* x, const float* y, const float* z, float L,
                                             int& i0, int& i1, int& j0, int& j1)
{
    const float2 sx = make_float2(A.b.x, A.c.x), sy = make_float2(A.b.y, A.c.y), sz = make_float2(A.b.z, A.c.z);
    float2 uv[3];
    float mag = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float dx = x[k] - A.a.x, dy = y[k] - A.a.y, dz = z[k] - A.a.z;
        if (k == 0) mag = fmaf(fabsf(dx) + fabsf(dy) + fabsf(dz), A.c.w, L * A.c.w);
        uv[k] = fma2(make_float2(dx, dx), sx, fma2(make_float2(dy, dy), sy, make_float2(dz * sz.x, dz * sz.y)));
    }
    const float umin = fminf(fminf(uv[0].x, uv[1].x), uv[2].x), umax = fmaxf(fmaxf(uv[0].x, uv[1].x), uv[2].x);
    const float vmin = fminf(fminf(uv[0].y, uv[1].y), uv[2].y), vmax = fmaxf(fmaxf(uv[0].y, uv[1].y), uv[2].y);
    const float m = A.m0 + (umax - umin + vmax - vmin) * (1.f / 1024.f) + mag * (1.f / 262144.f);
    i0 = max(0, __float2int_ru(umin - m));
    i1 = min(__float_as_int(A.a.w) - 1, __float2int_rd(umax + m));
    j0 = max(0, __float2int_ru(vmin - m));
    j1 = min(__float_as_int(A.b.w) - 1, __float2int_rd(vmax + m));
    return i0 <= i1 && j0 <= j1;
}

// Lists triangle t of aspect ang for the lanes of m (every lane of the warp calls it, those of m learn whether there
// was room). Out of line, so that it does not burden the projection.
__device__ __noinline__ bool sparse_list(const TraceArgs& a, unsigned m, int t, int ang)
{
    const int lane = threadIdx.x & 31;
    const unsigned cap = sparse_list_cap(a);
    unsigned slot = cap;  // (a full list is left alone, so that its counter cannot wrap)
    if (lane == 0 && __ldcg(a.big_ctr + 1) < cap) slot = atomicAdd(a.big_ctr + 1, (unsigned)__popc(m));
    slot = __shfl_sync(kFull, slot, 0) + __popc(m & ((1u << lane) - 1u));
    if (!((m >> lane) & 1u) || slot >= cap) return false;
    reinterpret_cast<int2*>(a.q_out)[slot] = make_int2(t, ang);
    return true;
}

__global__ void __launch_bounds__(256, 3) k_raster_sparse(const TraceArgs a, int n_tri, int aspects, unsigned long long* vis,
                                                       unsigned* full, int count)
{
    __shared__ int s_t[kRasterWarps][64], s_a[kRasterWarps][64], s_ij[kRasterWarps][64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int *qt = s_t[warp], *qa = s_a[warp], *qij = s_ij[warp];
    const int n_blk = (n_tri + 31) >> 5;
    const long long n_items = (long long)((a.n_angles + aspects - 1) / aspects) * n_blk;
    unsigned long long ntri = 0;
    int n_wait = 0;
    for (long long item = (long long)blockIdx.x * kRasterWarps + warp; item < n_items;
         item += (long long)gridDim.x * kRasterWarps) {
        const int ang0 = (int)(item / n_blk) * aspects, t = ((int)(item % n_blk) << 5) + lane;
        const int ang1 = min(a.n_angles, ang0 + aspects);
        float x[3], y[3], z[3], L = 0.f;
        if (t < n_tri) {
            const float4* tp = a.tris + 3 * (size_t)t;
            const float4 P = __ldg(tp), B = __ldg(tp + 1), C = __ldg(tp + 2);
            x[0] = P.x, x[1] = P.x + B.x, x[2] = P.x + C.x;
            y[0] = P.y, y[1] = P.y + B.y, y[2] = P.y + C.y;
            z[0] = P.z, z[1] = P.z + B.z, z[2] = P.z + C.z;
            L = B.w * (1.f / (24.f * kU));  // bUV = 24 u L (1 + 2^-10); 0: degenerate, no hits
        }
        for (int ang = ang0; ang < ang1; ++ang) {
            int n_cell = 0, i0 = 0, i1 = 0, j0 = 0, j1 = 0;
            bool want_big = false;
            if (L > 0.f) {
                const AspectView A = aspect_view(a.angles + ang);
                if (sparse_cells(A, x, y, z, L, i0, i1, j0, j1)) {
                    const long long nc = (long long)(i1 - i0 + 1) * (j1 - j0 + 1);
                    if (nc > kRasterMaxCells || __float_as_int(A.a.w) > 65535 || __float_as_int(A.b.w) > 65535) {
                        atomicOr(full + ang, 1u);
                        atomicOr(full + a.n_angles, 1u);  // some aspect of the chunk traverses
                    } else if (nc > kSparseFlat) {
                        want_big = true;
                    } else {
                        n_cell = (int)nc;
                    }
                }
            }
            if (__any_sync(kFull, want_big)) append_some(a, full, want_big, t, ang, i0, i1, j0, j1);
            unsigned mc = __ballot_sync(kFull, n_cell > 0);
            if (!mc) continue;
            const unsigned ml = __ballot_sync(kFull, n_cell > kSparseCells);
            if (ml) {
                if (sparse_list(a, ml, t, ang)) n_cell = 0;
                mc = __ballot_sync(kFull, n_cell > 0);
            }
            // the triangle's cells row by row, one of each lane's at a time
            int ci = i0, cj = j0;
            for (; mc; mc = __ballot_sync(kFull, n_cell > 0)) {
                if (n_cell > 0) {
                    const int at = n_wait + __popc(mc & ((1u << lane) - 1u));
                    qt[at] = t;
                    qa[at] = ang;
                    qij[at] = ci | (cj << 16);
                    --n_cell;
                    if (++ci > i1) {
                        ci = i0;
                        ++cj;
                    }
                }
                n_wait += __popc(mc);
                if (n_wait < 32) continue;
                __syncwarp();
                sparse_pair(a, vis, qt[lane], qa[lane], qij[lane], count);
                n_wait -= 32;
                ntri += 1;
                __syncwarp();
                if (lane < n_wait) {  // at most 31 move to the front
                    qt[lane] = qt[lane + 32];
                    qa[lane] = qa[lane + 32];
                    qij[lane] = qij[lane + 32];
                }
                __syncwarp();
            }
        }
    }
    __syncwarp();
    if (lane < n_wait) {
        sparse_pair(a, vis, qt[lane], qa[lane], qij[lane], count);
        ntri += 1;
    }
    if (count) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ntri += __shfl_xor_sync(kFull, ntri, o);
        if (lane == 0 && ntri) {
            atomicAdd(a.stats + kStatTris, ntri);
            atomicAdd(a.stats + kStatRaster, ntri);
        }
    }
}

// contiguous tile range [t0, t1) of warp gw of nw over n_tiles tiles
__device__ __forceinline__ void warp_tiles(long long n_tiles, long long gw, long long nw, long long& t0, long long& t1)
{
    const long long per = (n_tiles + nw - 1) / nw;
    t0 = gw * per;
    t1 = t0 + per < n_tiles ? t0 + per : n_tiles;
}

// scratch of the two kernels below: the blocks' sums and, per warp, the sum of
// its block's earlier warps
__device__ __forceinline__ unsigned* slot_blocks(const TraceArgs& a) { return a.slot_scr; }
__device__ __forceinline__ unsigned* slot_warps(const TraceArgs& a) { return a.slot_scr + kSlotBlocks; }

// Valid bits of the primary rays from their keys, each warp a contiguous range
// of tiles, and the sums of the bits. Bound by the keys' 8 bytes a ray: 0.72 ms
// for the 476M rays of 37 aircraft aspects at 10 GHz, 5.3 TB/s (0.77 with cached
// loads, 0.87 with two keys a load and their bits interleaved).
__global__ void __launch_bounds__(256) k_vis_mask(const TraceArgs a)
{
    __shared__ unsigned s_w[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long t0, t1;
    warp_tiles(a.total_rays >> 5, (long long)blockIdx.x * 8 + warp, (long long)gridDim.x * 8, t0, t1);
    unsigned sum = 0;
    for (long long tb = t0; tb < t1; tb += 32) {
        unsigned mine = 0;
        const int n = (int)min(32ll, t1 - tb);
#pragma unroll 8
        for (int k = 0; k < n; ++k) {
            const unsigned m = __ballot_sync(kFull, __ldcs(a.vis + ((tb + k) << 5) + lane) != ~0ull);
            if (lane == k) mine = m;
        }
        sum += __popc(mine);
        if (lane < n) a.mask[tb + lane] = mine;
    }
    sum = __reduce_add_sync(kFull, sum);
    if (lane == 0) s_w[warp] = sum;
    __syncthreads();
    if (threadIdx.x < 8) {
        unsigned run = 0;
        for (int w = 0; w < (int)threadIdx.x; ++w) run += s_w[w];
        slot_warps(a)[blockIdx.x * 8 + threadIdx.x] = run;
        if (threadIdx.x == 7) slot_blocks(a)[blockIdx.x] = run + s_w[7];
    }
}

// Slot of every tile's first hit (k_vis_mask's ranges), the first record of
// every aspect, and with a hit list its entries (ray, aspect). Every block adds
// up the sums of the blocks before it (at most 10 loads a thread), which is less
// than a scan kernel between the two or its last block doing so (8 us). With
// k_vis_mask it replaces two scans of three kernels each, a copy and two
// kernels that read their result: 30 us of a small call.
template <bool kList>
__global__ void __launch_bounds__(256) k_vis_slots(const TraceArgs a)
{
    const int lane = threadIdx.x & 31;
    const long long gtid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long gw = gtid >> 5;
    // one primary query per grid ray of every rasterised aspect
    unsigned nq = 0;
    for (long long ang = gtid; ang < a.n_angles; ang += (long long)gridDim.x * blockDim.x)
        if (!a.vis_full[ang]) nq += (unsigned)a.angles[ang].nu * (unsigned)a.angles[ang].nv;
    // the hits of earlier blocks
    __shared__ unsigned s_sum[8];
    unsigned before = 0;
    const unsigned* bsum = slot_blocks(a);
#pragma unroll
    for (int k = 0; k < (kSlotBlocks + 255) / 256; ++k) {
        const int b = k * 256 + threadIdx.x;
        if (b < (int)blockIdx.x) before += __ldg(bsum + b);
    }
    before = __reduce_add_sync(kFull, before);
    if (lane == 0) s_sum[threadIdx.x >> 5] = before;
    __syncthreads();
    before = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) before += s_sum[w];
    auto put = [&](int ang, unsigned at) {
        a.rec_off[ang] = at;
        if (a.rec_off_host) a.rec_off_host[ang] = at;
    };
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        const unsigned total = before + bsum[blockIdx.x];
        *a.q_out_count = total;
        for (int ang = a.n_angles; ang >= 0 && a.ray_off[ang] >= a.total_rays; --ang) put(ang, total);
    }
    long long t0, t1;
    warp_tiles(a.total_rays >> 5, gw, (long long)gridDim.x * 8, t0, t1);
    if (t0 < t1) {
        unsigned run = before + slot_warps(a)[gw];
        int ang = find_angle_warp(a.ray_off, a.n_angles, t0 << 5);  // the aspect of the tile at hand
        long long next = a.ray_off[ang + 1];
        int start = ang;  // the first aspect that starts at tile t0 or later
        while (start > 0 && a.ray_off[start - 1] == (t0 << 5)) --start;
        if (a.ray_off[start] < (t0 << 5)) ++start;
        for (; t0 < t1; t0 += 32) {
            const long long t = t0 + lane;
            const unsigned m = t < t1 ? a.mask[t] : 0u, c = (unsigned)__popc(m);
            unsigned incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            const unsigned slot = run + incl - c;
            run += __shfl_sync(kFull, incl, 31);
            if (t < t1) const_cast<unsigned*>(a.tile_base)[t] = slot;
            for (; start < a.n_angles; ++start) {
                const long long ts = a.ray_off[start] >> 5;
                if (ts >= t1 || ts >= t0 + 32) break;
                if (t == ts) put(start, slot);
            }
            if (!kList) continue;
            unsigned todo = __ballot_sync(kFull, m != 0u);
            while (todo) {
                const int k = __ffs(todo) - 1;
                todo &= todo - 1u;
                const unsigned mk = __shfl_sync(kFull, m, k), sk = __shfl_sync(kFull, slot, k);
                const long long base = (t0 + k) << 5;
                while (next <= base) next = a.ray_off[++ang + 1];  // the tiles of a warp only move forward
                if ((mk >> lane) & 1u)
                    a.hit_list[sk + __popc(mk & ((1u << lane) - 1u))] = make_uint2((unsigned)(base + lane), (unsigned)ang);
            }
        }
    }
    flush_stats<false>(a, nq, 0u, 0u, false);
}

// ---------------------------------------------------------------- pass 0: primary rays
// state of a primary ray before its first hit: receive basis field, path
// term k.o0 (two-float), no bounce yet
__device__ __forceinline__ void start_ray(const AngleDev& A, Ray& r)
{
    r.ev = make_float3(A.vhat[0], A.vhat[1], A.vhat[2]);
    tf_dot(A.dir, r.o, r.lacc_hi, r.lacc_lo);
    r.cos0 = 0.f;
    r.nb = 0;
    r.last = -1;
}

template <bool kCount, int kStack, int kMode>
__global__ void __launch_bounds__(kTraceThreads, 4) k_primary(const TraceArgs a)
{
    // with rasterised hits this kernel only traverses for flagged aspects, and leaves their keys
    if (a.vis && !a.vis_full[a.n_angles]) return;
    const int lane = threadIdx.x & 31;
    unsigned nq = 0, nvis = 0, ntri = 0;
    bool ovf = false;
    while (true) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(a.work, 32ull);
        base = __shfl_sync(kFull, base, 0);
        if ((long long)base >= a.total_rays) break;
        int ang = 0;
        if (lane == 0) ang = find_angle(a.ray_off, a.n_angles, (long long)base);
        ang = __shfl_sync(kFull, ang, 0);
        if (a.vis && !a.vis_full[ang]) continue;  // warp-uniform; rasterised
        const AngleDev& A = a.angles[ang];
        const int local = (int)((long long)base + lane - a.ray_off[ang]);
        int i, j;
        tile_ij(A, local, i, j);
        bool active = i < A.nu && j < A.nv;
        if (a.cover)
            active = active && (((a.cover[base >> 5] >> lane) & 1u) || a.cover[(a.total_rays >> 5) + ang]);
        bool hit = false;
        Ray r;
        r.angle = ang;
        r.local = local;
        r.o = make_float3(0.f, 0.f, 0.f);
        r.d = make_float3(0.f, 0.f, 1.f);
        if (active) {
            r.o = primary_origin(A, i, j);
            r.d = make_float3(A.dir[0], A.dir[1], A.dir[2]);
        }
        Hit h;
        query<kCount, kStack, kMode>(a, active, r.o, r.d, -1, h, nvis, ntri, ovf);
        if (active) ++nq;
        if (a.vis) {
            const bool any = active && h.k >= 0;
            const_cast<unsigned long long*>(a.vis)[base + lane] =
                any ? ((unsigned long long)__float_as_uint(h.t) << 32) | (unsigned)h.orig : ~0ull;
            continue;
        }
        if (active) {
            if (h.k >= 0) {
                start_ray(a.angles[ang], r);
                hit = true;
                apply_hit(A, a.tri_nrm, h, a.flags, r);
                record_hit(a, r, h);
            }
        }
        const unsigned m = __ballot_sync(kFull, hit);
        if (lane == 0) a.mask[base >> 5] = m;
        push(a, hit, r);
    }
    flush_stats<kCount>(a, nq, nvis, ntri, ovf);
}

// State of rasterised primary hit (ray g of the chunk, aspect ang) after its
// first hit.
__device__ __forceinline__ void primary_state(const TraceArgs& a, unsigned g, int ang, Ray& r)
{
    const AngleDev& A = a.angles[ang];
    const int local = (int)((long long)g - a.ray_off[ang]);
    int i, j;
    tile_ij(A, local, i, j);
    const unsigned long long key = __ldcs(a.vis + g);
    Hit h;
    h.t = __uint_as_float((unsigned)(key >> 32));
    h.orig = (int)(unsigned)key;
    h.k = __ldg(a.tri_pos + h.orig);
    r.angle = ang;
    r.local = local;
    r.o = primary_origin(A, i, j);
    r.d = make_float3(A.dir[0], A.dir[1], A.dir[2]);
    start_ray(A, r);
    apply_hit(A, a.tri_nrm, h, a.flags, r);
    record_hit(a, r, h);
}

// Primary pass of the keyed rays where no hit list takes them to a bounce pass:
// each ray reads its key, and its state goes to its queue slot or, where one
// bounce is all there is (kEmit), its record is written. The tiles are assigned
// statically, in chunks interleaved over the warps (hits cluster in the grid).
template <bool kEmit>
__global__ void __launch_bounds__(kTraceThreads) k_primary_vis(const TraceArgs a)
{
    const int lane = threadIdx.x & 31;
    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                    nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const long long n_tiles = a.total_rays >> 5;
    constexpr int kChunk = 4;  // tiles
    const long long n_chunks = (n_tiles + kChunk - 1) / kChunk;
    int ang = 0;
    if (gw < n_chunks) {
        if (lane == 0) ang = find_angle(a.ray_off, a.n_angles, (gw * kChunk) << 5);
        ang = __shfl_sync(kFull, ang, 0);
    }
    for (long long chunk = gw; chunk < n_chunks; chunk += nw) {
        for (long long tile = chunk * kChunk; tile < (chunk + 1) * kChunk && tile < n_tiles; ++tile) {
            const long long base = tile << 5;
            while (a.ray_off[ang + 1] <= base) ++ang;  // the tiles of a warp only move forward
            const unsigned vmask = a.mask[tile];
            if (!((vmask >> lane) & 1u)) continue;
            Ray r;
            primary_state(a, (unsigned)(base + lane), ang, r);
            if (kEmit) emit(a, r, false);
            else store_state(a.q_out, a.tile_base[tile] + __popc(vmask & ((1u << lane) - 1u)), r);
        }
    }
}

// ---------------------------------------------------------------- pass b >= 1: live rays
// Origin, direction and triangle after the first hit of a rasterised primary
// ray (ray g of the chunk, aspect ang): the stored-state steps of apply_hit
// alone (hit point, orientation, reflection, offset origin).
__device__ __forceinline__ void primary_geom(const TraceArgs& a, unsigned g, int ang, float3& o, float3& d, int& last)
{
    const AngleDev& A = a.angles[ang];
    int i, j;
    tile_ij(A, (int)((long long)g - a.ray_off[ang]), i, j);
    const unsigned long long key = __ldcs(a.vis + g);
    const float t = __uint_as_float((unsigned)(key >> 32));
    const int k = __ldg(a.tri_pos + (int)(unsigned)key);
    const float3 o0 = primary_origin(A, i, j), d0 = make_float3(A.dir[0], A.dir[1], A.dir[2]);
    const float3 x = make_float3(__fmaf_rn(t, d0.x, o0.x), __fmaf_rn(t, d0.y, o0.y), __fmaf_rn(t, d0.z, o0.z));
    const float4 N4 = __ldg(a.tri_nrm + k);
    const float3 n = make_float3(N4.x, N4.y, N4.z);
    float dn, dnl;
    tf_dot3(d0, n, dn, dnl);
    const float3 nf = dn < 0.f ? n : make_float3(-n.x, -n.y, -n.z);
    const float m2 = -2.f * dn;
    d = make_float3(__fmaf_rn(m2, n.x, d0.x), __fmaf_rn(m2, n.y, d0.y), __fmaf_rn(m2, n.z, d0.z));
    o = make_float3(__fmaf_rn(A.eps, nf.x, x.x), __fmaf_rn(A.eps, nf.y, x.y), __fmaf_rn(A.eps, nf.z, x.z));
    last = k;
}

// the rest of a ray's visit after its closest-hit query (full state in r): its record, or its next state; true if
// it goes on
template <bool kCount, bool kBi>
__device__ __forceinline__ bool finish_query(const TraceArgs& a, const Hit& h, Ray& r, unsigned& nq, unsigned& nhit,
                                             bool& ovf)
{
    const AngleDev& A = a.angles[r.angle];
    ++nq;
    bool again = false, zero = false;
    if (h.k < 0) {
        // escaped: its last hit radiates
    } else if (r.nb >= a.max_bounces) {
        zero = true;  // still trapped after B_max: invalid
    } else {
        if (kCount) ++nhit;
        apply_hit(A, a.tri_nrm, h, a.flags, r);
        record_hit(a, r, h);
        again = r.nb < a.max_bounces || (a.flags & kFlagEscape);
    }
    if (!again) {
        if (kBi && !zero && A.bistatic) zero = !rx_visible(a, A, r, nq, ovf);
        emit(a, r, zero);
    }
    return again;
}

template <bool kCount, int kStack, int kMode, bool kBi = false, bool kList = false>
__global__ void __launch_bounds__(kTraceThreads, 4) k_bounce(const TraceArgs a)
{
    const int lane = threadIdx.x & 31;
    const unsigned n_in = *a.q_in_count;
    if (n_in <= a.tail_rays) return;  // none left, or k_tail has taken them
    unsigned nq = 0, nvis = 0, ntri = 0, nhit = 0, nlist = 0;  // hits processed, hits rebuilt (counting runs)
    unsigned long long wvis = 0;  // counting runs: 32 x the warp's largest node visit count, per query
    bool ovf = false;
    while (true) {
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(a.work, 32ull);
        base = __shfl_sync(kFull, base, 0);
        if (base >= n_in) break;
        const unsigned idx = (unsigned)base + lane;
        bool again = false;
        Ray r;
        const bool active = idx < n_in;
        r.o = make_float3(0.f, 0.f, 0.f);
        r.d = make_float3(0.f, 0.f, 1.f);
        r.last = -1;
        uint2 e = make_uint2(0u, 0u);
        unsigned src = idx;
        if (kList) {
            if (active) {
                // only the geometry during the query; the full state after it
                e = a.hit_list[idx];
                primary_geom(a, e.x, (int)e.y, r.o, r.d, r.last);
                if (kCount && !a.vis_full[e.y]) ++nlist;
            }
        } else {
            // the pass's i-th entry, in the order of q_order when the rays were grouped by place
            if (a.q_order && active) src = __ldcs(a.q_order + idx);
            if (active) load_geom(a.q_in, src, r);
        }
        Hit h;
        const unsigned nvis0 = nvis;
        query<kCount, kStack, kMode>(a, active, r.o, r.d, r.last, h, nvis, ntri, ovf);
        if (kCount) wvis += 32ull * __reduce_max_sync(kFull, nvis - nvis0);
        if (active) {
            if (kList) primary_state(a, e.x, (int)e.y, r);
            else load_payload(a.q_in, src, r);
            again = finish_query<kCount, kBi>(a, h, r, nq, nhit, ovf);
        }
        push(a, again, r);
    }
    flush_stats<kCount>(a, nq, nvis, ntri, ovf, nhit, nlist, (threadIdx.x & 31) == 0 ? wvis : 0ull);
}

// A pass over so few rays that they no longer fill the GPU (at most a.tail_rays)
// lasts as long as its slowest ray's traversal, a chain of dependent fetches and
// tests, whatever the others do: 130 to 200 us per pass for the 900 rays trapped
// in the aircraft's inlets, 95 passes of 100. Here every ray goes on through
// its remaining bounces without waiting for the others, its state kept at its
// queue slot between them; the rays are spread over all warps, so few share one.
// Up to one ray per resident thread (155,648): with more, the lanes whose rays
// have ended are worth the compaction between passes. aircraft_deep_cavity
// (3 GHz, 45 aspects, 100 bounces): 11.9 ms, 22.5 pass by pass. Rays still there after
// kHandAfter bounces are trapped: where many more may follow (a.hand_count) they
// go to k_trapped. Handed over after 6, 10, 14, 20 bounces: the 983k-triangle
// aircraft at 3 GHz, 100 bounces 10.4, 10.0, 10.1, 10.2 ms; 250k triangles 6.8,
// 6.8, 6.9, 7.0; 60k at 6 GHz, 60 bounces 4.37, 4.40, 4.45, 4.50; 983k at 1.5
// GHz, 40 bounces, no escape rule 5.92, 6.02, 6.08, 6.23 (after 4: 11.7, 8.0,
// 4.8, 6.0; never: 11.4, 7.8, 4.7, 6.4).
constexpr int kHandAfter = 10;
template <bool kCount, int kStack, int kMode, bool kBi>
__global__ void __launch_bounds__(kTraceThreads, 4) k_tail(const TraceArgs a)
{
    const int lane = threadIdx.x & 31;
    const unsigned n_in = *a.q_in_count;
    if (n_in == 0 || n_in > a.tail_rays) return;
    const unsigned warps = (gridDim.x * blockDim.x) >> 5, per = (n_in + warps - 1) / warps;
    unsigned nq = 0, nvis = 0, ntri = 0, nhit = 0;
    unsigned long long wvis = 0;
    bool ovf = false;
    RayState* q = const_cast<RayState*>(a.q_in);
    const unsigned idx = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) + (unsigned)lane * warps;
    bool active = lane < per && idx < n_in;
    const unsigned src = a.q_order && active ? __ldcs(a.q_order + idx) : idx;
    Ray r;
    r.o = make_float3(0.f, 0.f, 0.f);
    r.d = make_float3(0.f, 0.f, 1.f);
    r.last = -1;
    if (active) load_geom(q, src, r);
    int turn = 0;
    while (__any_sync(kFull, active)) {
        Hit h;
        const unsigned nvis0 = nvis;
        query<kCount, kStack, kMode>(a, active, r.o, r.d, r.last, h, nvis, ntri, ovf);
        if (kCount) wvis += 32ull * __reduce_max_sync(kFull, nvis - nvis0);
        if (active) {
            const float3 o = r.o, d = r.d;
            const int last = r.last;
            load_state(q, src, r);
            r.o = o, r.d = d, r.last = last;
            active = finish_query<kCount, kBi>(a, h, r, nq, nhit, ovf);
        }
        if (!kCount && a.hand_count && ++turn == kHandAfter) {
            const unsigned left = __ballot_sync(kFull, active);
            if (left) append(a.q_out, a.hand_count, left, r);
            break;
        }
        if (active) store_state(q, src, r);
    }
    flush_stats<kCount>(a, nq, nvis, ntri, ovf, nhit, 0u, (threadIdx.x & 31) == 0 ? wvis : 0ull);
}

// Closest hit of one ray by a whole warp (o, d, skip and the result the same in
// every lane). Up to eight 4-wide nodes are taken from a stack at a time, a lane
// per child, the nearest on top, and up to 32 triangles of the leaves reached, a
// lane each, their loads in flight together: a ray's chain of dependent fetches
// is as long as the tree is deep instead of one for every node and triangle it
// meets. Every lane keeps its own candidates and the smallest (t32, original
// triangle index) of the lanes' closest is taken at the end, while a single
// lane (consider_hit) drops a candidate whose distance interval lies beyond
// another's and compares stored distances only where the intervals overlap. The
// two agree where the interval's half-width (at least 28 u |S| / |d.n|, S from
// vertex 0 to the origin) covers the plane slack u L / |d.n| by which a stored
// distance may differ: unless the origin is within about L / 28 of vertex 0.
// There the two candidates would have to lie within that slack of each other,
// far inside the edge band. A nearly full stack is left to
// one node at a time; false where the children did not fit all the same (the
// caller's to trace). That takes more than 21 levels one below the other, each
// with four children that the ray enters, on top of some 60 boxes that wait: a
// balanced tree of that depth has 4^21 nodes, and no test reaches it.
constexpr int kCoopStack = 128, kCoopWide = 40, kCoopTris = 32 + 8 * 4 * 16;
struct CoopQueue {
    int2 node[kCoopStack];  // node, its near distance
    int tri[kCoopTris];
};
__device__ __forceinline__ bool closest_hit_coop(const TraceArgs& a, CoopQueue& q, float3 o, float3 d, int skip, Hit& h)
{
    const int l = threadIdx.x & 31, g = l >> 2, c = l & 3;
    const unsigned lt = (1u << l) - 1u;
    const float3 inv = make_float3(safe_rcp(d.x), safe_rcp(d.y), safe_rcp(d.z));
    const float3 oi = make_float3(o.x * inv.x, o.y * inv.y, o.z * inv.z);
    h.t = FLT_MAX;
    h.k = -1;
    h.orig = INT_MAX;
    h.lo = FLT_MAX;
    h.key = -1.f;
    float tmax = FLT_MAX;
    int sp = 1, tp = 0;
    bool fits = true;
    if (l == 0) q.node[0] = make_int2(0, 0);
    for (int it = 0; it < a.visit_limit && (sp > 0 || tp > 0); ++it) {
        __syncwarp();
        const int nt = min(32, tp);
        tp -= nt;
        const int n = tp > 0 ? 0 : min(sp > kCoopWide ? 1 : 8, sp);
        const int2 e = g < n ? q.node[sp - 1 - g] : make_int2(0, 0);
        const int k = l < nt ? q.tri[tp + l] : skip;
        sp -= n;
        const bool open = g < n && __int_as_float(e.y) <= tmax * kBoxGrow;
        const float* nd = reinterpret_cast<const float*>(a.nodes4 + (size_t)kNode4Float4 * e.x) + c;
        const float4* tq = a.tris + 3 * (size_t)k;
        float b[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        int ref = kEmptyRef;
        float4 A = make_float4(0.f, 0.f, 0.f, 0.f), B = A, C = A;
        if (open) {
#pragma unroll
            for (int u = 0; u < 6; ++u) b[u] = __ldg(nd + 4 * u);
            ref = __float_as_int(__ldg(nd + 24));
        }
        if (k != skip) A = __ldg(tq), B = __ldg(tq + 1), C = __ldg(tq + 2);
        const float x0 = fmaf(b[0], inv.x, -oi.x), x1 = fmaf(b[1], inv.x, -oi.x);
        const float y0 = fmaf(b[2], inv.y, -oi.y), y1 = fmaf(b[3], inv.y, -oi.y);
        const float z0 = fmaf(b[4], inv.z, -oi.z), z1 = fmaf(b[5], inv.z, -oi.z);
        const float tn = fmaxf(fmaxf(fminf(x0, x1), fminf(y0, y1)), fmaxf(fminf(z0, z1), 0.f));
        const float tf = fminf(fminf(fmaxf(x0, x1), fmaxf(y0, y1)), fminf(fmaxf(z0, z1), tmax));
        const bool in = ref != kEmptyRef && tn <= tf * kBoxGrow;
        if (k != skip) {
            float tc = 0.f, et = FLT_MAX;
            int f = tri_filter(A, B, C, o, d, tc, et);
            if (f >= 2) {
                f = tri_refine(a.tris, a.tri_v12, k, o, d, f + 2, tc) & 1;
                et = FLT_MAX;
            }
            if (f) consider_hit(tri_refs(a), k, __float_as_int(A.w), tc, et, o, d, h);
        }
        if (__any_sync(kFull, k != skip)) {
            float t = h.t;
#pragma unroll
            for (int u = 16; u > 0; u >>= 1) t = fminf(t, __shfl_xor_sync(kFull, t, u));
            tmax = t;
        }
        // inner children: those of deeper entries below, the farther of a node's below the nearer
        const unsigned mi = __ballot_sync(kFull, in && ref >= 0);
        int at = g < 7 ? __popc(mi >> (4 * g + 4)) : 0;
#pragma unroll
        for (int u = 1; u < 4; ++u) {
            const float t = __shfl_xor_sync(kFull, tn, u);
            at += ((mi >> (l ^ u)) & 1u) && (t > tn || (t == tn && (l ^ u) > l)) ? 1 : 0;
        }
        if (sp + __popc(mi) > kCoopStack) {
            fits = false;
            break;
        }
        if (in && ref >= 0) q.node[sp + at] = make_int2(ref, __float_as_int(tn));
        sp += __popc(mi);
        const int first = leaf_first(ref), cnt = in && ref < 0 ? leaf_count(ref) : 0;
        for (int u = 0;; ++u) {
            const unsigned m = __ballot_sync(kFull, u < cnt);
            if (!m) break;
            if (u < cnt) q.tri[tp + __popc(m & lt)] = first + u;
            tp += __popc(m);
        }
    }
    fits = fits && sp == 0 && tp == 0;  // (not out of iterations)
    key_closest(tri_refs(a), o, d, h);
    // the smallest (t32, index) of the ray's lanes, and whose it is
    float t = h.k >= 0 ? h.t : FLT_MAX;
    int orig = h.k >= 0 ? h.orig : INT_MAX, k = h.k;
#pragma unroll
    for (int u = 16; u > 0; u >>= 1) {
        const float ot = __shfl_xor_sync(kFull, t, u);
        const int oo = __shfl_xor_sync(kFull, orig, u), ok = __shfl_xor_sync(kFull, k, u);
        if (ok >= 0 && (k < 0 || ot < t || (ot == t && oo < orig))) {
            t = ot;
            orig = oo;
            k = ok;
        }
    }
    h.t = t;
    h.orig = orig;
    h.k = k;
    __syncwarp();
    return fits;
}

// The rays k_tail has handed over (a.q_out, *a.hand_count), each followed to its
// end by a warp: a bounce takes 18k cycles instead of the 30k of one
// lane, and no warp has several of them by chance. Its own kernel, since the
// queues' shared memory is L1 that the other traversals use (inside k_tail:
// aircraft_1ghz_cut 1.5 % slower). aircraft_deep_cavity in 10.3 ms with 32
// lanes a ray (16 lanes 10.4, 8 lanes 10.9, 11.8 left to k_tail). With more than
// two rays per warp the GPU is busy with a lane each: 40,000 rays of a bistatic
// trace with 67 bounces in 3.5 ms, 8.5 ms by whole warps.
constexpr unsigned kTrappedPerWarp = 2;
template <bool kBi>
__global__ void __launch_bounds__(kTraceThreads, 2) k_trapped(const TraceArgs a)
{
    __shared__ CoopQueue s_queue[kTraceThreads / 32];
    const unsigned n_in = *a.q_in_count, n = *a.hand_count;
    if (n_in == 0 || n_in > a.tail_rays || n == 0) return;  // k_tail has not had this pass
    const int lane = threadIdx.x & 31;
    const unsigned warps = (gridDim.x * blockDim.x) >> 5, warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    unsigned nq = 0, unused = 0;
    bool ovf = false;
    Ray r;
    r.o = make_float3(0.f, 0.f, 0.f);
    r.d = make_float3(0.f, 0.f, 1.f);
    r.last = -1;
    auto alone = [&](Hit& h) {
        closest_hit<false, 64>(a.nodes2, tri_refs(a), r.o, r.d, r.last, a.visit_limit, h, unused, unused, ovf);
        key_closest(tri_refs(a), r.o, r.d, h);
    };
    if (n > kTrappedPerWarp * warps) {
        // a ray per lane, over the blocks that are resident at once
        const unsigned w = warps / 2;
        for (unsigned idx = warp + (unsigned)lane * w; warp < w && idx < n; idx += 32u * w) {
            load_state(a.q_out, idx, r);
            bool again = true;
            while (again) {
                Hit h;
                alone(h);
                again = finish_query<false, kBi>(a, h, r, nq, unused, ovf);
            }
        }
    } else {
        for (unsigned idx = warp; idx < n; idx += warps) {
            if (lane == 0) load_state(a.q_out, idx, r);
            for (bool again = true; again;) {
                r.o = make_float3(__shfl_sync(kFull, r.o.x, 0), __shfl_sync(kFull, r.o.y, 0), __shfl_sync(kFull, r.o.z, 0));
                r.d = make_float3(__shfl_sync(kFull, r.d.x, 0), __shfl_sync(kFull, r.d.y, 0), __shfl_sync(kFull, r.d.z, 0));
                r.last = __shfl_sync(kFull, r.last, 0);
                Hit h;
                const bool fits = closest_hit_coop(a, s_queue[threadIdx.x >> 5], r.o, r.d, r.last, h);
                again = false;
                if (lane == 0) {
                    if (!fits) alone(h);
                    again = finish_query<false, kBi>(a, h, r, nq, unused, ovf);
                }
                again = __shfl_sync(kFull, (int)again, 0) != 0;
            }
        }
    }
    __syncwarp();
    flush_stats<false>(a, nq, 0u, 0u, ovf);
}

// every ray of the queue writes its record (B_max = 1 without the escape check)
template <bool kBi>
__global__ void __launch_bounds__(kTraceThreads) k_emit_all(const TraceArgs a)
{
    const unsigned n_in = *a.q_in_count;
    unsigned nq = 0;
    bool ovf = false;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n_in; i += gridDim.x * blockDim.x) {
        Ray r;
        load_state(a.q_in, i, r);
        const AngleDev& A = a.angles[r.angle];
        emit(a, r, kBi && A.bistatic && !rx_visible(a, A, r, nq, ovf));
    }
    if (nq) atomicAdd(a.stats + kStatQueries, (unsigned long long)nq);
    if (ovf) atomicAdd(a.stats + kStatOverflow, 1ull);
}

// ---------------------------------------------------------------- pooled late passes
// The live rays that a chunk's early passes leave for the next pass go to a
// pool shared by the chunks (push above), so that the late passes run once over
// the rays of every chunk: a late pass holds few rays per chunk, and a launch
// over few rays leaves most of the GPU idle while its slowest rays finish.
// k_pool_append moves rays that a chunk kept because the pool was full into the
// pool once it has been traced (their aspect index shifted by angle_shift, 0
// for rays push already gave the trace's index).
__global__ void __launch_bounds__(256) k_pool_append(const RayState* __restrict__ src, const unsigned* src_count,
                                                     RayState* __restrict__ pool, const unsigned* pool_count,
                                                     unsigned cap, int angle_shift)
{
    const unsigned n = *src_count, at = *pool_count;
    if ((unsigned long long)at + n > cap) return;  // k_pool_commit raises the flag
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float4* p = reinterpret_cast<const float4*>(src + i);
        float4* q = reinterpret_cast<float4*>(pool + at + i);
#pragma unroll
        for (int w = 0; w < 5; ++w) __stcs(q + w, __ldcs(p + w));
        int4 g = __ldcs(reinterpret_cast<const int4*>(p) + 5);
        g.x += angle_shift;
        __stcs(reinterpret_cast<int4*>(q) + 5, g);
    }
}

// Rays grouped by place before a pooled pass: the rays of one aspect that
// leave neighbouring triangles (the reordered triangles follow the tree's
// leaves) start close together, in similar directions, and share much of
// their traversal. A counting sort by bucket with atomic cursors; the order
// within a bucket varies between runs and changes no result, since every ray
// writes its record to the slot its primary ray reserved.
__device__ __forceinline__ unsigned ray_bucket(const RayState* __restrict__ q, unsigned i, int tri_shift,
                                               unsigned groups)
{
    const int4 g = __ldcs(reinterpret_cast<const int4*>(q + i) + 5);  // aspect, ray, triangle left, bounces
    return (unsigned)g.x * groups + ((unsigned)g.z >> tri_shift);
}

// Neighbouring queue entries mostly share a bucket (a warp's survivors are
// appended together), so the lanes of a warp that share one make a single
// atomic for all of them. The loops run whole warps (every lane reaches the
// match).
__global__ void __launch_bounds__(256) k_bucket_count(const RayState* __restrict__ q, const unsigned* count,
                                                      int tri_shift, unsigned groups, unsigned* counts)
{
    const unsigned n = *count;
    const int lane = threadIdx.x & 31;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned w = blockIdx.x * blockDim.x + threadIdx.x - lane; w < n; w += stride) {
        const unsigned i = w + lane;
        const unsigned b = i < n ? ray_bucket(q, i, tri_shift, groups) : 0xFFFFFFFFu;
        const unsigned peers = __match_any_sync(kFull, b);
        if (i < n && lane == __ffs(peers) - 1) atomicAdd(counts + b, (unsigned)__popc(peers));
    }
}

__global__ void __launch_bounds__(256) k_bucket_scatter(const RayState* __restrict__ q, const unsigned* count,
                                                        int tri_shift, unsigned groups, unsigned* cursor,
                                                        unsigned* order)
{
    const unsigned n = *count;
    const int lane = threadIdx.x & 31;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned w = blockIdx.x * blockDim.x + threadIdx.x - lane; w < n; w += stride) {
        const unsigned i = w + lane;
        const unsigned b = i < n ? ray_bucket(q, i, tri_shift, groups) : 0xFFFFFFFFu;
        const unsigned peers = __match_any_sync(kFull, b);
        const int leader = __ffs(peers) - 1;
        unsigned base = 0;
        if (i < n && lane == leader) base = atomicAdd(cursor + b, (unsigned)__popc(peers));
        base = __shfl_sync(kFull, base, leader);
        if (i < n) order[base + __popc(peers & ((1u << lane) - 1u))] = i;
    }
}

__global__ void k_pool_commit(const unsigned* src_count, unsigned* pool_count, unsigned cap, unsigned* flag)
{
    const unsigned n = *src_count, at = *pool_count;
    if ((unsigned long long)at + n > cap) *flag = 1u;
    else *pool_count = at + n;
}

__global__ void k_angle_offsets(const long long* ray_off, const unsigned* tile_base, const unsigned* total,
                                int n_angles, unsigned* rec_off, unsigned* rec_off_host)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n_angles) return;
    const unsigned at = i < n_angles ? tile_base[ray_off[i] >> 5] : *total;
    rec_off[i] = at;
    if (rec_off_host) rec_off_host[i] = at;
}

// The start of a chunk's trace in one launch: the aspect table and ray offsets
// from pinned host memory, the primary keys set to "none", counters and flags
// cleared. As two copies and six fills of about 3.5 us each from the first to
// the next they were 40 of the 223 us of one look at a 20k-triangle sphere.
__global__ void __launch_bounds__(256) k_trace_begin(const TraceInit b)
{
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x, n = (long long)gridDim.x * blockDim.x;
    for (long long i = tid; i < b.n_table; i += n) b.table[i] = b.table_host[i];
    for (long long i = tid; i < b.n_off; i += n) b.off[i] = b.off_host[i];
#pragma unroll
    for (int k = 0; k < TraceInit::kRanges; ++k)
        for (long long i = tid; i < b.n_zero[k]; i += n) b.zero[k][i] = 0u;
    const uint4 none = make_uint4(~0u, ~0u, ~0u, ~0u);
    for (long long i = tid; i < b.n_vis16; i += n) b.vis16[i] = none;
}

}  // namespace

int trace_blocks_per_sm()
{
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_bounce<false, 64, 0>, kTraceThreads, 0);
    return nb > 0 ? nb : 1;
}

template <int kStack, int kMode>
void launch_trace_s(const TraceArgs& a, int n_blocks, bool count_visits, cudaStream_t st)
{
    if (a.bounce == 0) {
        if (count_visits) k_primary<true, kStack, kMode><<<n_blocks, kTraceThreads, 0, st>>>(a);
        else k_primary<false, kStack, kMode><<<n_blocks, kTraceThreads, 0, st>>>(a);
        if (!a.vis) return;
        // 32 tiles a warp or more: whole steps of the slot kernel (61 requests of a small target, 200k tiles, 42 a
        // warp: 12 us for it, 17 with 10 a warp)
        const int g = (int)std::max(1ll, std::min<long long>(((a.total_rays >> 5) + 255) / 256, kSlotBlocks));
        k_vis_mask<<<g, 256, 0, st>>>(a);
        if (a.hit_list) {
            k_vis_slots<true><<<g, 256, 0, st>>>(a);
        } else {
            k_vis_slots<false><<<g, 256, 0, st>>>(a);
            if (a.emit_primary) k_primary_vis<true><<<n_blocks, kTraceThreads, 0, st>>>(a);
            else k_primary_vis<false><<<n_blocks, kTraceThreads, 0, st>>>(a);
        }
    } else if (a.bounce == 1 && a.hit_list) {
        if (count_visits) k_bounce<true, kStack, kMode, false, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
        else k_bounce<false, kStack, kMode, false, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
    } else {
        if (count_visits) k_bounce<true, kStack, kMode><<<n_blocks, kTraceThreads, 0, st>>>(a);
        else k_bounce<false, kStack, kMode><<<n_blocks, kTraceThreads, 0, st>>>(a);
    }
}

template <int kMode>
void launch_trace_m(const TraceArgs& a, int n_blocks, bool count_visits, int stack_depth, cudaStream_t st)
{
    if (stack_depth == 32) {
        launch_trace_s<32, kMode>(a, n_blocks, count_visits, st);
        return;
    }
    if constexpr (kMode != 2) {
        if (stack_depth == 128) {
            launch_trace_s<128, kMode>(a, n_blocks, count_visits, st);
            return;
        }
    }
    launch_trace_s<64, kMode>(a, n_blocks, count_visits, st);
}

template <int kMode>
void launch_tail(const TraceArgs& a, int n_blocks, bool count_visits, cudaStream_t st)
{
    if (a.bistatic) {
        if (count_visits) k_tail<true, 64, kMode, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
        else k_tail<false, 64, kMode, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
    } else {
        if (count_visits) k_tail<true, 64, kMode, false><<<n_blocks, kTraceThreads, 0, st>>>(a);
        else k_tail<false, 64, kMode, false><<<n_blocks, kTraceThreads, 0, st>>>(a);
    }
}

template <int kMode>
void launch_bistatic(const TraceArgs& a, int n_blocks, bool count_visits, cudaStream_t st)
{
    if (a.bounce == 1 && a.hit_list) {
        if (count_visits) k_bounce<true, 64, kMode, true, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
        else k_bounce<false, 64, kMode, true, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
    } else {
        if (count_visits) k_bounce<true, 64, kMode, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
        else k_bounce<false, 64, kMode, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
    }
}

unsigned trace_tail_rays(int n_blocks) { return (unsigned)n_blocks * kTraceThreads; }

cudaError_t launch_trace(const TraceArgs& a, int n_blocks, bool count_visits, int stack_depth, cudaStream_t st)
{
    if (a.bounce > 0 && a.tail_rays) {
        if (a.octant) launch_tail<3>(a, n_blocks, count_visits, st);
        else launch_tail<0>(a, n_blocks, count_visits, st);
        if (a.hand_count) {
            const int g = (n_blocks + 1) & ~1;  // half of them resident at a time
            if (a.bistatic) k_trapped<true><<<g, kTraceThreads, 0, st>>>(a);
            else k_trapped<false><<<g, kTraceThreads, 0, st>>>(a);
        }
    }
    if (a.bistatic && a.bounce > 0) {
        // bounce passes of chunks with a bistatic aspect: per-lane traversal, 64-entry stack, visibility tests
        if (a.wide) {
            if (count_visits) k_bounce<true, 64, 1, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
            else k_bounce<false, 64, 1, true><<<n_blocks, kTraceThreads, 0, st>>>(a);
        } else if (a.octant) {
            launch_bistatic<3>(a, n_blocks, count_visits, st);
        } else {
            launch_bistatic<0>(a, n_blocks, count_visits, st);
        }
        return cudaGetLastError();
    }
    if (a.wide) launch_trace_m<1>(a, n_blocks, count_visits, stack_depth, st);
    else if (a.packet) launch_trace_m<2>(a, n_blocks, count_visits, stack_depth, st);
    else if (a.octant) launch_trace_m<3>(a, n_blocks, count_visits, stack_depth, st);
    else launch_trace_m<0>(a, n_blocks, count_visits, stack_depth, st);
    return cudaGetLastError();
}

cudaError_t launch_emit_all(const TraceArgs& a, int n_blocks, cudaStream_t st)
{
    if (a.bistatic) k_emit_all<true><<<n_blocks, kTraceThreads, 0, st>>>(a);
    else k_emit_all<false><<<n_blocks, kTraceThreads, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_group_rays(const RayState* q, const unsigned* count, int tri_shift, unsigned groups,
                              unsigned* counts, long long n_buckets, unsigned* order, void* scratch, int n_blocks,
                              cudaStream_t st)
{
    k_bucket_count<<<n_blocks, 256, 0, st>>>(q, count, tri_shift, groups, counts);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = scan_exclusive_u32(counts, counts, n_buckets, false, nullptr, scratch, st);
    if (e != cudaSuccess) return e;
    k_bucket_scatter<<<n_blocks, 256, 0, st>>>(q, count, tri_shift, groups, counts, order);
    return cudaGetLastError();
}

cudaError_t launch_pool_append(const RayState* src, const unsigned* src_count, RayState* pool, unsigned* pool_count,
                               unsigned cap, int angle_shift, unsigned* flag, int n_blocks, cudaStream_t st)
{
    k_pool_append<<<n_blocks, 256, 0, st>>>(src, src_count, pool, pool_count, cap, angle_shift);
    k_pool_commit<<<1, 1, 0, st>>>(src_count, pool_count, cap, flag);
    return cudaGetLastError();
}

cudaError_t launch_silhouette(const TraceArgs& a, int n_tri, unsigned* cover, cudaStream_t st)
{
    if (a.n_angles <= 0 || n_tri <= 0) return cudaSuccess;
    const int bx = (int)std::min<long long>((n_tri + 255) / 256, 64);
    const int by = std::min(a.n_angles, 4096);
    k_silhouette<<<dim3(bx, by), 256, 0, st>>>(a.tris, n_tri, a.angles, a.ray_off, a.n_angles, a.total_rays >> 5,
                                               cover);
    return cudaGetLastError();
}

cudaError_t launch_raster(const TraceArgs& a, int n_tri, unsigned long long* vis, unsigned* full, bool count,
                          int n_blocks, cudaStream_t st)
{
    if (a.n_angles <= 0 || n_tri <= 0) return cudaErrorInvalidValue;
    cudaError_t e = cudaSuccess;
    static int smem_set[64] = {0};  // per device: k_raster's dynamic shared memory above 48 KB allowed
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!smem_set[dev]) {
        e = cudaFuncSetAttribute(k_raster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRasterSmem);
        if (e != cudaSuccess) return e;
        smem_set[dev] = 1;
    }
    const long long per_aspect = a.total_rays / a.n_angles;
    // Fewer than three rays for two triangles (primary pass of 40 aspects, sparse against k_raster, ms): 983k
    // triangles at 0.14 rays per triangle 0.48 / 1.33, 0.57: 1.06 / 1.70, 1.29: 1.99 / 2.19; 97k triangles at 0.71:
    // 0.171 / 0.218, 1.45: 0.265 / 0.267, 5.8: 1.16 / 0.52; 10k at 0.6: 0.052 / 0.056, 1.36: 0.064 / 0.060
    if (2 * per_aspect < 3ll * n_tri) {
        // as many aspects per triangle as leave every resident warp a few items
        const long long n_blk = ((long long)n_tri + 31) / 32;
        int aspects = kSparseAspects;
        auto items = [&]() { return n_blk * ((a.n_angles + aspects - 1) / aspects); };
        while (aspects > 1 && items() < 8ll * n_blocks) aspects /= 2;
        k_raster_sparse<<<(int)std::min<long long>((items() + kRasterWarps - 1) / kRasterWarps, n_blocks),
                          32 * kRasterWarps, 0, st>>>(a, n_tri, aspects, vis, full, count ? 1 : 0);
        k_raster_big<true><<<std::max(1, n_blocks * 3 / 16), 256, 0, st>>>(a, vis, count ? 1 : 0);
    } else {
        const long long need = ((long long)a.n_angles * n_tri + 255) / 256;
        k_raster<<<(int)std::max(1ll, std::min<long long>(need, n_blocks)), 32 * kRasterWarps, kRasterSmem, st>>>(
            a, n_tri, vis, full, count ? 1 : 0);
        k_raster_big<false><<<n_blocks, 256, 0, st>>>(a, vis, count ? 1 : 0);
    }
    return cudaGetLastError();
}

cudaError_t launch_trace_begin(const TraceInit& b, int n_sms, cudaStream_t st)
{
    const long long most = std::max(std::max(b.n_table, b.n_off), b.n_vis16);
    const int blocks = (int)std::max(4ll, std::min<long long>((most + 255) / 256, (long long)n_sms * 8));
    k_trace_begin<<<blocks, 256, 0, st>>>(b);
    return cudaGetLastError();
}

cudaError_t launch_angle_offsets(const long long* ray_off, const unsigned* tile_base, const unsigned* total,
                                 int n_angles, unsigned* rec_off, unsigned* rec_off_host, cudaStream_t st)
{
    k_angle_offsets<<<(n_angles + 1 + 255) / 256, 256, 0, st>>>(ray_off, tile_base, total, n_angles, rec_off,
                                                                rec_off_host);
    return cudaGetLastError();
}

}  // namespace sbr
