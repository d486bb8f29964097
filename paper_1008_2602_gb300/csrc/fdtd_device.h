// fdtd_device.h -- device arithmetic shared by the kernel files: storage
// access, curls, the UPML component updates, sources.  A value computed by
// any kernel goes through these (or forms that round alike), so every path
// gives the same bits.
#pragma once

#include <cuda_fp16.h>

#include "fdtd_internal.h"

namespace fdtd {

// ------------------------------------------------------------------ storage
template <typename T>
struct Io;
template <>
struct Io<float> {
    static __device__ __forceinline__ float ld(const float *p) { return __ldg(p); }
    static __device__ __forceinline__ float ldw(const float *p) { return *p; }
    static __device__ __forceinline__ void st(float *p, float v) { *p = v; }
};
template <>
struct Io<__half> {
    static __device__ __forceinline__ float ld(const __half *p) { return __half2float(__ldg(p)); }
    static __device__ __forceinline__ float ldw(const __half *p) { return __half2float(*p); }
    static __device__ __forceinline__ void st(__half *p, float v) { *p = __float2half_rn(v); }
};

// ------------------------------------------------------------------ arithmetic
// Eq. 8 pulse of a source at the half step n + 1/2: J for a current source,
// Vs for a voltage source.
__device__ __forceinline__ double src_pulse(const Source &S, long long step, double dt)
{
    const double t = ((double)step + 0.5) * dt;
    const double u = (t - S.t0) / S.tau;
    return S.J0 * u * exp(-u * u);
}

// A source applied to the plainly updated edge value ep (as stored), given the
// edge's previous value en (as stored); returns the new value before storage
// rounding.  Current source: E -= coef J.  Resistive voltage source: the lumped
// current (l E^{n+1/2} + Vs) / Rs in Ampere's law turns the plain update
// E_p = E^n + ce S curl into E^{n+1} = (E_p - beta E^n - gam Vs) / (1 + beta).
__device__ __forceinline__ float src_apply(const Source &S, double w, float ep, float en)
{
    if (S.kind == kSrcCurrent) return __fsub_rn(ep, (float)(S.coef * w));
    return (float)(((double)ep - S.beta * (double)en - S.gam * w) / (1.0 + S.beta));
}

// Two adjacent elements of one row (8-byte aligned for FP32, 4-byte for the
// 16-bit storage types), converted to/from FP32.
template <typename T>
struct Pair;
template <>
struct Pair<float> {
    static __device__ __forceinline__ float2 lds(const float *p) { return *reinterpret_cast<const float2 *>(p); }
    static __device__ __forceinline__ float2 ldg(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
    static __device__ __forceinline__ void st(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
};
template <>
struct Pair<__half> {
    static __device__ __forceinline__ float2 lds(const __half *p)
    {
        return __half22float2(*reinterpret_cast<const __half2 *>(p));
    }
    static __device__ __forceinline__ float2 ldg(const __half *p)
    {
        return __half22float2(__ldg(reinterpret_cast<const __half2 *>(p)));
    }
    static __device__ __forceinline__ void st(__half *p, float2 v) { *reinterpret_cast<__half2 *>(p) = __float22half2_rn(v); }
};

// h - s and one component of S * curl, Sa (a1 - a0) - Sb (b1 - b0), on a pair.
// a - b == fma(b, -1, a) (the product is exact), so each element rounds as
// the difference, one product and one fused multiply-add would.
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 curl2v(float2 a1, float2 a0, float2 b1, float2 b0, float2 Sa, float2 nSb)
{
    return __ffma2_rn(nSb, sub2(b1, b0), __fmul2_rn(Sa, sub2(a1, a0)));
}

// One row of a 1D UPML factor table through the read-only cache (the
// tables are 16-byte aligned, one Coef per position).
__device__ __forceinline__ Coef ldcoef(const Coef *p)
{
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return Coef{v.x, v.y, v.z, v.w};
}

// Factor of the image of tangential H~ across an outer wall (PMC: odd mirror,
// -1; PEC: 0).
__device__ __forceinline__ float hsign(int wall) { return wall == 1 ? -1.0f : 0.0f; }

// ------------------------------------------------------------------ quads
struct F4 {       // four neighbouring nodes of a row
    float2 a, b;
};
__device__ __forceinline__ float2 two(float x) { return make_float2(x, x); }
__device__ __forceinline__ F4 four(float x) { return F4{two(x), two(x)}; }
__device__ __forceinline__ F4 ld4(const float *p)   // 16-byte aligned
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    return F4{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ F4 ld4(const __half *p)   // 8-byte aligned
{
    const uint2 v = *reinterpret_cast<const uint2 *>(p);
    return F4{__half22float2(*reinterpret_cast<const __half2 *>(&v.x)), __half22float2(*reinterpret_cast<const __half2 *>(&v.y))};
}
__device__ __forceinline__ void st4(float *p, const F4 &v, unsigned own)
{
    if (own == 15u) {
        *reinterpret_cast<float4 *>(p) = make_float4(v.a.x, v.a.y, v.b.x, v.b.y);
    } else {
        if (own & 1u) p[0] = v.a.x;
        if (own & 2u) p[1] = v.a.y;
        if (own & 4u) p[2] = v.b.x;
        if (own & 8u) p[3] = v.b.y;
    }
}
__device__ __forceinline__ void st4(__half *p, const F4 &v, unsigned own)
{
    const __half2 a = __float22half2_rn(v.a), b = __float22half2_rn(v.b);
    if (own == 15u) {
        *reinterpret_cast<uint2 *>(p) = make_uint2(*reinterpret_cast<const unsigned *>(&a), *reinterpret_cast<const unsigned *>(&b));
    } else {
        if (own & 1u) p[0] = __low2half(a);
        if (own & 2u) p[1] = __high2half(a);
        if (own & 4u) p[2] = __low2half(b);
        if (own & 8u) p[3] = __high2half(b);
    }
}
__device__ __forceinline__ F4 neg4(const F4 &x) { return F4{make_float2(-x.a.x, -x.a.y), make_float2(-x.b.x, -x.b.y)}; }
__device__ __forceinline__ F4 mul4(const F4 &x, const F4 &y) { return F4{__fmul2_rn(x.a, y.a), __fmul2_rn(x.b, y.b)}; }
__device__ __forceinline__ F4 fma4(const F4 &x, const F4 &y, const F4 &z)
{
    return F4{__ffma2_rn(x.a, y.a, z.a), __ffma2_rn(x.b, y.b, z.b)};
}
__device__ __forceinline__ F4 sub4(const F4 &x, const F4 &y) { return F4{sub2(x.a, y.a), sub2(x.b, y.b)}; }
__device__ __forceinline__ F4 curl4(const F4 &a1, const F4 &a0, const F4 &b1, const F4 &b0, float Sa, float Sb)
{
    return F4{curl2v(a1.a, a0.a, b1.a, b0.a, two(Sa), two(-Sb)), curl2v(a1.b, a0.b, b1.b, b0.b, two(Sa), two(-Sb))};
}
__device__ __forceinline__ float get(const F4 &v, int q) { return q == 0 ? v.a.x : q == 1 ? v.a.y : q == 2 ? v.b.x : v.b.y; }
__device__ __forceinline__ void set(F4 &v, int q, float x)
{
    if (q == 0) v.a.x = x;
    else if (q == 1) v.a.y = x;
    else if (q == 2) v.b.x = x;
    else v.b.y = x;
}

// UPML factors of a quad (the same four times along y and z).
struct C4 {
    F4 b1, g, ap, am;
};
__device__ __forceinline__ C4 fac_one() { return C4{four(1.f), four(1.f), four(1.f), four(1.f)}; }

// Gedney two-step update of one H~ component of a quad (B~ recurrence along
// w+1, H~ recurrence along w+2, B~->H~ along w).  sc = S * (curl E)_w; Bo/Bn
// are the old/new auxiliaries.  No auxiliary (aux == false): c is trivial and
// at most one of a, b is graded, so their products are exact.  Same for E
// (D~ along w+1, E along w+2, D~->E along w); ce = 1/eps_r.
__device__ __forceinline__ F4 upml_h4(const F4 &h, const F4 &sc, const C4 &a, const C4 &b, const C4 &c, bool aux, const F4 &Bo,
                                      F4 &Bn)
{
    if (aux) {
        Bn = fma4(neg4(a.g), sc, mul4(a.b1, Bo));
        return fma4(b.g, fma4(c.ap, Bn, neg4(mul4(c.am, Bo))), mul4(b.b1, h));
    }
    return fma4(neg4(mul4(a.g, b.g)), sc, mul4(mul4(a.b1, b.b1), h));
}
__device__ __forceinline__ F4 upml_e4(const F4 &e, const F4 &sc, const F4 &ce, const C4 &a, const C4 &b, const C4 &c, bool aux,
                                      const F4 &Do, F4 &Dn)
{
    if (aux) {
        Dn = fma4(a.g, sc, mul4(a.b1, Do));
        return fma4(mul4(ce, b.g), fma4(c.ap, Dn, neg4(mul4(c.am, Do))), mul4(b.b1, e));
    }
    return fma4(mul4(ce, mul4(a.g, b.g)), sc, mul4(mul4(a.b1, b.b1), e));
}

// Nodes of the quad at column i below the last column n (where x-directed samples exist).
__device__ __forceinline__ unsigned below(int i, int n) { return 15u >> min(max(i + 4 - n, 0), 4); }

// Images of tangential H~ across the outer walls: a low wall mirrors the
// node's own value, a high wall its - neighbour's.
__device__ __forceinline__ void image(bool lo, bool hi, int wlo, int whi, float &p, float &m)
{
    if (hi) p = hsign(whi) * m;
    if (lo) m = hsign(wlo) * p;
}
__device__ __forceinline__ void image4(bool lo, bool hi, int wlo, int whi, F4 &p, F4 &m)
{
    image(lo, hi, wlo, whi, p.a.x, m.a.x);
    image(lo, hi, wlo, whi, p.a.y, m.a.y);
    image(lo, hi, wlo, whi, p.b.x, m.b.x);
    image(lo, hi, wlo, whi, p.b.y, m.b.y);
}

// Along x the wall falls on one node of the quad at column i (n: last column).
__device__ __forceinline__ void image_x(int i, int n, int wlo, int whi, F4 &p, F4 &m)
{
    image(i == 0, i == n, wlo, whi, p.a.x, m.a.x);
    image(false, i + 1 == n, wlo, whi, p.a.y, m.a.y);
    image(false, i + 2 == n, wlo, whi, p.b.x, m.b.x);
    image(false, i + 3 == n, wlo, whi, p.b.y, m.b.y);
}

}  // namespace fdtd
