// plic_pair.cuh -- the FP32 fast paths of the optimised and of Kawano's SZ
// solution (Sec. 2.4) and of the analytic solution (Sec. 2.3) for two cells
// at once, on the paired FP32 instructions of sm_100+ (one FFMA2/FADD2/FMUL2
// issues two FP32 operations).  Comparisons, selects and
// MUFU operations stay per component.
//
// All cases are evaluated and selected.  The optimised SZ and the analytic
// solution form the root of cases (3)/(4) from the depressed cubic
// (centre_distance) with a Newton step in both FP32 precisions; Kawano's form
// keeps its arccosine, and for the polished precision one Newton step on the
// cubic of Eq. 10 (the closed forms of cases 1, 2, 5 are accurate to a few ulp).
#pragma once
#include "plic_solvers.cuh"

namespace plic {
namespace p2 {

typedef float2 f2;

__device__ __forceinline__ f2 mk(float a) { return make_float2(a, a); }
__device__ __forceinline__ f2 add(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 mul(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ f2 sub(f2 a, f2 b) { return __ffma2_rn(b, mk(-1.0f), a); }
__device__ __forceinline__ f2 fmax0(f2 a) { return make_float2(fmaxf(a.x, 0.0f), fmaxf(a.y, 0.0f)); }

struct b2 { bool x, y; };
__device__ __forceinline__ f2 sel(b2 c, f2 a, f2 b) { return make_float2(c.x ? a.x : b.x, c.y ? a.y : b.y); }
__device__ __forceinline__ b2 lt(f2 a, f2 b) { return {a.x < b.x, a.y < b.y}; }
__device__ __forceinline__ b2 le(f2 a, f2 b) { return {a.x <= b.x, a.y <= b.y}; }

__device__ __forceinline__ f2 rsqrt(f2 a) { return make_float2(rsqrtf(a.x), rsqrtf(a.y)); }
__device__ __forceinline__ f2 rcp(f2 a) { return make_float2(rcp_approx(a.x), rcp_approx(a.y)); }

// cube root of x >= 0 as MUFU exp2(log2(x)/3): relative error below 6e-6
// even for x = 1e-30 (the MUFU log2's absolute error, times |log2 x|/3), and
// the cube root is only the case-(1) offset d1 <= n1, whose absolute error
// then stays below 2e-7 -- no Newton step.  1e-30 is added to x (its cube root,
// 1e-10, is far below the FP32 resolution of an offset), which removes the
// zero/denormal branches on the FMA pipe.
__device__ __forceinline__ f2 cbrt_(f2 x) {
    x = add(x, mk(1e-30f));
    return make_float2(Fm<float>::exp2f_approx(Fm<float>::__log2f_approx(x.x) * (1.0f / 3.0f)),
                       Fm<float>::exp2f_approx(Fm<float>::__log2f_approx(x.y) * (1.0f / 3.0f)));
}

// sqrt of x >= 0 as x rsqrt(x) with 1e-30 added (no zero branch).  The callers
// (centre_distance, sz_orig, and offset_two of the curvature step, which clamps it)
// pass the case-(2) radicand 2 n2 n3 V - n1^2/12, which is >= n1^2/4 where the result is
// used (6 n2 n3 V >= n1^2 there) and exactly 2 n2 n3 V >= 0 for n1 = 0.
__device__ __forceinline__ f2 sqrtp(f2 x) {
    x = add(x, mk(1e-30f));
    return mul(x, rsqrt(x));
}

// One Newton step on the cubic of Eq. 10 for cases (3)/(4) (d >= n2, n1 > 0),
// with g and g' multiplied through by n1 so that one reciprocal serves:
// n1 g = n1 (3 d (d - n1) + n1^2) - (d - n2)^3 - (d - n3)_+^3 - 6 n1 n2 n3 V,
// n1 g' = n1 (6 d - 3 n1) - 3 ((d - n2)^2 + (d - n3)_+^2) = 12 n1 n2 n3 x area > 0.
// V6 = 6 n1 n2 n3 V.
__device__ __forceinline__ f2 polish34(f2 d, f2 V6, f2 n1, f2 n2, f2 n3) {
    const f2 e2 = sub(d, n2), e3 = fmax0(sub(d, n3));
    const f2 e22 = mul(e2, e2), e33 = mul(e3, e3);
    const f2 cub = fma(e22, e2, mul(e33, e3));
    const f2 dd = sub(d, n1);
    f2 g = mul(n1, fma(mk(3.0f), mul(d, dd), mul(n1, n1)));
    g = sub(g, add(cub, V6));
    f2 gp = mul(n1, fma(mk(6.0f), d, mul(mk(-3.0f), n1)));
    gp = fma(mk(-3.0f), add(e22, e33), gp);
    return sub(d, mul(g, rcp(gp)));
}

// The smaller positive root w of the depressed cubic w^3 - Q w + R = 0 of cases
// (3)/(4), from nQ = -Q < 0 and R >= 0 (centre_distance below).  Viete's form is
// w = 2 t sin(asin(a)/3) with t^2 = Q/3, a = R/(2 t^3); in these cases
// a <= 0.8839, clear of the arcsine's singular end, so one odd polynomial (an
// equal-ripple fit of 2 sin(asin(a)/3) on a <= 0.886, degree 9, within 8e-5)
// stands for the arcsine, its half-angle reduction and the sine.  It is
// evaluated in x = R Q^(-3/2), the powers of 3^(1/2) in t and a folded into
// its coefficients.  One Newton step on the cubic (quadratic term: 9e-9 t) then
// makes the root as accurate as Q and R are.
__device__ __forceinline__ f2 depressed_root(f2 nQ, f2 R) {
    const f2 rq = make_float2(rsqrtf(-nQ.x), rsqrtf(-nQ.y));
    const f2 x = mul(mul(R, rq), mul(rq, rq));
    const f2 z = mul(x, x);
    f2 p = fma(mk(-704.3350219726562f), z, mk(107.44769287109375f));
    p = fma(p, z, mk(-10.902824401855469f));
    p = fma(p, z, mk(-0.8008332848548889f));
    p = fma(p, z, mk(-1.001369833946228f));
    const f2 w = mul(mul(nQ, rq), mul(x, p));
    const f2 q = fma(w, w, nQ);                                   // w^2 - Q
    const f2 f = fma(w, q, R), df = fma(add(w, w), w, q);         // 3 w^2 - Q < 0
    return sub(w, mul(f, rcp(df)));
}

// The optimised SZ and the analytic solution for two cells in the reduced
// space (n1 <= n2 <= n3, reduced volume V), as the distance s = L/2 - d of the
// plane from the cell's centre (L = n1 + n2 + n3; `half` = L/2, `twice` = 2 L:
// constants in the L1 units of SZ).  With p = n1 n2 and B = n1 + n2 - 2 n3 V,
// Eq. 10 about its inflection point is the depressed cubic w^3 - Q w + R = 0:
//   case (3), w = n1 + n2 - d: Q = 6 p,  R = 3 p B;
//   case (4), w = L/2 - d = s: Q = 3/4 (n1 (2 L - 3 n1) - (n3 - n2)^2),
//                              R = 3 p n3 (1/2 - V);
// the trigonometric roots of both solutions (Eq. 11 with Eqs. 12-22, and the
// merged arcsine of Sec. 2.4) are its smaller positive root.  The other cases
// are s = n3 (1/2 - V) (5), s = L/2 - n1/2 - (2 n2 n3 V - n1^2/12)^(1/2) (2)
// and s = L/2 - (6 p n3 V)^(1/3) (1).  Tests: (5) B <= 0; (1) or (2)
// 3 n2 (2 n1 - B) < n1^2, of these (1) where 6 n2 n3 V < n1^2; (4) where the
// case-(3) cubic is negative at d = n3 (g = n1 + n2 - n3 > 0):
// g^3 + 3 p (B - 2 g) < 0.  The tests use the B of the root, so a root is only
// taken with a <= 0.884.
__device__ __forceinline__ f2 centre_distance(f2 V, f2 n1, f2 n2, f2 n3, f2 half, f2 twice) {
    const f2 n12 = add(n1, n2), p3 = mul(mul(mk(3.0f), n1), n2);
    const f2 h = mul(n3, V), B = fma(mk(-2.0f), h, n12);
    const f2 s5 = mul(n3, sub(mk(0.5f), V));
    // cases (2) and (1)
    const f2 k = mul(n2, h), k6 = mul(mk(6.0f), k), sq1 = mul(n1, n1);
    const f2 d2 = fma(mk(0.5f), n1, sqrtp(fma(mk(2.0f), k, mul(mk(-0.083333333333333333f), sq1))));
    const f2 d12 = sel(lt(k6, sq1), cbrt_(mul(k6, n1)), d2);
    // case (3) or (4)
    const f2 g = sub(n12, n3);
    const f2 t4 = fma(mul(g, g), g, mul(p3, fma(mk(-2.0f), g, B)));
    const b2 c4 = {g.x > 0.0f && t4.x < 0.0f, g.y > 0.0f && t4.y < 0.0f};
    const f2 e = fma(n1, fma(mk(-3.0f), n1, twice), mul(sub(n3, n2), sub(n2, n3)));
    // 1e-36 keeps the reciprocal square root finite at n1 = 0 (case (2) or (5))
    const f2 nQ = sel(c4, mul(mk(-0.75f), e), fma(mk(-2.0f), p3, mk(-1e-36f)));
    const f2 w = depressed_root(nQ, mul(p3, sel(c4, s5, B)));
    f2 s = add(w, sel(c4, mk(0.0f), sub(half, n12)));
    s = sel(lt(mul(mul(mk(3.0f), n2), sub(add(n1, n1), B)), sq1), sub(half, d12), s);
    return sel(le(B, mk(0.0f)), s5, s);
}

// Kawano's Scardovelli-Zaleski solution (Sec. 2.4) for two cells, in the
// L1-normalised reduced space (m1 <= m2 <= m3, w the reduced volume), with
// the arithmetic of sz_orig_easy/sz_orig_hard<float> (plic_solvers.cuh): its
// volume thresholds Vb1 = m1^2/(6 m2 m3 + 1e-25) and Vb2 = Vb1 + (m2 -
// m1)/(2 m3), the case-(3) end Vb3 (the case-(5) threshold m12/(2 m3) when m3
// >= m1 + m2, else the volume of the plane through the vertex m3), and
// Viete's root of the monic cubic with s^2 and -q/2 multiplied out.  Every
// case is evaluated and the selects follow that implementation's order: (1),
// (2), then (5) unless its offset is 0 (that implementation then solves the
// case-(4) cubic, which gives NaN for m = (0, 0, 1), w = 0 through s^2 = -1/4),
// else (3)/(4).  With POLISH the root of cases (3)/(4) gets one Newton step;
// the closed forms are accurate as they are.
template <bool POLISH>
__device__ __forceinline__ f2 sz_orig(f2 w, f2 m1, f2 m2, f2 m3) {
    typedef Fm<float> F;
    const f2 m12 = add(m1, m2), m1m2 = mul(m1, m2);
    const f2 e3 = mul(m1m2, m3), sqm1 = mul(m1, m1);
    const f2 ir3 = rcp(m3);
    const f2 vb1 = mul(sqm1, rcp(fma(mk(6.0f), mul(m2, m3), mk(1e-25f))));
    const f2 vb2 = fma(mul(mk(0.5f), sub(m2, m1)), ir3, vb1);
    const b2 tall = {!(m3.x < m12.x), !(m3.y < m12.y)};
    const f2 vb5 = mul(mul(mk(0.5f), m12), ir3);
    const f2 d31 = sub(m3, m1), d32 = sub(m3, m2);
    const f2 cub3 = sub(mul(mul(m3, m3), m3),
                        fma(mul(d31, d31), d31, mul(mul(d32, d32), d32)));
    const f2 vb3 = sel(tall, vb5, mul(cub3, rcp(mul(mk(6.0f), e3))));
    const b2 c3 = lt(w, vb3);
    // Viete: s^2, -q/2 and the shift -a2/3 of the case
    const f2 s24 = mul(mk(0.25f), fma(m1, fma(mk(2.0f), add(m2, m3), make_float2(-m1.x, -m1.y)),
                                      make_float2(-d32.x * d32.x, -d32.y * d32.y)));
    const f2 s2 = sel(c3, add(m1m2, m1m2), s24);
    const f2 mq2 = sel(c3, mul(mul(mk(1.5f), m1m2), fma(mk(-2.0f), mul(m3, w), m12)),
                       mul(mul(mk(0.75f), e3), fma(mk(-2.0f), w, mk(1.0f))));
    const f2 shift = sel(c3, m12, mk(0.5f));
    const f2 s = make_float2(F::sqrt_(s2.x), F::sqrt_(s2.y));
    f2 r = mul(mq2, rcp(mul(s2, s)));
    r = make_float2(fminf(fmaxf(r.x, -1.0f), 1.0f), fminf(fmaxf(r.y, -1.0f), 1.0f));
    const f2 ang = mul(mk(0.33333333333333333f),
                       make_float2(F::acos_(r.x) + 12.566370614359172f, F::acos_(r.y) + 12.566370614359172f));
    f2 d = fma(add(s, s), make_float2(__cosf(ang.x), __cosf(ang.y)), shift);
    if (POLISH) d = polish34(d, mul(mul(mk(6.0f), e3), w), m1, m2, m3);
    // case (5): tall and w >= m12 / (2 m3), unless its offset is 0
    const f2 d5 = fma(m3, w, mul(mk(0.5f), m12));
    const b2 c5 = {tall.x && !(w.x < vb5.x) && d5.x != 0.0f, tall.y && !(w.y < vb5.y) && d5.y != 0.0f};
    d = sel(c5, d5, d);
    // case (2) below Vb2, case (1) below Vb1
    const f2 d2 = fma(mk(0.5f), m1, sqrtp(fma(mul(mk(2.0f), mul(m2, m3)), w,
                                              mul(mk(-0.083333333333333333f), sqm1))));
    d = sel(lt(w, vb2), d2, d);
    const f2 d1 = cbrt_(mul(mul(mk(6.0f), e3), w));
    return sel(lt(w, vb1), d1, d);
}

// Forward volume (Eq. 10) of two cells at their offsets d0, in the cell's
// L1-normalised reduced space (m1 <= m2 <= m3, m1 + m2 + m3 = 1; Eq. 10 is
// homogeneous of degree 0 in (d, n)), il = 1/L:
//   d = 1/2 - |d0|/L (clamped at 0), then case (5) (d - m12/2)/m3 for
//   d >= m1 + m2, case (1) d^3/(6 m1 m2 m3) for d < m1, else
//   (3 d (d - m1) + m1^2 - ((d - m2)_+^3 + (d - m3)_+^3)/m1) / (6 m2 m3),
// and V0 = 1 - V for d0 > 0.
__device__ __forceinline__ f2 volume_reduced(f2 d0, f2 il, f2 m1, f2 m2, f2 m3) {
    const f2 ad = make_float2(fabsf(d0.x), fabsf(d0.y));
    const f2 d = fmax0(fma(make_float2(-ad.x, -ad.y), il, mk(0.5f)));
    // reciprocals: 1/m3 (m3 >= 1/3), 1/m1 and 1/(6 m2 m3), infinite for
    // m1 = 0 / m2 = 0; 1/m1 is capped at FLT_MAX so that the case-(2) term
    // (e2 = e3 = 0 there) stays 0, and the products with an infinite factor
    // belong to cases that the selects below do not take
    const f2 m12 = add(m1, m2);
    const f2 v5 = mul(fma(mk(-0.5f), m12, d), rcp(m3));
    const f2 r1 = rcp(m1), r23 = rcp(mul(mk(6.0f), mul(m2, m3)));
    const f2 inv1 = make_float2(fminf(r1.x, 3.40282347e38f), fminf(r1.y, 3.40282347e38f));
    const f2 e2 = fmax0(sub(d, m2)), e3 = fmax0(sub(d, m3));
    const f2 cub = fma(mul(e2, e2), e2, mul(mul(e3, e3), e3));
    f2 num = fma(mul(mk(3.0f), d), sub(d, m1), mul(m1, m1));
    num = fma(make_float2(-cub.x, -cub.y), inv1, num);
    num = sel(lt(d, m1), mul(mul(mul(d, d), d), inv1), num);       // case (1)
    const f2 v = sel(le(m12, d), v5, mul(num, r23));
    return make_float2(d0.x > 0.0f ? 1.0f - v.x : v.x, d0.y > 0.0f ? 1.0f - v.y : v.y);
}

// Whole cells: two (n, V0) -> d0 in FP32 by the optimised SZ solution
// (METHOD = M_SZ_OPT, in L1 units), Kawano's SZ solution (M_SZ_ORIG, in L1
// units) or the analytic solution (M_ANALYTIC, in the unit normal's units);
// with ROUNDTRIP, also the forward volume of the returned d0 into *vrt; with
// COUNT, invalid cells are added to `bad` (one count per cell of the pair).
template <int METHOD, bool POLISH, bool ROUNDTRIP = false, bool COUNT = true>
__device__ __forceinline__ f2 offset_pair(f2 nx, f2 ny, f2 nz, f2 V0, int (&bad)[2],
                                          f2* vrt = nullptr) {
    const f2 ax = make_float2(fabsf(nx.x), fabsf(nx.y));
    const f2 ay = make_float2(fabsf(ny.x), fabsf(ny.y));
    const f2 az = make_float2(fabsf(nz.x), fabsf(nz.y));
    const f2 n1 = make_float2(fminf(fminf(ax.x, ay.x), az.x), fminf(fminf(ax.y, ay.y), az.y));
    const f2 n3 = make_float2(fmaxf(fmaxf(ax.x, ay.x), az.x), fmaxf(fmaxf(ax.y, ay.y), az.y));
    const f2 L = add(add(ax, ay), az);
    // V = min(V0, 1 - V0) equals the exact reduction of Eq. 5 on [0, 1], and is
    // negative or NaN exactly when V0 is outside [0, 1] or NaN
    const f2 W = sub(mk(1.0f), V0);
    const f2 V = make_float2(fminf(V0.x, W.x), fminf(V0.y, W.y));
    const bool okx = V.x >= 0.0f && L.x > 0.0f && L.x <= 3.0f;
    const bool oky = V.y >= 0.0f && L.y > 0.0f && L.y <= 3.0f;
    if (COUNT) {
        bad[0] += (int)!okx;
        bad[1] += (int)!oky;
    }
    const f2 il = rcp(L);
    const f2 m1 = mul(n1, il), m3 = mul(n3, il);
    const f2 m2 = fmax0(sub(mk(1.0f), add(m1, m3)));
    f2 h;
    if (METHOD == M_SZ_OPT) {
        h = mul(L, centre_distance(V, m1, m2, m3, mk(0.5f), mk(2.0f)));
    } else if (METHOD == M_SZ_ORIG) {
        h = mul(L, sub(mk(0.5f), sz_orig<POLISH>(V, m1, m2, m3)));
    } else {
        const f2 n2 = fmax0(sub(sub(L, n1), n3));
        h = centre_distance(V, n1, n2, n3, mul(mk(0.5f), L), add(L, L));
    }
    f2 r = make_float2(copysignf(h.x, V0.x - 0.5f), copysignf(h.y, V0.y - 0.5f));
    if (!okx) r.x = __int_as_float(0x7fffffff);
    if (!oky) r.y = __int_as_float(0x7fffffff);
    if (ROUNDTRIP) {
        // NaN where d0 is NaN: invalid inputs, and Kawano's NaN cells (the
        // volume's clamp of d would otherwise turn a NaN offset into a number)
        f2 v = volume_reduced(r, il, m1, m2, m3);
        if (r.x != r.x) v.x = __int_as_float(0x7fffffff);
        if (r.y != r.y) v.y = __int_as_float(0x7fffffff);
        *vrt = v;
    }
    return r;
}

}  // namespace p2
}  // namespace plic
