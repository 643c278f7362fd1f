// plic_fx.cuh -- the PLIC offset of a double cell to full double accuracy on
// the integer and FP32 pipes (the optimised SZ and the analytic solution in
// PLIC_FP64 and PLIC_FP64_REFINED).
//
// FP64 is scarce on GB300 (one FP64 operation per 72 FP32 ones), and the closed
// forms take about 58 FP64 instructions per cell.  Here the reduced problem is
// held in 64-bit fixed point (units of 2^-62), the cases are told apart from
// linear combinations of it that are exact but for truncation, an FP32 start (18
// bits) is formed for the unknown w of the case (p2::centre_distance: the depressed
// cubic of cases (3)/(4), the cube of (1), the square of (2)), and two Newton
// steps finish w: the residual once in fixed point, scaled by the exponents of the
// normal so that its derivative is at least 3 units, the second step's by the
// Taylor expansion of the polynomial about the start (exact: it is a cubic), with
// the corrections in FP32.  The offset from the cell's centre, s = L/2 - d, is
// summed in fixed point and rounded once: |d0 error| <= 5.9e-17 on 10^7 cells
// against quadruple precision, where the closed forms reach 6e-16 (and the
// double-float steps of the other refined methods 1.1e-14).
//
// Cells outside the scheme's range (a normal far from unit length, 0 < V0 or
// 1 - V0 below 2^-96, invalid input) and those whose steps do not come out as
// small as they must (none met in those 10^7) are refused, and the caller solves
// them in FP64.  Nothing here needs the GPU: with FX_HOST defined and the few
// primitives below supplied, the functions compile for the host.
#pragma once
#include <stdint.h>

#ifndef FX_HOST
#include "plic_solvers.cuh"
#define FX_D __device__ __forceinline__
namespace plic {
namespace fx {
typedef unsigned long long u64;
typedef long long i64;
FX_D u64 mulhi(u64 a, u64 b) { return __umul64hi(a, b); }
// shifts by any non-negative count (0 from 64 on)
FX_D u64 shr(u64 x, int s) { u64 r; asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s)); return r; }
FX_D u64 shl(u64 x, int s) { u64 r; asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s)); return r; }
FX_D int clz(u64 x) { return __clzll((long long)x); }
FX_D float asf(uint32_t u) { return __uint_as_float(u); }
FX_D uint32_t asu(float f) { return __float_as_uint(f); }
FX_D float rsq(float x) { return rsqrtf(x); }
FX_D float rcp(float x) { return rcp_approx(x); }
FX_D float cbrt_start(float x) { return Fm<float>::exp2f_approx(Fm<float>::__log2f_approx(x) * (1.0f / 3.0f)); }
FX_D int rint_sat(float x) { return __float2int_rn(x); }
#endif

// A 64-bit count as a float (2 conversions; exact to 24 bits)
FX_D float tof(u64 x) { return fmaf((float)(uint32_t)(x >> 32), 4294967296.0f, (float)(uint32_t)x); }
FX_D float exp2i(int e) { return asf((uint32_t)(e + 127) << 23); }
// three quarters
FX_D u64 q3(u64 x) { return x - (x >> 2); }
// floor(x m / 2^24) for m < 2^24
FX_D u64 mul24(u64 x, uint32_t m) {
    return (((x >> 32) * m) << 8) + (((x & 0xffffffffull) * m) >> 24);
}

constexpr u64 TOP = 0x8000000000000000ull, ABS = ~TOP, HALF = 0x3fe0000000000000ull, ONE = 0x3ff0000000000000ull;

// |n| in ascending order, by the high words: components within 2^-20 of each
// other may stay exchanged, which moves d0 by less than 2^-60 (the polynomials of
// the cases that meet there differ by the cube of that distance).
FX_D void sort(u64& b1, u64& b2, u64& b3) {
    u64 t;
    bool c = (uint32_t)(b1 >> 32) > (uint32_t)(b2 >> 32);
    t = c ? b2 : b1; b2 = c ? b1 : b2; b1 = t;
    c = (uint32_t)(b2 >> 32) > (uint32_t)(b3 >> 32);
    t = c ? b3 : b2; b3 = c ? b2 : b3; b2 = t;
    c = (uint32_t)(b1 >> 32) > (uint32_t)(b2 >> 32);
    t = c ? b2 : b1; b2 = c ? b1 : b2; b1 = t;
}

// Whether the scheme takes the cell (sorted |n|, V0's bits): n3 in [1/2, 1 +
// 2^-20) and n1 < 3/4 (then L < 3), and V0 = 0 or in [2^-96, 1].
FX_D bool in_range(u64 b1, u64 b3, u64 v0) {
    const uint32_t h1 = (uint32_t)(b1 >> 32), h3 = (uint32_t)(b3 >> 32);
    const u64 va = v0 & ABS;
    return h3 - 0x3fe00000u <= 0x00100000u && h1 < 0x3fe80000u && va <= ONE &&
           (va == 0ull || ((uint32_t)(va >> 32) >= (927u << 20) && (v0 >> 63) == 0ull));
}

constexpr float U62 = 2.168404344971009e-19f;        // 2^-62

// A component's bits as n = M 2^(e - 64) with the leading bit of M set (M = 0
// below 2^-61), and as a float (truncated to 24 bits).
FX_D bool tiny(u64 b) { return (uint32_t)(b >> 32) < (962u << 20); }
FX_D u64 mantissa(u64 b) { return tiny(b) ? 0ull : (b << 11) | TOP; }
FX_D int exponent(u64 b) { return (int)(b >> 52) - 1022; }
FX_D float flt(u64 b) { return tiny(b) ? 0.0f : asf((uint32_t)(b >> 29) + 0x40000000u); }

// What the root of a case needs: n1 and n2 (bits), and in units of 2^-62
//   (1), (2): n3 V = a 2^(ex - 64) (a normalised to 2 bits), s0 = L/2 or (n2 + n3)/2;
//   (3): a = B = n1 + n2 - 2 n3 V, s0 = (n3 - n1 - n2)/2;
//   (4): a = S5 = n3 (1/2 - V), s0 = n3.
struct Task {
    u64 b1, b2, a, s0;
    int ex;
};

// The reduced problem of a cell (sorted |n|, |V0|): its case, 5 (then s is the
// answer: n3 (1/2 - V), or L/2 for V = 0) or 1 to 4 (then t is filled).  Lengths
// in units of 2^-62; V = min(V0, 1 - V0) = Mv 2^(ev - 64).
FX_D int classify(u64 b1, u64 b2, u64 b3, u64 va, Task& t, u64& s) {
    const u64 M3 = (b3 << 11) | TOP;
    const int e3 = exponent(b3);
    const u64 N1 = shr(mantissa(b1), 2 - exponent(b1)), N2 = shr(mantissa(b2), 2 - exponent(b2)),
              N3 = shr(M3, 2 - e3);
    const bool upper = va > HALF, zero = va == 0ull || va == ONE;
    const u64 Mx = (va << 11) | TOP;
    const int x = exponent(va);
    u64 Vf = upper ? 0ull - Mx : shr(Mx, -x);        // V in units of 2^-64 (1 - V0 exactly)
    if (zero) Vf = 0ull;
    const u64 H = mulhi(N3, Vf), S5 = (N3 >> 1) - H, N12 = N1 + N2;
    const i64 B = (i64)(N12 - (H << 1));
    s = zero ? (N12 + N3) >> 1 : S5;
    if (zero || B <= 0) return 5;
    const int lz = clz(Vf | 1ull);
    const u64 Mv = upper ? shl(Vf, lz) : Mx;
    const int ev = upper ? -lz : x;
    const float f1 = flt(b1), f2 = flt(b2), f3 = flt(b3);
    const float fB = tof((u64)B) * U62, sq1 = f1 * f1;
    t.b1 = b1;
    t.b2 = b2;
    t.ex = e3 + ev;
    if (3.0f * f2 * fmaf(2.0f, f1, -fB) < sq1) {
        const float v48 = asf(((uint32_t)(Mv >> 40) & 0x7fffffu) | ((uint32_t)(ev + 174) << 23));  // V 2^48
        const bool c1 = 6.0f * f2 * (f3 * v48) < sq1 * 2.81474976710656e14f;                       // 2^48
        t.a = mulhi(M3, Mv);
        t.s0 = (c1 ? N12 + N3 : N2 + N3) >> 1;
        return c1 ? 1 : 2;
    }
    const i64 G = (i64)(N12 - N3);
    const float g = G > 0 ? tof((u64)G) * U62 : 0.0f;
    const bool c4 = G > 0 && fmaf(g * g, g, 3.0f * f1 * f2 * fmaf(-2.0f, g, fB)) < 0.0f;
    t.a = c4 ? S5 : (u64)B;
    t.s0 = c4 ? N3 : (u64)((i64)(N3 - N12) >> 1);
    return c4 ? 4 : 3;
}

// n3 V 2^48 of a task of case (1) or (2)
FX_D float h48(const Task& t) { return (float)(uint32_t)(t.a >> 32) * exp2i(t.ex + 16); }

// The two Newton steps from w = m 2^(j - 24): residual F, derivative P (units
// of 2^-58, scaled alike), the polynomial's second and third Taylor coefficients
// (scaled alike); wt: w in units of 2^-62.
FX_D bool finish_root(uint32_t m, int j, i64 F, i64 P, float quad, float cubic, u64& wt) {
    const float Pf = (float)(int)(P >> 32) * -1.4901161193847656e-08f;           // -P, 2^32 - 58
    const float Ff = F < 0 ? -tof((u64)-F) : tof((u64)F);
    // the first correction in units of 2^-44
    const float t1 = Ff * rcp(Pf) * 6.103515625e-05f;                            // 2^44 - 58
    bool ok = fabsf(t1) < 1.073741824e9f;                                        // 2^30: below 2^-14
    const int D1 = rint_sat(t1);
    const uint32_t aD = (uint32_t)(D1 < 0 ? -D1 : D1);
    const u64 aP = (u64)(P < 0 ? -P : P);
    const i64 lin = (i64)((((aP >> 32) * aD) + (((aP & 0xffffffffull) * aD) >> 32)) >> 12);
    const float d = (float)D1 * 5.684341886080802e-14f;                          // 2^-44
    const float tay = fmaf(cubic, d, quad) * (d * d) * 2.8823037615171174e17f;   // 2^58
    const float P2 = fmaf(fmaf(-3.0f * cubic, d, -2.0f * quad), d, Pf);          // -P there
    const i64 F2 = F + ((P < 0) == (D1 < 0) ? lin : -lin) + (i64)rint_sat(tay);
    ok = ok && F2 == (i64)(int)F2;
    const float t2 = (float)(int)F2 * rcp(P2) * 16.0f;                           // 2^62 - 58
    ok = ok && fabsf(t2) < 1.073741824e9f;
    wt = shr((u64)m << 40, 2 - j) + (u64)((i64)D1 << 18) + (u64)(i64)rint_sat(t2);
    return ok;
}

// The start as m 2^(j - 24); false where w is below 2^-57 and counts as 0.
FX_D bool split(float w, uint32_t& m, int& j) {
    w = w < 0.999f ? w : 0.999f;
    m = (asu(w) & 0x7fffffu) | 0x800000u;
    j = (int)(asu(w) >> 23) - 126;
    return w >= 6.938893903907228e-18f;
}

// Case (2): w^2 = 2 n2 n3 V - n1^2/12, s = (n2 + n3)/2 - w.  The residual
// 12 w^2 - 24 n2 n3 V + n1^2 scaled by 2^-j.
FX_D bool root_square(const Task& c, u64& s) {
    const float f1 = flt(c.b1);
    const float t = fmaf(7.105427357601002e-15f * flt(c.b2), h48(c), f1 * f1 * -0.083333333333f);  // 2^-47
    s = c.s0;
    uint32_t m;
    int j;
    if (!split(t * rsq(t), m, j)) return true;
    const u64 m2 = (u64)m * m, M1 = mantissa(c.b1);
    const u64 T = shr((m2 * 12ull) << 12, 4 - j) -
                  shr(q3(mulhi(mantissa(c.b2), c.a)), j - (exponent(c.b2) + c.ex) + 3) +
                  shr(mulhi(M1, M1), j - 2 * exponent(c.b1) + 8);
    u64 wt;
    const bool ok = finish_root(m, j, (i64)(T << 2), (i64)((u64)m * (24ull << 34)), 12.0f * exp2i(-j), 0.0f, wt);
    s -= wt;
    return ok;
}

// Cases (3), (4): w^3 - Q w + R = 0 (p2::centre_distance), s = (n3 - n1 - n2)/2 +
// w or w; case (1): w^3 = 6 n1 n2 n3 V, s = L/2 - w.  The residual 4 w^3 - 4 Q w
// + 4 R scaled by 2^-(e1 + e2), or 4 w^3 - 24 n1 n2 n3 V by 2^-2j.
FX_D bool root_cubic(const Task& c, int code, u64& s) {
    const float f1 = flt(c.b1), f2 = flt(c.b2);
    const bool c1 = code == 1, c4 = code == 4;
    float w;
    if (c1) {
        w = cbrt_start(6.0f * f1 * (f2 * h48(c))) * 1.52587890625e-5f;           // 2^-16
    } else {
        const float p3 = 3.0f * f1 * f2;
        float Q = 2.0f * p3;
        if (c4) {
            const float f3 = (float)(uint32_t)(c.s0 >> 32) * 9.31322574615478515625e-10f, d = f3 - f2;  // 2^-30
            Q = 0.75f * fmaf(f1, fmaf(2.0f, f2 + f3, -f1), -d * d);
        }
        const float rq = rsq(Q), x = (p3 * rq) * (tof(c.a) * U62 * rq) * rq, z = x * x;
        // 2 sin(asin(a)/3) as in p2::depressed_root, here to 5e-6 of itself
        float p = fmaf(483863.59375f, z, -151864.34375f);
        p = fmaf(p, z, 20440.373046875f);
        p = fmaf(p, z, -1284.3223876953125f);
        p = fmaf(p, z, 58.092891693115234f);
        p = fmaf(p, z, 2.2411532402038574f);
        p = fmaf(p, z, 1.004689335823059f);
        p = fmaf(p, z, 0.9999952912330627f);
        w = Q * rq * (x * p);
    }
    s = c4 ? 0ull : c.s0;
    uint32_t m;
    int j;
    if (!split(w, m, j)) return true;
    const int e1 = exponent(c.b1), e2 = exponent(c.b2), sc = c1 ? 2 * j : e1 + e2;
    const u64 M1 = mantissa(c.b1), M2 = mantissa(c.b2);
    const u64 m2 = (u64)m * m, P12 = mulhi(M1, M2), X = q3(mulhi(P12, c.a));
    u64 q = c1 ? 0ull : P12 >> 1;
    if (c4) {
        const u64 N1 = shr(M1, 2 - e1), N2 = shr(M2, 2 - e2), N3 = c.s0, D = N3 > N2 ? N3 - N2 : N2 - N3;
        q = shr(mulhi(M1, ((N2 + N3) << 1) - N1), 2 + e2) - shl(mulhi(D, shl(D, -e1)), -e2);
    }
    const u64 R = c1 ? 0ull - shr(X, 1 + 2 * j - (e1 + e2 + c.ex)) : X;
    const u64 w3 = (((m2 >> 24) * m) << 16) + (((m2 & 0xffffffull) * m) >> 8);
    const i64 F = (i64)(shr(w3, 4 + sc - 3 * j) - shr(q3(mul24(q, m)), -j) + R);
    const i64 P = (i64)(shr(q3(m2 << 16), 2 + sc - 2 * j) - q3(q));
    const float es = exp2i(-sc);
    u64 wt;
    const bool ok = finish_root(m, j, F, P, 12.0f * w * es, 4.0f * es, wt);
    s = c1 ? s - wt : s + wt;
    return ok;
}

// s 2^-62 as a double (bits), rounded to nearest, negative for V0 < 1/2.
FX_D u64 round_s(u64 s, bool negative) {
    if ((i64)s < 0) s = 0ull;
    const int ls = clz(s | 1ull);
    const u64 n = shl(s, ls);
    const u64 d0 = s == 0ull ? 0ull : ((u64)(uint32_t)(1023 - ls) << 52) + (n >> 11) + ((n >> 10) & 1ull);
    return negative ? d0 | TOP : d0;
}

// The offset d0 (as bits) of a cell given as bits; false: not settled here.
FX_D bool offset(u64 nx, u64 ny, u64 nz, u64 v0, u64& d0) {
    u64 b1 = nx & ABS, b2 = ny & ABS, b3 = nz & ABS, s;
    const u64 va = v0 & ABS;
    sort(b1, b2, b3);
    if (!in_range(b1, b3, v0)) return false;
    Task t;
    const int code = classify(b1, b2, b3, va, t, s);
    const bool ok = code == 5 ? true : code == 2 ? root_square(t, s) : root_cubic(t, code, s);
    d0 = round_s(s, va < HALF);
    return ok;
}

#ifndef FX_HOST
}  // namespace fx
}  // namespace plic
#endif
