// plic_fx.cuh -- the PLIC offset of a double cell to full double accuracy, its
// root on the integer and FP32 pipes (the optimised SZ and the analytic solution
// in PLIC_FP64 and PLIC_FP64_REFINED).
//
// FP64 is scarce on GB300 (one FP64 operation per 72 FP32 ones), and the closed
// forms take about 58 FP64 instructions per cell.  Here six FP64 operations set the
// reduced problem up (classify), an FP32 start (18 bits) is formed for the unknown w
// of the case (p2::centre_distance: the depressed cubic of cases (3)/(4), the cube
// of (1), the square of (2)), and two Newton steps finish w: the residual once
// in 64-bit fixed point, scaled by the exponents of the normal so that its
// derivative is at least 3 units, the second step's by the Taylor expansion of the
// polynomial about the start (exact: it is a cubic), with the corrections in
// FP32.  The offset from the cell's centre, s = L/2 - d, is summed in units of
// 2^-62 and rounded once.  |d0 error| <= 1.8e-16 on 10^7 cells against quadruple
// precision (rms 2.9e-17; the rounding of s, and of n1 + n2 and y in classify),
// where the closed forms reach 8e-16 and the double-float steps of the other refined
// methods 1.1e-14.  With the set-up in fixed point as well the error was 5.9e-17, but
// the kernel 359 instead of 285 us.
//
// The scheme takes normals with n3 in [1/2, 1 + 2^-20) and n1 < 3/4 as they are (all of
// unit length; nothing in it assumes that), others times a power of two (rescale): the
// offset is homogeneous in the normal, and the errors above then scale with it.
// Cells with 0 < V0 or 1 - V0 below 2^-96, with L > 3 or n3 below 2^-60, invalid input and
// those whose steps do not come out as small as they must (none met in those 10^7) are
// refused, and the caller solves them in FP64.  Nothing here needs the GPU: with FX_HOST defined and the few
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
FX_D double asd(u64 u) { return __longlong_as_double((long long)u); }
FX_D u64 bits(double d) { return (u64)__double_as_longlong(d); }
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

// Whether the scheme takes the cell as it is (sorted |n|, V0's bits): n3 in [1/2, 1 +
// 2^-20) and n1 < 3/4 (then L < 3), and V0 = 0, in [2^-96, 1) or 1.
FX_D bool volume_in_range(u64 v0) {
    const uint32_t hv = (uint32_t)(v0 >> 32);
    return hv - (927u << 20) < 0x3ff00000u - (927u << 20) || (v0 & ABS) == 0ull || v0 == ONE;
}
FX_D bool in_range(u64 b1, u64 b3, u64 v0) {
    const uint32_t h1 = (uint32_t)(b1 >> 32), h3 = (uint32_t)(b3 >> 32);
    return h3 - 0x3fe00000u <= 0x00100000u && h1 < 0x3fe80000u && volume_in_range(v0);
}

// b 2^k for the bits of a non-negative double (0 below the normal range).
FX_D u64 times2(u64 b, int k) {
    const int e = (int)(b >> 52);
    return e > 0 && e + k > 0 ? b + ((u64)(i64)k << 52) : 0ull;
}

// A normal outside the range brought into it by a power of two, exactly: n3 to [1/2,
// 1), halved once more where n1 then is 3/4 or more (L up to 3) or n2 31/32 or more (case
// (2) with w near 1).  k: its exponent (|k| < 64), by which d0 is to be divided; false
// where L > 3 (a little less: the closed forms decide) or n3 < 2^-60.
FX_D bool rescale(u64& b1, u64& b2, u64& b3, int& k) {
    const uint32_t h3 = (uint32_t)(b3 >> 32);
    if (h3 - (963u << 20) >= (62u << 20)) return false;
    k = 1022 - (int)(h3 >> 20);
    if (k < 0 && asd(b1) + asd(b2) + asd(b3) > 2.99999999) return false;
    k -= (uint32_t)(times2(b1, k) >> 32) >= 0x3fe80000u || (uint32_t)(times2(b2, k) >> 32) >= 0x3fef0000u;
    b1 = times2(b1, k);
    b2 = times2(b2, k);
    b3 = times2(b3, k);
    return true;
}
// d0 of the cell itself, from that of the scaled one (bits, any sign).
FX_D u64 unscale(u64 d0, int k) { return (d0 & ABS) == 0ull ? d0 : d0 - ((u64)(i64)k << 52); }

// A non-negative double's bits as M 2^(e - 64) with the leading bit of M set (M =
// 0 below 2^-61), and in units of 2^-62 (truncated).
FX_D u64 mantissa(u64 b) { return (uint32_t)(b >> 32) < (962u << 20) ? 0ull : (b << 11) | TOP; }
FX_D int exponent(u64 b) { return (int)(b >> 52) - 1022; }
FX_D u64 fixed(u64 b) { return shr((b << 11) | TOP, 2 - exponent(b)); }
// A double's magnitude as a float, truncated to 24 bits; 0 (a denormal) below 2^-127.  The
// conversion instruction runs on the FP64 pipe: 572 us with it where these three
// integer instructions take 396 (2^24 cells, at an earlier stage).
FX_D float flt(u64 b) {
    int t = (int)((uint32_t)(b >> 32) & 0x7fffffffu) - 0x38000000;
    t = t > 0 ? t : 0;
    return asf(((uint32_t)t << 3) | ((uint32_t)b >> 29));
}

// What the root of a case needs, as doubles' bits: n1, n2, and
//   (1): a = n3 V,             y = n1 + n2 + n3      (s = y/2 - w);
//   (2): a = n3 V,             y = n2 + n3           (s = y/2 - w);
//   (3): a = n1 + n2 - 2 n3 V, y = n3 - n1 - n2      (s = y/2 + w);
//   (4): a = n3 (1/2 - V),     y = n3 - n1 - n2      (s = w).
struct Task {
    u64 b1, b2, a, y;
};

// The case of a cell (sorted |n|, |V0|): 5, with s = n3 (1/2 - V) as a double's
// bits, or 1 to 4, with t filled.  Six FP64 operations, the tests of
// p2::centre_distance on floats.  B = n1 + n2 - 2 n3 V carries the rounding of n1 +
// n2 (y too, with half the opposite effect on s); the tests stay sound however small
// n1 is, since the cases meet to the third order and the test of cases (1)/(2) uses
// the B of the root.
FX_D int classify(u64 b1, u64 b2, u64 b3, u64 va, Task& t, u64& s) {
    const double n1 = asd(b1), n2 = asd(b2), n3 = asd(b3);
    const double V = va > HALF ? 1.0 - asd(va) : asd(va);
    const double h = n3 * V, n12 = n1 + n2;
    const double B = fma(n3, asd(bits(V) + 0x8010000000000000ull), n12);         // - 2 V (V = 0: -2^-1022)
    const double S5 = fma(-n3, V, asd(b3 - 0x0010000000000000ull));
    s = bits(S5);
    if ((i64)bits(B) <= 0) return 5;
    const float f1 = flt(b1), f2 = flt(b2), fB = flt(bits(B)), sq1 = f1 * f1;
    const bool c12 = 3.0f * f2 * fmaf(2.0f, f1, -fB) < sq1;
    const bool c1 = c12 && 6.0f * f2 * flt(bits(h)) < sq1;
    const double y = n3 + asd(c12 ? (c1 ? bits(n12) : b2) : bits(n12) ^ TOP);    // (selected before the one addition)
    const float g = flt(bits(y));                    // n1 + n2 - n3, where y < 0
    const bool c4 = !c12 && (i64)bits(y) < 0 && fmaf(g * g, g, 3.0f * f1 * f2 * fmaf(-2.0f, g, fB)) < 0.0f;
    t.b1 = b1;
    t.b2 = b2;
    t.a = bits(c12 ? h : c4 ? S5 : B);
    t.y = bits(y);
    return c12 ? (c1 ? 1 : 2) : c4 ? 4 : 3;
}

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
    const bool some = w >= 6.938893903907228e-18f;
    w = w < 0.999f ? w : 0.999f;
    m = (asu(w) & 0x7fffffu) | 0x800000u;
    j = (int)(asu(w) >> 23) - 126;
    return some;
}

// Case (2): w^2 = 2 n2 n3 V - n1^2/12.  The residual 12 w^2 - 24 n2 n3 V + n1^2
// scaled by 2^-j.
FX_D bool root_square(const Task& c, u64& s) {
    const float f1 = flt(c.b1);
    const float t = fmaf(2.0f * flt(c.b2), flt(c.a), f1 * f1 * -0.083333333333f);
    s = fixed(c.y) >> 1;
    uint32_t m;
    int j;
    if (!split(t * rsq(fmaxf(t, 1e-37f)), m, j)) return true;
    const u64 m2 = (u64)m * m, M1 = mantissa(c.b1);
    const u64 T = shr((m2 * 12ull) << 12, 4 - j) -
                  shr(q3(mulhi(mantissa(c.b2), ((c.a << 11) | TOP))), j - (exponent(c.b2) + exponent(c.a)) + 3) +
                  shr(mulhi(M1, M1), j - 2 * exponent(c.b1) + 8);
    u64 wt;
    const bool ok = finish_root(m, j, (i64)(T << 2), (i64)((u64)m * (24ull << 34)), 12.0f * exp2i(-j), 0.0f, wt);
    s -= wt;
    return ok;
}

// Cases (3), (4): w^3 - Q w + R = 0 (p2::centre_distance); case (1): w^3 =
// 6 n1 n2 n3 V.  The residual 4 w^3 - 4 Q w + 4 R scaled by 2^-(e1 + e2), or
// 4 w^3 - 24 n1 n2 n3 V by 2^-2j.  c1, c4: case (1), (4); with them known at compile time the
// selections fold away.
FX_D bool root_cubic(const Task& c, bool c1, bool c4, u64& s) {
    const float f1 = flt(c.b1), f2 = flt(c.b2), fa = flt(c.a);
    const int e1 = exponent(c.b1), e2 = exponent(c.b2), ea = exponent(c.a);
    const u64 M1 = mantissa(c.b1), M2 = mantissa(c.b2);
    const i64 yh = (i64)(fixed(c.y & ABS) >> 1), Y = c.y >> 63 ? -yh : yh;       // y/2
    // (case 4)
    const u64 N1 = shr(M1, 2 - e1), N2 = shr(M2, 2 - e2), N3 = N1 + N2 + (u64)(2 * Y);
    const u64 D = N3 > N2 ? N3 - N2 : N2 - N3;
    float w;
    if (c1) {
        w = cbrt_start(6.0f * f1 * (f2 * (fa * 2.81474976710656e14f))) * 1.52587890625e-5f;  // 2^48, 2^-16
    } else {
        const float p3 = 3.0f * f1 * f2;
        float Q = 2.0f * p3;
        if (c4) {
            // d = n3 - n2 < n1 from the exact difference, truncated (of two rounded floats it
            // would leave Q < 0 where n1 < 1e-14)
            const float f3 = (float)(uint32_t)(N3 >> 32) * 9.31322574615478515625e-10f;      // 2^-30
            const float d = (float)(uint32_t)(D >> 32) * 9.31322574615478515625e-10f;
            Q = 0.75f * fmaf(f1, fmaf(2.0f, f2 + f3, -f1), -d * d);
        }
        const float rq = rsq(Q), x = (p3 * rq) * (fa * rq) * rq, z = x * x;
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
    s = c4 ? 0ull : (u64)Y;
    uint32_t m;
    int j;
    if (!split(w, m, j)) return true;
    const int sc = c1 ? 2 * j : e1 + e2;
    const u64 m2 = (u64)m * m, P12 = mulhi(M1, M2);
    const u64 X = q3(mulhi(P12, c1 ? ((c.a << 11) | TOP) : fixed(c.a)));
    u64 q = c1 ? 0ull : P12 >> 1;
    if (c4) {
        q = shr(mulhi(M1, ((N2 + N3) << 1) - N1), 2 + e2) - shl(mulhi(D, shl(D, -e1)), -e2);
    }
    const u64 R = c1 ? 0ull - shr(X, 1 + 2 * j - (e1 + e2 + ea)) : X;
    const u64 w3 = (((m2 >> 24) * m) << 16) + (((m2 & 0xffffffull) * m) >> 8);
    const i64 F = (i64)(shr(w3, 4 + sc - 3 * j) - (c1 ? 0ull : shr(q3(mul24(q, m)), -j)) + R);
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
    int k = 0;
    if (!in_range(b1, b3, v0) && !(volume_in_range(v0) && rescale(b1, b2, b3, k))) return false;
    Task t;
    const int code = classify(b1, b2, b3, va, t, s);
    if (code == 5) {
        d0 = unscale(va < HALF ? s | TOP : s, k);
        return true;
    }
    const bool ok = code == 2 ? root_square(t, s) : root_cubic(t, code == 1, code == 4, s);
    d0 = unscale(round_s(s, va < HALF), k);
    return ok;
}

#ifndef FX_HOST
}  // namespace fx
}  // namespace plic
#endif
