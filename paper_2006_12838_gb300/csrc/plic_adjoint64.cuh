// plic_adjoint64.cuh -- area and centroid of the cut polygon in FP64 (what
// plic_polygon.cuh computes), written for the FP64 pipe.
//
// That pipe bounds the FP64 adjoints (one FP64 operation per 72 FP32 ones), so: one
// branch-free path for all cases of Eq. 10 (in area_centroid the three cases
// diverge and a warp pays for each), reciprocals from FP32 starts, finished by one
// third-order step each (three FP64 operations; a division takes about ten), |n| by
// its expansion about 1, and signs, comparisons, maxima, the sort and its undoing on
// the integer pipe.  8 M cells, offset and its
// adjoint: 1973 -> 1044 us (the offset about 140 of it), 62 FP64 operations per cell;
// errors against 64-bit differentiation 1.6e-15 -> 1.1e-15 (d0 by V0), 4.8e-16 -> 4.4e-16.
//
// With e_k = (d - n_k)_+ and Eq. 10's 6 n1 n2 n3 V = d^3 - sum e_k^3 (d <= n1 + n2),
//   N = 6 n2 n3 V     = (d^3 - e1^3)/n1 - (e2^3 + e3^3)/n1,
//   G = 6 n2 n3 dV/dd = 3 (d^2 - e1^2)/n1 - 3 (e2^2 + e3^2)/n1,
//   c1 = ((d^3 - e1^3)/n1^2 - 3 e1^2/n1 - (e2^3 + e3^3)/n1^2)/G,
//   ck = (N/nk - 3 ek^2/n1)/G for k = 2, 3;
// the terms of d and e1 are d^2/n1, d^3/n1 and d^3/n1^2 for d < n1 (case (1)),
// and 2d - n1, 3d(d - n1) + n1^2 and 3d - 2n1 above, where nothing cancels and
// n1 may be 0.  Case (5), d >= n1 + n2: c = (1/2, 1/2, (d - (n1 + n2)/2)/n3),
// dV/dd = 1/n3.
//
// Nothing here needs the GPU (plic_fx.cuh's primitives).
#pragma once
#include "plic_fx.cuh"

#ifndef FX_HOST
namespace plic {
namespace fx {
#endif

// A positive normal float as a double (F2F would take the FP64 pipe)
FX_D double widen(float x) { return asd(((u64)asu(x) << 29) + ((u64)896 << 52)); }
// 1/x for x in [2^-126, 2^126]: start y (1 - x y = e below 2^-21), then y (1 + e + e^2)
FX_D double recip(double x) {
    const double y = widen(rcp(flt(bits(x)))), e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
FX_D void swap_if(bool c, double& a, double& b) { const double t = c ? b : a; b = c ? a : b; a = t; }

// dd0/dV0 = 1/A (INVERSE) or A, and the centroid, for components, signs and offset as
// bits; false for cells that the caller hands to area_centroid: n_k or d = L/2 - |d0|
// below 2^-30 (n_k = 0 is taken) or d from 2 on, invalid input.
template <bool INVERSE>
FX_D bool area_centroid64(u64 nx, u64 ny, u64 nz, u64 d0, double& A, double& cx, double& cy, double& cz) {
    u64 b1 = nx & ABS, b2 = ny & ABS, b3 = nz & ABS, t;
    const bool s1 = b1 > b2;
    t = s1 ? b2 : b1; b2 = s1 ? b1 : b2; b1 = t;
    const bool s2 = b2 > b3;
    t = s2 ? b3 : b2; b3 = s2 ? b2 : b3; b2 = t;
    const bool s3 = b1 > b2;
    t = s3 ? b2 : b1; b2 = s3 ? b1 : b2; b1 = t;
    const double n1 = asd(b1), n2 = asd(b2), n3 = asd(b3);
    const double n12 = n1 + n2, d = fma(0.5, n12 + n3, asd(d0 | TOP));
    // |n|: 1 + q with q = n . n - 1
    const double q = fma(n3, n3, fma(n2, n2, fma(n1, n1, -1.0)));
    const uint32_t LO = (uint32_t)(1023 - 30) << 20;
    const uint32_t h1 = (uint32_t)(b1 >> 32), h2 = (uint32_t)(b2 >> 32), hd = (uint32_t)(bits(d) >> 32);
    if (!(hd - LO < (31u << 20) && (h1 >= LO || b1 == 0ull) && (h2 >= LO || b2 == 0ull))) return false;
    // |n| or 1/|n| to q^3/16 (5 q^3/16) < 2^-55
    double rs = INVERSE ? fma(fma(0.375, q, -0.5), q, 1.0) : fma(fma(-0.125, q, 0.5), q, 1.0);
    if (((uint32_t)(bits(q) >> 32) & 0x7fffffffu) >= (1023u - 18u) << 20) {
        // |n|^2 off 1 by 2^-18 or more: 1/|n| from an FP32 start and a third-order step
        // (these cells by the general formula instead: 4015 us per 2^24, this way 2125)
        const double nn = fma(n3, n3, fma(n2, n2, n1 * n1)), y = widen(rsq(flt(bits(nn)))), e = fma(-nn * y, y, 1.0);
        const double r = fma(y, e * fma(0.375, e, 0.5), y);
        rs = INVERSE ? r : nn * r;
    }
    const bool five = (i64)bits(d) >= (i64)bits(n12), low = (i64)bits(d) < (i64)b1;
    u64 be2 = bits(d - n2), be3 = bits(d - n3);
    be2 = (i64)be2 < 0 ? 0ull : be2;
    be3 = (i64)be3 < 0 ? 0ull : be3;
    const double e2 = asd(be2), e3 = asd(be3);
    const double r1 = b1 == 0ull ? 0.0 : recip(n1);
    const double e22 = e2 * e2, e33 = e3 * e3;
    const double cub = fma(e22, e2, e33 * e3) * r1, m = d - n1, d3 = 3.0 * d;
    const double u = d * r1, a2l = d * u;
    const double a2 = low ? 3.0 * a2l : fma(3.0, m, d3), r13 = -3.0 * r1;
    const double a3 = low ? d * a2l : fma(d3, m, n1 * n1);
    const double a4 = low ? u * a2l : fma(-2.0, n1, d3);
    const double G = fma(e22 + e33, r13, a2), N = a3 - cub;
    const double iG = recip(five ? 1.0 : G), r2 = recip(five ? 1.0 : n2), r3 = recip(n3);
    double c1 = fma(-cub, r1, a4) * iG;
    double c2 = fma(N, r2, e22 * r13) * iG;
    double c3 = fma(N, r3, e33 * r13) * iG;
    c1 = five ? 0.5 : c1;
    c2 = five ? 0.5 : c2;
    c3 = five ? fma(-0.5, n12, d) * r3 : c3;
    if (INVERSE) A = (five ? n3 : n2 * n3 * (6.0 * iG)) * rs;
    else A = (five ? 1.0 : G * (1.0 / 6.0) * r2) * r3 * rs;
    c1 -= 0.5; c2 -= 0.5; c3 -= 0.5;
    swap_if(s3, c1, c2);
    swap_if(s2, c2, c3);
    swap_if(s1, c1, c2);
    // c - 1/2 with the sign of n, mirrored for d0 > 0
    cx = asd(bits(c1) ^ (~(nx ^ d0) & TOP));
    cy = asd(bits(c2) ^ (~(ny ^ d0) & TOP));
    cz = asd(bits(c3) ^ (~(nz ^ d0) & TOP));
    return true;
}

#ifndef FX_HOST
}  // namespace fx
}  // namespace plic
#endif
