// vof_curvature.cuh -- the per-cell curvature step (Sec. 4.2, Appendix B),
// shared by the single-field and the batched kernels.
//
// For one interface cell c of a field phi (x-fastest):
//   1. gather the 3^3 stencil (D3Q27 order of Appendix B);
//   2. Parker-Youngs normal n = -sum w_i e_i phi_i / |.| (Eq. 38; the weights
//      4/2/1 make it a separable [1 2 1] x [1 2 1] smoothed central difference);
//   3. frame b_z = n, b_y = (n x r)/|.|, b_x = b_y x b_z (Sec. 4.2), r rotated
//      cyclically in the event that it is parallel to n;
//   4. PLIC offsets d0(phi_0, n) and d0(phi_i, n) of the interface neighbours,
//      all with the centre normal (FP32 solver + one Newton polish), giving the
//      points p_i = (e_i . b_x, e_i . b_y, e_i . b_z + d0_i - d0_0) (Eq. 36), or
//      the cut-polygon centroids with PLIC_FLAG_POINT_CENTROID;
//   5. normal equations M = sum Q Q^T, b = sum z Q, Q = (x^2, y^2, xy, x, y),
//      accumulated in FP32 (Appendix B);
//   6. LDL^T solve of the leading block (dimension min(m, 5), reduced while a
//      pivot is <= 1e-6 trace(M)) in FP64, FP32 or double-float;
//   7. mean curvature of the paraboloid at the origin (Eq. 42), negated by
//      default so that a convex fluid region has kappa > 0.
#pragma once
#include <type_traits>
#include "plic_polygon.cuh"

namespace plic {

enum { FIT_FP64 = 0, FIT_FP32 = 1, FIT_DF32 = 2, FIT_AUTO = 3 };

// D3Q27 directions e_0..e_26, packed as (ex+1) + 3 (ey+1) + 9 (ez+1).
#define PLIC_E27_PACKED          \
    13,                          \
    14, 12, 16, 10, 22, 4,       \
    17, 9, 23, 3, 25, 1,         \
    11, 15, 5, 21, 19, 7,        \
    26, 0, 8, 18, 20, 6,         \
    24, 2
__constant__ unsigned char c_e27[27] = {PLIC_E27_PACKED};
struct E27Table {
    static constexpr unsigned char v[27] = {PLIC_E27_PACKED};
};

// e_i from the constant table: the cheapest in registers; the lanes of a warp
// that ask for different i are served one address at a time.
__device__ __forceinline__ void e_of(int i, int& ex, int& ey, int& ez) {
    const int p = c_e27[i];
    ex = p % 3 - 1;
    ey = (p / 3) % 3 - 1;
    ez = p / 9 - 1;
}

// e_i decoded from immediates, for indices that differ across the lanes of a
// warp: the components (+1) are 2-bit fields of two 32-bit words per axis
// (entries 0-15 and 16-26), entry i at bits 2 (i mod 16).
constexpr uint32_t e27_word(int axis, int half) {
    uint32_t w = 0;
    for (int i = 16 * half; i < 27 && i < 16 * half + 16; ++i) {
        const int p = E27Table::v[i];
        const int e = axis == 0 ? p % 3 : axis == 1 ? (p / 3) % 3 : p / 9;
        w |= (uint32_t)e << (2 * (i - 16 * half));
    }
    return w;
}
template <int AXIS>
struct E27Words {
    static constexpr uint32_t lo = e27_word(AXIS, 0), hi = e27_word(AXIS, 1);
};
template <int AXIS>
__device__ __forceinline__ int e27_comp(int i) {
    const uint32_t w = i < 16 ? E27Words<AXIS>::lo : E27Words<AXIS>::hi;
    return (int)((w >> (2 * (i & 15))) & 3u) - 1;
}

__device__ __forceinline__ void e_of_lanes(int i, int& ex, int& ey, int& ez) {
    ex = e27_comp<0>(i);
    ey = e27_comp<1>(i);
    ez = e27_comp<2>(i);
}

// The D3Q27 directions as a block-shared table (integer and float
// components), filled by the first 27 threads of the block (every thread of
// the block must call fill()): loops over per-lane entries look their
// directions up (one shared load each) instead of decoding them.
struct E27Shared {
    int4 ei[27];
    float4 ef[27];
    __device__ __forceinline__ void fill() {
        if (threadIdx.x < 27) {
            int ex, ey, ez;
            e_of_lanes((int)threadIdx.x, ex, ey, ez);
            ei[threadIdx.x] = make_int4(ex, ey, ez, 0);
            ef[threadIdx.x] = make_float4((float)ex, (float)ey, (float)ez, 0.0f);
        }
        __syncthreads();
    }
};

// The same table for a compile-time index (fully unrolled loops): folds to
// constants.
template <int I>
__device__ __forceinline__ void e_of_c(int& ex, int& ey, int& ez) {
    constexpr int p = E27Table::v[I];
    ex = p % 3 - 1;
    ey = (p / 3) % 3 - 1;
    ez = p / 9 - 1;
}
// f(std::integral_constant<int, Q>) for Q = FROM..26, in order.
template <int FROM, typename F>
__device__ __forceinline__ void for_e27(F&& f) {
    if constexpr (FROM < 27) {
        f(std::integral_constant<int, FROM>{});
        for_e27<FROM + 1>(f);
    }
}

template <int FIT> struct FitReal;
template <> struct FitReal<FIT_FP64> {
    typedef double R;
    static __device__ __forceinline__ R mk(float a) { return (double)a; }
    static __device__ __forceinline__ R add(R a, R b) { return a + b; }
    static __device__ __forceinline__ R sub(R a, R b) { return a - b; }
    static __device__ __forceinline__ R mul(R a, R b) { return a * b; }
    static __device__ __forceinline__ R div(R a, R b) { return a / b; }
    static __device__ __forceinline__ float tof(R a) { return (float)a; }
    static __device__ __forceinline__ bool gt(R a, R b) { return a > b; }
};
template <> struct FitReal<FIT_FP32> {
    typedef float R;
    static __device__ __forceinline__ R mk(float a) { return a; }
    static __device__ __forceinline__ R add(R a, R b) { return a + b; }
    static __device__ __forceinline__ R sub(R a, R b) { return a - b; }
    static __device__ __forceinline__ R mul(R a, R b) { return a * b; }
    // MUFU reciprocal and a multiply (2 ulp): the divisors are the LDL^T pivots,
    // positive and far inside the normal range
    static __device__ __forceinline__ R div(R a, R b) { return a * rcp_approx(b); }
    static __device__ __forceinline__ float tof(R a) { return a; }
    static __device__ __forceinline__ bool gt(R a, R b) { return a > b; }
};
template <> struct FitReal<FIT_DF32> {
    typedef df R;
    static __device__ __forceinline__ R mk(float a) { return df_make(a); }
    static __device__ __forceinline__ R add(R a, R b) { return df_add(a, b); }
    static __device__ __forceinline__ R sub(R a, R b) { return df_add(a, df_neg(b)); }
    static __device__ __forceinline__ R mul(R a, R b) { return df_mul(a, b); }
    static __device__ __forceinline__ R div(R a, R b) { return df_div(a, b); }
    static __device__ __forceinline__ float tof(R a) { return a.hi + a.lo; }
    static __device__ __forceinline__ bool gt(R a, R b) {
        return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo);
    }
};

// Packed upper triangle of the symmetric 5x5 normal matrix.
__host__ __device__ constexpr int uidx(int i, int j) {
    return i <= j ? i * 5 - i * (i - 1) / 2 + (j - i) : j * 5 - j * (j - 1) / 2 + (i - j);
}

// LDL^T factorisation of the leading block of the symmetric normal matrix
// (Appendix B reduces the fit dimension when fewer than 5 points exist).  The
// dimension is min(m, 5), reduced to j at the first pivot D_j <= 1e-6 trace(M)
// (D_j is the ratio of consecutive leading principal minors).  solve() uses
// the factors for any right-hand side (the fit, and the adjoint system of the
// backward pass); unused parameters are 0.
template <int FIT>
struct Ldlt {
    typedef FitReal<FIT> F;
    typedef typename F::R R;
    R Lm[5][5], D[5];
    int dim;
    __device__ __forceinline__ void factor(const float* Mf, int m) {
        const float trace = Mf[uidx(0, 0)] + Mf[uidx(1, 1)] + Mf[uidx(2, 2)] + Mf[uidx(3, 3)] + Mf[uidx(4, 4)];
        const R tol = F::mk(1e-6f * trace);
        dim = m < 5 ? m : 5;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            R dj = F::mk(Mf[uidx(j, j)]);
#pragma unroll
            for (int k = 0; k < j; ++k) dj = F::sub(dj, F::mul(F::mul(Lm[j][k], Lm[j][k]), D[k]));
            const bool act = j < dim;
            if (act && !F::gt(dj, tol)) dim = j;
            D[j] = dj;
            const bool use = j < dim;
            const R inv = use ? F::div(F::mk(1.0f), dj) : F::mk(0.0f);
#pragma unroll
            for (int i = j + 1; i < 5; ++i) {
                R s = F::mk(Mf[uidx(i, j)]);
#pragma unroll
                for (int k = 0; k < j; ++k) s = F::sub(s, F::mul(F::mul(Lm[i][k], Lm[j][k]), D[k]));
                Lm[i][j] = F::mul(s, inv);
            }
        }
    }
    __device__ __forceinline__ void solve(const float* bf, float x[5]) const {
        R y[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            R s = F::mk(bf[i]);
#pragma unroll
            for (int k = 0; k < i; ++k) s = F::sub(s, F::mul(Lm[i][k], y[k]));
            y[i] = i < dim ? s : F::mk(0.0f);
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) y[i] = i < dim ? F::div(y[i], D[i]) : F::mk(0.0f);
        R xs[5];
#pragma unroll
        for (int i = 4; i >= 0; --i) {
            R s = y[i];
#pragma unroll
            for (int k = i + 1; k < 5; ++k) s = F::sub(s, F::mul(Lm[k][i], xs[k]));
            xs[i] = i < dim ? s : F::mk(0.0f);
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) x[i] = F::tof(xs[i]);
    }
};

// Adaptive factorisation (the FIT_AUTO policy): LDL^T in FP32, replaced by an
// FP64 factorisation when the FP32 pivots show an ill-conditioned matrix
// (smallest pivot below 1e-2 of the largest, or a dimension reduced by the
// FP32 pivots).  Same interface as Ldlt (factor(), solve(), dim).  The FP64
// factors are not kept: the rare wide solve refactorises from Mf, which must
// stay valid between factor() and the solves; this keeps the FP64 factors out
// of the registers of the common path.
struct LdltAuto {
    Ldlt<FIT_FP32> f;
    const float* Mf;
    int m, dim;
    bool wide;
    __device__ __forceinline__ void factor(const float* M, int mm) {
        Mf = M;
        m = mm;
        f.factor(M, mm);
        const int want = mm < 5 ? mm : 5;
        float dmin = 3.4e38f, dmax = 0.0f;
#pragma unroll
        for (int j = 0; j < 5; ++j)
            if (j < f.dim) { dmin = fminf(dmin, f.D[j]); dmax = fmaxf(dmax, f.D[j]); }
        wide = !(f.dim == want && dmin > 1e-2f * dmax);
        dim = f.dim;
        if (wide) {
            Ldlt<FIT_FP64> w;
            w.factor(M, mm);
            dim = w.dim;
        }
    }
    __device__ __forceinline__ void solve(const float* bf, float x[5]) const {
        if (wide) {
            Ldlt<FIT_FP64> w;
            w.factor(Mf, m);
            w.solve(bf, x);
        } else {
            f.solve(bf, x);
        }
    }
};

template <int FIT>
__device__ __forceinline__ int fit_solve(const float* Mf, const float* bf, int m, float x[5]) {
    Ldlt<FIT> f;
    f.factor(Mf, m);
    f.solve(bf, x);
    return f.dim;
}

// Eq. 42 at the origin: (A (I^2+1) + B (H^2+1) - C H I) / (H^2 + I^2 + 1)^(3/2).
__device__ __forceinline__ float paraboloid_kappa(const float x[5]) {
    const float A = x[0], B = x[1], C = x[2], H = x[3], I = x[4];
    const float s = fmaf(H, H, fmaf(I, I, 1.0f));
    const float r = rsqrtf(s);
    return (A * fmaf(I, I, 1.0f) + B * fmaf(H, H, 1.0f) - C * H * I) * (r * r * r);
}

// The reduced normal of the centre cell, shared by all PLIC solves of the cell.
template <int METHOD>
struct CellPlic {
    float n1, n2, n3, L, m1, m2, m3;
    __device__ __forceinline__ void prepare(float nx, float ny, float nz) {
        reduce_normal<float, false>(nx, ny, nz, n1, n2, n3);
        L = fabsf(nx) + fabsf(ny) + fabsf(nz);
        if (METHOD == M_SZ_ORIG) {
            m1 = n1 / L;
            m3 = n3 / L;
            m2 = fmaxf(1.0f - (m1 + m3), 0.0f);
        }
    }
    // d0(V0, n) in FP32 with one Newton polish (PLIC_FP32_POLISHED); V0 in (0, 1).
    __device__ __forceinline__ float offset(float V0) const {
        const float V = V0 <= 0.5f ? V0 : 1.0f - V0;
        if (METHOD == M_SZ_ORIG) {
            float a = solve_sz_orig<float, false>(V, m1, m2, m3);
            a = polish<float>(a, V, m1, m2, m3);
            return L * copysignf(0.5f - a, V0 - 0.5f);
        }
        float d = METHOD == M_ANALYTIC ? solve_analytic<float, false>(V, n1, n2, n3)
                : METHOD == M_NEWTON   ? solve_newton<float, false>(V, n1, n2, n3)
                                       : solve_nested<float, false>(V, n1, n2, n3);
        d = polish<float>(d, V, n1, n2, n3);
        return copysignf(0.5f * (n1 + n2 + n3) - d, V0 - 0.5f);
    }
};

// The smaller positive root w of the depressed cubic w^3 - Q w + R = 0 of cases
// (3)/(4) (p2::centre_distance) as a function of X = R/Q, its limit for small w: with
// z = X^2/Q <= 0.1158 in these cases, w = X P(z) by the polynomial of
// p2::depressed_root (signs turned), h = w^2/Q, and one Newton step on
// w h - w + X = 0, w + (w h - w + X)/(1 - 3 h).  X is linear in the volume, k V + c, and
// the step's residual takes c - w first, so that neither X's rounding nor the step's
// stays in w; the constants of the normal are k, c and 1/Q.
// |d0| error, rms, against 64 bits for random (nearly equal) components: case (3)
// 2.1e-8 (2.4e-8), case (4) 1.2e-8 (1.8e-8); with the argument and the root in units of
// (Q/3)^(1/2), five constants rounded before the volume is known, 3.3e-8 (7.3e-8) and
// 1.4e-8 (2.7e-8); the arcsine and a Newton step on Eq. 10 2.6e-8 (2.5e-8) and
// 2.9e-8 (2.7e-8).
struct CentreRoot {
    static constexpr float c0 = 1.001369833946228f, c1 = 0.8008332848548889f, c2 = 10.902824401855469f,
                           c3 = -107.44769287109375f, c4 = 704.3350219726562f;
    // z is held below 0.12: where m1 < 1e-14 m2 the thresholds' rounding lets volumes of
    // cases (2) and (5) in, with X of either sign below 1e-7 and Q far below X^2
    // (1/Q up to infinity: X^2/Q infinite or NaN, taken as 0.12).
    static constexpr float zmax = 0.12f;
    static __device__ __forceinline__ float eval(float k, float V, float c, float iq, float b) {
        const float X = fmaf(k, V, c), z = fminf(X * X * iq, zmax);
        const float p = fmaf(fmaf(fmaf(fmaf(c4, z, c3), z, c2), z, c1), z, c0);
        const float w = X * p, h = p * p * z;
        const float f = fmaf(w, h, fmaf(k, V, c - w));
        return fmaf(f, rcp_approx(fmaf(-3.0f, h, 1.0f)), w + b);
    }
};

// The optimised SZ solution (Sec. 2.4) with everything that depends on the
// normal alone computed once per curvature cell (all neighbour solves of a
// cell use the centre normal, Eq. 36).  Per solve there remain: the reduced
// volume, four threshold tests on V, the closed forms of cases (5), (2), (1)
// (the last as cbrt(6 m1 m2 m3) * cbrt(V)), and the root of the depressed cubic
// of cases (3)/(4) (CentreRoot).  All as distances s = 1/2 - d from the
// cell's centre.  The thresholds are the product-form tests of
// solve_sz_opt_default divided through once.
template <>
struct CellPlic<M_SZ_OPT> {
    float L, m3;
    float V5, V1, V2, V3;
    float c3, i3, b3, k4, c4, i4, k2a, k2b, h2, cb1;
    __device__ __forceinline__ void prepare(float nx, float ny, float nz) {
        const float ax = fabsf(nx), ay = fabsf(ny), az = fabsf(nz);
        L = ax + ay + az;
        // MUFU reciprocals (no IEEE division): the thresholds only choose
        // between case formulas that agree at the case boundaries
        const float il = rcp_approx(L);
        const float m1 = fminf(fminf(ax, ay), az) * il;
        m3 = fmaxf(fmaxf(ax, ay), az) * il;
        const float m2 = fmaxf(1.0f - (m1 + m3), 0.0f);
        const float n12 = m1 + m2;
        const float m1m2 = m1 * m2, sq1 = m1 * m1;
        const float k23 = 6.0f * m2 * m3;
        const float rk = k23 > 0.0f ? rcp_approx(k23) : 0.0f;
        const float inv1 = m1 > 0.0f ? rcp_approx(m1) : 0.0f;
        V5 = 0.5f * n12 * rcp_approx(m3);                  // case (5): V >= V5
        V1 = sq1 * rk;                                           // case (1): V < V1
        V2 = (sq1 - 3.0f * m2 * (m1 - m2)) * rk;                 // case (2): V < V2
        const float num3 = m3 * m3 * (3.0f * n12 - m3) + sq1 * (m1 - 3.0f * m3) + m2 * m2 * (m2 - 3.0f * m3);
        // (below 1e-30 case (4) is no wider than a rounding, and its constants overflow)
        V3 = (m3 < n12 && m1m2 > 1e-30f) ? num3 * rk * inv1 : 3.4e38f;  // case (3): V < V3
        // case (3): X = (m1 + m2)/2 - m3 V, Q = 6 m1 m2, s = 1/2 - m1 - m2 + w
        c3 = 0.5f * n12;
        i3 = rcp_approx(6.0f * m1m2);
        b3 = 0.5f - n12;
        // case (4): X = c (1 - 2 V), Q = 3/4 q, s = w with q = m1 (2 - 3 m1) - (m3 - m2)^2 and
        // c = 2 m1 m2 m3 / q, a division with the products' roundings carried along
        const float d32 = m3 - m2, e = fmaf(-3.0f, m1, 2.0f), me = m1 * e, q = fmaf(-d32, d32, me);
        const float num = m1m2 * (2.0f * m3);
        const float rnum = fmaf(m1m2, 2.0f * m3, -num) + 2.0f * m3 * fmaf(m1, m2, -m1m2);
        const float r = rcp_approx(q), c = num * r;
        c4 = fmaf(fmaf(-c, q, num) + fmaf(-c, fmaf(m1, e, -me), rnum), r, c);
        k4 = -2.0f * c4;
        i4 = (4.0f / 3.0f) * r;
        k2a = 2.0f * m2 * m3;
        k2b = sq1 * (1.0f / 12.0f);
        h2 = 0.5f - 0.5f * m1;
        cb1 = Fm<float>::cbrt_(k23 * m1);
    }
    __device__ __forceinline__ float offset(float V0) const {
        const float V = fminf(V0, 1.0f - V0);
        const bool three = V < V3;
        float s = CentreRoot::eval(three ? -m3 : k4, V, three ? c3 : c4, three ? i3 : i4, three ? b3 : 0.0f);
        if (V < V2) s = h2 - Fm<float>::sqrt_(fmaxf(fmaf(k2a, V, -k2b), 1e-30f));
        if (V < V1) s = fmaf(-cb1, Fm<float>::cbrt_(V), 0.5f);
        if (V >= V5) s = m3 * (0.5f - V);
        return copysignf(L * s, V0 - 0.5f);
    }
};

// Normal of the 3^3 stencil around cell c (Appendix B): Parker-Youngs
// weights 4/2/1 (Eq. 38), or all 1 for the centre-of-mass normal.  Row by
// row: the weights of the x-difference of row (dy, dz) are w(dy) w(dz) with
// w(0) = 2, w(+-1) = 1; the row sums for the y and z components weigh the
// middle entry 2 (all 1 for CM).  Returns false for a zero weighted sum.
__device__ __forceinline__ bool stencil_normal(const float* __restrict__ phi, int64_t c, int nx,
                                               int64_t nxy, bool cm, float& nx_, float& ny_,
                                               float& nz_) {
    float gx = 0.0f, gy = 0.0f, gz = 0.0f;
    const float w0 = cm ? 1.0f : 2.0f;
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy) {
            const float* row = phi + c + dz * nxy + (int64_t)dy * nx;
            const float a = __ldg(row - 1), b = __ldg(row), e = __ldg(row + 1);
            const float wy = dy == 0 ? w0 : 1.0f, wz = dz == 0 ? w0 : 1.0f;
            const float sum = fmaf(w0, b, a + e);
            gx = fmaf(wy * wz, e - a, gx);
            gy = fmaf((float)dy * wz, sum, gy);
            gz = fmaf((float)dz * wy, sum, gz);
        }
    const float gl = sqrtf(gx * gx + gy * gy + gz * gz);
    if (!(gl > 0.0f)) { nx_ = ny_ = nz_ = 0.0f; return false; }
    const float inv = -1.0f / gl;
    nx_ = gx * inv; ny_ = gy * inv; nz_ = gz * inv;
    return true;
}

// The neighbour-normal variant (PLIC_FLAG_NEIGHBOR_NORMAL), one thread per
// list entry; defined in vof_curvature_nn.cu.  out[k] = scale * kappa[k].
plic_status launch_curvature_nn(const float* phi, int nx, int ny, int nz, const int32_t* idx,
                                int64_t n_iface, const int64_t* d_n_iface, float* out,
                                plic_method m, uint32_t flags, int fit, float scale,
                                void* stream, const char* who);

}  // namespace plic
