// The fixed-point FP64 offset (csrc/plic_fx.cuh) on the host, against bisection
// in quadruple precision: fx_host CELLS KIND prints the number of cells
// refused though inside the scheme's range and the largest error.  The MUFU
// approximations are replaced by exact values with a relative error of their
// documented size.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <utility>

#define FX_HOST
#define FX_D inline
typedef unsigned long long u64;
typedef long long i64;
#if defined(__x86_64__)
typedef __float128 quad;
#else
typedef long double quad;
#endif
static std::minstd_rand noise(1);
static double off(double size) { return 1 + size * ((noise() % 20001) / 10000.0 - 1); }
static long bad_shifts = 0;
FX_D u64 mulhi(u64 a, u64 b) { return (u64)(((unsigned __int128)a * b) >> 64); }
FX_D u64 shr(u64 x, int s) { bad_shifts += s < 0 && x; return s < 0 || s > 63 ? 0 : x >> s; }
FX_D u64 shl(u64 x, int s) { bad_shifts += s < 0 && x; return s < 0 || s > 63 ? 0 : x << s; }
FX_D int clz(u64 x) { return x ? __builtin_clzll(x) : 64; }
FX_D float asf(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
FX_D double asd(u64 u) { double d; memcpy(&d, &u, 8); return d; }
FX_D u64 bits(double d) { u64 u; memcpy(&u, &d, 8); return u; }
FX_D uint32_t asu(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
FX_D float rsq(float x) { return (float)(1 / std::sqrt((double)x) * off(1.2e-7)); }
FX_D float rcp(float x) { return (float)(1 / (double)x * off(1.2e-7)); }
FX_D float cbrt_start(float x) { return (float)(std::cbrt((double)x) * off(6e-6)); }
FX_D int rint_sat(float x) {
    return x != x ? 0 : x >= 2147483647.f ? 2147483647 : x <= -2147483648.f ? -2147483647 - 1 : (int)lrintf(x);
}
#include "../paper_2006_12838_gb300/csrc/plic_fx.cuh"

static quad qabs(quad x) { return x < 0 ? -x : x; }
static void order(double a[3]) {
    for (int k = 0; k < 3; ++k) a[k] = std::fabs(a[k]);
    if (a[0] > a[1]) std::swap(a[0], a[1]);
    if (a[1] > a[2]) std::swap(a[1], a[2]);
    if (a[0] > a[1]) std::swap(a[0], a[1]);
}
// Eq. 10 for 0 <= d <= L/2
static quad volume(quad d, quad n1, quad n2, quad n3) {
    if (d <= 0) return 0;
    if (d >= n1 + n2) return (d - (n1 + n2) / 2) / n3;
    if (d < n1) return d * d * d / (6 * n1 * n2 * n3);
    quad num = 3 * d * (d - n1) + n1 * n1;
    if (d > n2) {
        const quad e2 = d - n2, e3 = d > n3 ? d - n3 : 0;
        num -= (e2 * e2 * e2 + e3 * e3 * e3) / n1;
    }
    return num / (6 * n2 * n3);
}
static quad solve(const double n[3], double v) {
    double a[3] = {n[0], n[1], n[2]};
    order(a);
    const quad n1 = a[0], n2 = a[1], n3 = a[2], half = (n1 + n2 + n3) / 2, V = v <= 0.5 ? (quad)v : 1 - (quad)v;
    quad d = n3 * V + (n1 + n2) / 2;
    if (d < n1 + n2) {
        quad lo = 0, hi = half;
        for (int i = 0; i < 100 && hi - lo > (quad)1e-30; ++i) {
            const quad m = (lo + hi) / 2;
            if (volume(m, n1, n2, n3) < V) lo = m; else hi = m;
        }
        d = (lo + hi) / 2;
    }
    if (V <= 0) d = 0;
    return v >= 0.5 ? half - d : d - half;
}

int main(int argc, char** argv) {
    const long cells = atol(argv[1]);
    const int kind = atoi(argv[2]);
    std::mt19937_64 r(99 + kind);
    std::normal_distribution<double> g;
    std::uniform_real_distribution<double> u(0, 1);
    long refused = 0;
    double worst = 0;
    for (long i = 0; i < cells; ++i) {
        double n[3] = {g(r), g(r), g(r)}, v = u(r);
        if (kind == 1) {                             // components down to 1e-16
            n[0] *= std::pow(10, -16 * u(r));
            if (u(r) < 0.4) n[1] *= std::pow(10, -16 * u(r));
        }
        if (kind == 2) {                             // zero, equal and nearly equal components
            const int w = (int)(5 * u(r));
            if (w <= 1) n[0] = 0;
            if (w == 1) n[1] = 0;
            if (w == 2) n[0] = n[1] = n[2] = 1;
            if (w == 3) n[1] = n[0];
            if (w == 4) { n[0] = n[1] * (1 + 1e-6 * g(r)); n[2] = n[1] * (1 + 1e-9 * g(r)); }
        }
        const double L = std::sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
        for (int k = 0; k < 3; ++k) n[k] = n[k] / L * (u(r) < 0.5 ? -1 : 1);
        std::swap(n[0], n[(int)(3 * u(r))]);
        if (kind == 3 || (kind && kind < 3 && u(r) < 0.5)) {        // at and beside the case boundaries
            double a[3] = {n[0], n[1], n[2]};
            order(a);
            const quad half = ((quad)a[0] + a[1] + a[2]) / 2;
            const quad at[5] = {a[0], a[1], a[2], (quad)a[0] + a[1], half};
            quad d = at[(int)(5 * u(r))] + std::pow(10, -17 * u(r)) * (u(r) < 0.5 ? -1 : 1) * (u(r) < 0.5 ? 1 : a[0]);
            d = d < 0 ? 0 : d > half ? half : d;
            v = std::fmin((double)volume(d, a[0], a[1], a[2]), 0.5);
            if (u(r) < 0.5) v = 1 - v;
        }
        if (kind == 4) {                             // volumes down to 2^-96
            v = std::pow(2, -96 * u(r));
            if (u(r) < 0.3) v = 1 - v;
        }
        if (kind == 5) {
            const double ends[5] = {0.0, 1.0, 0.5, std::nextafter(0.5, 0), std::nextafter(0.5, 1)};
            v = ends[(int)(5 * u(r))];
        }
        u64 b[4], o;
        for (int k = 0; k < 3; ++k) memcpy(&b[k], &n[k], 8);
        memcpy(&b[3], &v, 8);
        double d0;
        if (!offset(b[0], b[1], b[2], b[3], o)) {
            refused += v == 0 || v >= std::pow(2, -96);
            continue;
        }
        memcpy(&d0, &o, 8);
        const double err = (double)qabs((quad)d0 - solve(n, v));
        if (!(err <= worst)) worst = err;
    }
    printf("%ld %.4g %ld\n", refused, worst, bad_shifts);
    return 0;
}
