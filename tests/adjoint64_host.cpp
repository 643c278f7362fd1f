// adjoint64_host.cpp -- area_centroid64 (csrc/plic_adjoint64.cuh) on the host against
// quadruple precision, beside the general formula in doubles: CELLS KIND prints the cells
// refused, then for 1/A and A (relative) and c the scheme's largest and rms error and the
// general formula's.  The primitives are those of fx_host.cpp.
#define main unit_main
#include "fx_host.cpp"
#undef main
#include "../paper_2006_12838_gb300/csrc/plic_adjoint64.cuh"

static double root(double x) { return std::sqrt(x); }
static quad root(quad x) {
#if defined(__x86_64__)
    quad y = std::sqrt((double)x);
    for (int i = 0; i < 3; ++i) y = (y + x / y) / 2;
    return y;
#else
    return std::sqrt(x);
#endif
}

// A and c (plic_polygon.cuh's formulas) in T
template <typename T> static void general(const double n[3], double d0, T& A, T c[3]) {
    int id[3] = {0, 1, 2};
    auto less = [&](int a, int b) { return std::fabs(n[a]) < std::fabs(n[b]); };
    if (less(id[1], id[0])) std::swap(id[0], id[1]);
    if (less(id[2], id[1])) std::swap(id[1], id[2]);
    if (less(id[1], id[0])) std::swap(id[0], id[1]);
    const T n1 = std::fabs(n[id[0]]), n2 = std::fabs(n[id[1]]), n3 = std::fabs(n[id[2]]);
    const T d = (n1 + n2 + n3) / 2 - (T)std::fabs(d0), n12 = n1 + n2;
    const T r3 = 1 / n3, r2 = n2 > 0 ? 1 / n2 : (T)0, r1 = n1 > 0 ? 1 / n1 : (T)0;
    T vp, k[3];
    if (d >= n12) {
        vp = r3; k[0] = k[1] = (T)0.5; k[2] = (d - n12 / 2) * r3;
    } else if (d < n1) {
        vp = d * d * r1 * r2 * r3 / 2; k[0] = d * r1 / 3; k[1] = d * r2 / 3; k[2] = d * r3 / 3;
    } else {
        const T e2 = d > n2 ? d - n2 : (T)0, e3 = d > n3 ? d - n3 : (T)0;
        const T cub = (e2 * e2 * e2 + e3 * e3 * e3) * r1, N = 3 * d * (d - n1) + n1 * n1 - cub;
        const T G = 6 * d - 3 * n1 - 3 * (e2 * e2 + e3 * e3) * r1;
        vp = G * r2 * r3 / 6;
        k[0] = (3 * d - 2 * n1 - cub * r1) / G;
        k[1] = (N * r2 - 3 * e2 * e2 * r1) / G;
        k[2] = (N * r3 - 3 * e3 * e3 * r1) / G;
    }
    A = root((T)(n1 * n1 + n2 * n2 + n3 * n3)) * vp;
    for (int j = 0; j < 3; ++j) {
        const T u = d0 > 0 ? (T)0.5 - k[j] : k[j] - (T)0.5;
        c[id[j]] = n[id[j]] < 0 ? -u : u;
    }
}

int main(int argc, char** argv) {
    const long cells = argc > 1 ? atol(argv[1]) : 20000;
    const int kind = argc > 2 ? atoi(argv[2]) : 0;
    std::mt19937_64 r(5 + kind);
    std::uniform_real_distribution<double> u(0, 1);
    std::normal_distribution<double> g;
    long refused = 0, count = 0;
    double worst[3][2] = {}, sum[3][2] = {};
    for (long i = 0; i < cells; ++i) {
        // unit length; 1/2 to 2; unit L1 length; 2^-8 to 1
        double n[3], l = 0;
        for (double& x : n) x = g(r);
        if (u(r) < 0.2) n[0] = 0;
        if (u(r) < 0.2) n[1] = n[2];
        for (double x : n) l += kind == 2 ? std::fabs(x) : x * x;
        l = kind == 2 ? l : std::sqrt(l);
        const double scale = kind == 1 ? std::pow(2, 2 * u(r) - 1) : kind == 3 ? std::pow(2, -8 * u(r)) : 1;
        double L = 0, least = 1;
        for (double& x : n) {
            x *= scale / l;
            L += std::fabs(x);
            if (x != 0) least = std::fmin(least, std::fabs(x));
        }
        const double d = L / 2 * (1e-3 + 0.999 * u(r)), d0 = (u(r) < 0.5 ? -1 : 1) * (L / 2 - d);
        if (least < 1e-6 || L > 3.9) continue;
        quad A, c[3];
        double Ad, cd[3], iA, As, cs[3];
        general(n, d0, A, c);
        general(n, d0, Ad, cd);
        if (!area_centroid64<true>(bits(n[0]), bits(n[1]), bits(n[2]), bits(d0), iA, cs[0], cs[1], cs[2]) ||
            !area_centroid64<false>(bits(n[0]), bits(n[1]), bits(n[2]), bits(d0), As, cs[0], cs[1], cs[2])) {
            ++refused;
            continue;
        }
        ++count;
        auto add = [&](int k, int w, quad e) {
            const double x = (double)qabs(e);
            if (!(x <= worst[k][w])) worst[k][w] = x;
            sum[k][w] += x * x;
        };
        add(0, 0, (quad)iA * A - 1);
        add(0, 1, (quad)(1 / Ad) * A - 1);
        add(1, 0, (quad)As / A - 1);
        add(1, 1, (quad)Ad / A - 1);
        for (int k = 0; k < 3; ++k) {
            add(2, 0, (quad)cs[k] - c[k]);
            add(2, 1, (quad)cd[k] - c[k]);
        }
    }
    printf("%ld", refused);
    for (int k = 0; k < 3; ++k)
        for (int w = 0; w < 2; ++w) printf(" %.4g %.4g", worst[k][w], std::sqrt(sum[k][w] / count));
    printf("\n");
    return 0;
}
