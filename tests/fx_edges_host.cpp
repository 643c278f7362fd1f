// fx_edges_host.cpp -- the fixed-point FP64 offset on the host at edges that
// fx_host.cpp's draws do not meet: CELLS KIND prints the cells refused, the largest
// error (of the cell scaled by the power of two that brings n3 to [1/2, 1)) and the
// negative shifts.  Helpers and the reference are those of fx_host.cpp.
#define main unit_main
#include "fx_host.cpp"
#undef main

int main(int argc, char** argv) {
    const long cells = argc > 1 ? atol(argv[1]) : 20000;
    const int kind = argc > 2 ? atoi(argv[2]) : 0;
    std::mt19937_64 r(11 + kind);
    std::uniform_real_distribution<double> u(0, 1);
    std::normal_distribution<double> g;
    long refused = 0;
    double worst = 0;
    for (long i = 0; i < cells; ++i) {
        double n[3], a[3], v = u(r);
        if (kind == 0) {
            // n1 down to 1e-18, n3 - n2 of its size or a few ulp, V0 beside 1/2
            const double e = std::pow(10, -12 - 6 * u(r));
            n[1] = 0.5 + 0.45 * u(r);
            n[0] = e * (1 + u(r)) * n[1];
            n[2] = n[1] * (1 + (u(r) < 0.5 ? (int)(4 * u(r)) * 1.2e-16 : 2 * e * u(r)));
            v = 0.5 + (u(r) < 0.5 ? -1 : 1) * std::pow(10, -12 - 5 * u(r));
        }
        if (kind > 0) {
            // off unit length: 1/2 to 2; unit L1 length; down to 2^-58; components near 3/4
            double scale = 1, l = 0;
            for (double& x : n) x = g(r);
            if (u(r) < 0.3) n[0] *= std::pow(10, -17 * u(r));
            if (u(r) < 0.3) n[1] = n[0] * (1 + std::pow(10, -16 * u(r)));
            if (u(r) < 0.3) n[2] = n[1] * (1 + std::pow(10, -16 * u(r)));
            for (double x : n) l += kind == 2 ? std::fabs(x) : x * x;
            if (kind != 2) l = std::sqrt(l);
            if (kind == 1) scale = std::pow(2, 2 * u(r) - 1);
            if (kind == 3) scale = std::pow(2, -58 * u(r));
            if (kind == 4) scale = 0.75 + 0.25 * u(r);
            const bool near = kind == 4 && u(r) < 0.5;
            for (double& x : n) x = near ? 0.374 + 0.63 * u(r) : x * scale / l;
        }
        for (int k = 0; k < 3; ++k) a[k] = n[k];
        order(a);
        if (a[0] + a[1] + a[2] > 2.999 || a[2] < std::pow(2, -59.9)) continue;
        if (kind > 0 && u(r) < 0.4) {                    // at and beside the case boundaries
            const quad half = ((quad)a[0] + a[1] + a[2]) / 2;
            const quad at[5] = {a[0], a[1], a[2], (quad)a[0] + a[1], half};
            quad d = at[(int)(5 * u(r))] + std::pow(10, -17 * u(r)) * (u(r) < 0.5 ? -a[0] : a[0]);
            d = d < 0 ? 0 : d > half ? half : d;
            v = std::fmin((double)volume(d, a[0], a[1], a[2]), 0.5);
            v = std::fmax(v, std::pow(2, -96));
            if (u(r) < 0.5) v = 1 - v;
        }
        u64 b[4], o;
        for (int k = 0; k < 3; ++k) memcpy(&b[k], &n[k], 8);
        memcpy(&b[3], &v, 8);
        if (!offset(b[0], b[1], b[2], b[3], o)) {
            ++refused;
            continue;
        }
        double d0;
        memcpy(&d0, &o, 8);
        const double unit = std::pow(2, -std::ilogb(a[2]) - 1);
        for (double& x : n) x *= unit;
        const double err = (double)qabs((quad)(d0 * unit) - solve(n, v));
        if (!(err <= worst)) worst = err;
    }
    printf("%ld %.4g %ld\n", refused, worst, bad_shifts);
    return 0;
}
