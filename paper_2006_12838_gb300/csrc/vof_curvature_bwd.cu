// vof_curvature_bwd.cu -- vector-Jacobian product of the curvature step
// (Sec. 4.2, Appendix B) with respect to the fill field:
//   g_phi = d(sum_k g_kappa[k] kappa[k]) / d phi,
// with the interface set (the list and the 0 < phi < 1 flags of the stencil)
// held fixed.
//
// Per interface cell (k_vof_curvature_vjp, one thread) the forward step is
// recomputed and reversed:
//   kappa = s N / (1 + H^2 + I^2)^(3/2), N = A (I^2+1) + B (H^2+1) - C H I (Eq. 42)
//     -> pbar = dkappa/d(A,B,C,H,I) * g_kappa
//   M p = b (leading block, Appendix B)  ->  bbar = M^-1 pbar (same LDL^T factors),
//     Mbar = -bbar p^T
//   M = sum Q Q^T, b = sum z Q  ->  Qbar_i = bbar (z_i - p.Q_i) - p (bbar.Q_i),
//     zbar_i = bbar.Q_i; Q = (x^2, y^2, xy, x, y) -> xbar_i, ybar_i
//   x_i = e_i.b_x, y_i = e_i.b_y, z_i = e_i.n + d0_i - d0_0 (Eq. 36)
//   d0_i = d0(phi_i, n): dd0/dphi = 1/A_i, dd0/dn = c_i (cut-polygon area and
//     centroid, implicit function theorem on Eq. 1)
//   b_x = b_y x n, b_y = u/|u|, u = n x r (Sec. 4.2)
//   n = -g/|g|, g = sum w_i e_i phi_i (Eq. 38)
// The 27 partial derivatives of each cell go to the workspace; then
// k_curv_gather sums, for every field cell j in a stencil, the entries of the
// (at most 27) listed cells whose stencil contains j, in a fixed order --
// deterministic, no floating-point atomics -- and writes 0 everywhere else.
// Which cells j those are is marked in one bit per field cell; the marks live
// in g_phi itself (the first words of each run of 1024 cells, read by the one
// warp that then writes the run; where g_phi overlaps an input, as in a gradient in
// place, they are set by a kernel of their own once the reverse pass has read it).  The map from a field cell to its list entry
// is not cleared: entry s of cell c counts only if idx[s] == c.
// Only the foot-point variant (Eq. 36) is differentiated.
//
// 42 M cells, 115 704 of them listed: reverse pass 104 (eight lanes per cell, the
// normal, frame and fit repeated in each) -> 30 us, gather 118 (27 x 27 map
// look-ups per listed cell) and two clears of 168 MB (50) -> 4 + 47.5 us; bound
// below by the write of g_phi (25 us).
#include <type_traits>

#include "host_common.h"
#include "plic_pair.cuh"
#include "vof_curvature_coop.cuh"
#include "vof_curvature_pair.cuh"

namespace plic {

constexpr int CB_THREADS = 128;

// f(std::integral_constant<int, I>) for I = FROM..TO-1
template <int FROM, int TO, typename F>
__device__ __forceinline__ void for_range(F&& f) {
    if constexpr (FROM < TO) {
        f(std::integral_constant<int, FROM>{});
        for_range<FROM + 1, TO>(f);
    }
}
constexpr int RUN = 1024;             // cells per run of g_phi (one warp of the gather)

__device__ __forceinline__ void cross3(float ax, float ay, float az, float bx, float by, float bz,
                                       float& cx, float& cy, float& cz) {
    cx = ay * bz - az * by;
    cy = az * bx - ax * bz;
    cz = ax * by - ay * bx;
}

// The marks of the cells of a run: bit j % 32 of word (j / 32) % 32 of the run.
__device__ __forceinline__ unsigned* mark_word(float* g_phi, unsigned j) {
    return reinterpret_cast<unsigned*>(g_phi) + (j & ~(unsigned)(RUN - 1)) + ((j >> 5) & 31u);
}

__global__ void __launch_bounds__(256)
k_curv_clear_marks(float* __restrict__ g_phi, int64_t cells) {
    const int64_t words = (cells + 31) / 32;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words;
         w += (int64_t)gridDim.x * blockDim.x)
        *mark_word(g_phi, (unsigned)(32 * w)) = 0u;
}

// Marks the 27 cells of the stencil of cell c: three bits per row.
__device__ __forceinline__ void mark_stencil(float* g_phi, int c, int nx, int nxy) {
#pragma unroll
    for (int r = 0; r < 9; ++r) {
        const unsigned j = (unsigned)(c + (r % 3 - 1) * nx + (r / 3 - 1) * nxy - 1);
        const unsigned sh = j & 31u;
        atomicOr(mark_word(g_phi, j), 7u << sh);
        if (sh > 29u) atomicOr(mark_word(g_phi, j + 2u), 7u >> (32u - sh));
    }
}

__global__ void __launch_bounds__(256)
k_curv_mark(const int32_t* __restrict__ idx, int64_t n, const int64_t* __restrict__ d_n, int nx, int nxy,
            float* __restrict__ g_phi) {
    const int64_t lim = d_n && *d_n < n ? *d_n : n;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < lim; k += (int64_t)gridDim.x * blockDim.x)
        mark_stencil(g_phi, __ldg(idx + k), nx, nxy);
}

// Area and centroid of the cut polygons of a cell's planes (all with the
// normal n): area_centroid() of plic_polygon.cuh with what depends on the
// normal alone kept, every case evaluated and selected, and the centroid left
// in the order of the sorted normal, without its signs (unsort()).
struct CellArea {
    float n1, n2, n3, n12, half, nn, r1, r2, r3;
    int rx, ry, rz;
    bool sx, sy, sz;
    __device__ __forceinline__ void prepare(float nx, float ny, float nz) {
        const float ax = fabsf(nx), ay = fabsf(ny), az = fabsf(nz);
        n1 = fminf(fminf(ax, ay), az);
        n3 = fmaxf(fmaxf(ax, ay), az);
        n2 = fmaxf(fminf(ax, ay), fminf(fmaxf(ax, ay), az));
        n12 = n1 + n2;
        half = 0.5f * (ax + ay + az);
        nn = Fm<float>::sqrt_(n1 * n1 + n2 * n2 + n3 * n3);
        r1 = n1 > 0.0f ? rcp_approx(n1) : 0.0f;
        r2 = n2 > 0.0f ? rcp_approx(n2) : 0.0f;
        r3 = rcp_approx(n3);
        rx = (ax > ay) + (ax > az); ry = (ay >= ax) + (ay > az); rz = (az >= ax) + (az >= ay);
        sx = nx < 0.0f; sy = ny < 0.0f; sz = nz < 0.0f;
    }
    // area A (false for none) and the centroid's sorted components from the
    // cube's centre, as if n had no negative component
    __device__ __forceinline__ bool eval(float d0, float& A, float c[3]) const {
        const float d = half - fabsf(d0);
        const float e2 = fmaxf(d - n2, 0.0f), e3 = fmaxf(d - n3, 0.0f);
        const float e22 = e2 * e2, e33 = e3 * e3;
        const float cub = (e22 * e2 + e33 * e3) * r1;
        const float N = 3.0f * d * (d - n1) + n1 * n1 - cub;
        const float G = 6.0f * d - 3.0f * n1 - 3.0f * (e22 + e33) * r1;
        const float iG = rcp_approx(G), r23 = r2 * r3;
        const bool c1 = d < n1, c5 = d >= n12;
        float vp = G * (1.0f / 6.0f) * r23;
        c[0] = (3.0f * d - 2.0f * n1 - cub * r1) * iG;
        c[1] = (N * r2 - 3.0f * e22 * r1) * iG;
        c[2] = (N * r3 - 3.0f * e33 * r1) * iG;
        const float t = d * (1.0f / 3.0f);
        vp = c1 ? 0.5f * d * d * r1 * r23 : vp;
        c[0] = c1 ? t * r1 : c[0]; c[1] = c1 ? t * r2 : c[1]; c[2] = c1 ? t * r3 : c[2];
        vp = c5 ? r3 : vp;
        c[0] = c5 ? 0.5f : c[0]; c[1] = c5 ? 0.5f : c[1]; c[2] = c5 ? (d - 0.5f * n12) * r3 : c[2];
        A = nn * vp;
        const bool mirror = d0 > 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) c[k] = mirror ? 0.5f - c[k] : c[k] - 0.5f;
        return d > 0.0f && A > 0.0f;
    }
    __device__ __forceinline__ void unsort(const float v[3], float& x, float& y, float& z) const {
        x = rx == 0 ? v[0] : (rx == 1 ? v[1] : v[2]);
        y = ry == 0 ? v[0] : (ry == 1 ? v[1] : v[2]);
        z = rz == 0 ? v[0] : (rz == 1 ? v[1] : v[2]);
        if (sx) x = -x;
        if (sy) y = -y;
        if (sz) z = -z;
    }
};

// One thread per list entry (as the forward kernel, vof_curvature_tpc.cu):
// two neighbours per trip in the forward loop, whose offsets stay in the
// entry's row of shared memory for the reverse loop, which leaves the entry's
// partial derivatives there; the block then writes its rows out together.
// The thread also marks its stencil in g_phi (unless that is null) and enters itself into
// the map.
template <int METHOD, int FIT>
__global__ void __launch_bounds__(CB_THREADS)
k_vof_curvature_vjp(const float* __restrict__ phi, int nx, int ny, const int32_t* __restrict__ idx,
                    int64_t n, const int64_t* __restrict__ d_n, const float* __restrict__ g_kappa,
                    float* __restrict__ contrib, int32_t* __restrict__ slot, float* __restrict__ g_phi,
                    uint32_t flags) {
    __shared__ float rows[CB_THREADS * 27];
    __shared__ E27Shared tab;
    tab.fill();
    int64_t lim = n;
    if (d_n) {
        const int64_t dn = *d_n;
        lim = dn < n ? dn : n;
    }
    const bool cm = (flags & PLIC_FLAG_NORMAL_CM) != 0;
    const float sgn = (flags & PLIC_FLAG_KAPPA_PAPER_SIGN) ? 1.0f : -1.0f;
    const int nxy = nx * ny;
    float* row = rows + threadIdx.x * 27;
    for (int64_t k0 = (int64_t)blockIdx.x * CB_THREADS; k0 < lim; k0 += (int64_t)gridDim.x * CB_THREADS) {
        const int64_t k = k0 + threadIdx.x;
        const bool on = k < lim;
        const int c = on ? __ldg(idx + k) : 0;
        const float gk = on ? __ldg(g_kappa + k) : 0.0f;
        const float* p0 = phi + c;
        float gx = 0.0f, gy = 0.0f, gz = 0.0f, phi0 = 0.0f;
        unsigned mask = 0u;
        if (on) {
            slot[c] = (int32_t)k;
            phi0 = __ldg(p0);
            if (g_phi) mark_stencil(g_phi, c, nx, nxy);
            for_e27<1>([&](auto I) {
                constexpr int i = decltype(I)::value;
                constexpr int p = E27Table::v[i];
                constexpr int ex = p % 3 - 1, ey = (p / 3) % 3 - 1, ez = p / 9 - 1;
                constexpr int e2 = ex * ex + ey * ey + ez * ez;
                constexpr float wpy = e2 == 1 ? 4.0f : (e2 == 2 ? 2.0f : 1.0f);
                const float v = __ldg(p0 + (ex + ey * nx + ez * nxy));
                const float w = cm ? 1.0f : wpy;
                if (ex != 0) gx = fmaf(w * (float)ex, v, gx);
                if (ey != 0) gy = fmaf(w * (float)ey, v, gy);
                if (ez != 0) gz = fmaf(w * (float)ez, v, gz);
                if (__float_as_uint(v) - 1u < 0x3F7FFFFFu) mask |= 1u << i;
            });
        }
#pragma unroll
        for (int i = 0; i < 27; ++i) row[i] = 0.0f;
        const float gl = sqrtf(gx * gx + gy * gy + gz * gz);
        float gbx = 0.0f, gby = 0.0f, gbz = 0.0f;
        const int m = __popc(mask);
        // (a listed cell whose own fill is not finite has no gradient)
        if (gl > 0.0f && gk != 0.0f && m > 0 && fabsf(phi0) <= 3.40282347e38f) {
            const float inv = -1.0f / gl;
            const float nx_ = gx * inv, ny_ = gy * inv, nz_ = gz * inv;
            // ---- frame: u = n x r, b_y = u/|u|, b_x = b_y x n (Sec. 4.2) ----
            float rx = 0.56270900f, ry = 0.32704452f, rz = 0.75921047f, ux, uy, uz;
            cross3(nx_, ny_, nz_, rx, ry, rz, ux, uy, uz);
            float u2 = ux * ux + uy * uy + uz * uz;
            if (!(u2 > 1e-12f)) {
                rx = 0.32704452f; ry = 0.75921047f; rz = 0.56270900f;
                cross3(nx_, ny_, nz_, rx, ry, rz, ux, uy, uz);
                u2 = ux * ux + uy * uy + uz * uz;
            }
            const float iu = 1.0f / sqrtf(u2);
            const float byx = ux * iu, byy = uy * iu, byz = uz * iu;
            float bxx, bxy, bxz;
            cross3(byx, byy, byz, nx_, ny_, nz_, bxx, bxy, bxz);
            // ---- points (Eq. 36) and normal equations ----
            CellPlic<METHOD> pl;
            pl.prepare(nx_, ny_, nz_);
            const float d00 = pl.offset(phi0);
            float rec[20];
#pragma unroll
            for (int q = 0; q < 20; ++q) rec[q] = 0.0f;
#pragma unroll 1
            for (unsigned list = mask; list;) {
                const int i1 = __ffs(list) - 1;
                list &= list - 1u;
                const bool two = list != 0u;
                const int i2 = two ? __ffs(list) - 1 : i1;
                list &= list - 1u;
                const int4 e1 = tab.ei[i1], e2 = tab.ei[i2];
                const float4 f[2] = {tab.ef[i1], tab.ef[i2]};
                const p2::f2 d = offset_two<METHOD>(
                    pl, make_float2(__ldg(p0 + (e1.x + e1.y * nx + e1.z * nxy)),
                                    __ldg(p0 + (e2.x + e2.y * nx + e2.z * nxy))));
                row[i1] = d.x;
                row[i2] = d.y;
                const float dd[2] = {d.x, d.y};
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const float w = (j == 0 || two) ? 1.0f : 0.0f;
                    const float x = w * (f[j].x * bxx + f[j].y * bxy + f[j].z * bxz);
                    const float y = w * (f[j].x * byx + f[j].y * byy + f[j].z * byz);
                    const float z = w * (f[j].x * nx_ + f[j].y * ny_ + f[j].z * nz_ + (dd[j] - d00));
                    const float Q[5] = {x * x, y * y, x * y, x, y};
#pragma unroll
                    for (int a = 0; a < 5; ++a) {
#pragma unroll
                        for (int b = a; b < 5; ++b)
                            if (a != 2) rec[uidx(a, b)] = fmaf(Q[a], Q[b], rec[uidx(a, b)]);
                        rec[15 + a] = fmaf(z, Q[a], rec[15 + a]);
                    }
                }
            }
            rec[uidx(2, 2)] = rec[uidx(0, 1)];
            rec[uidx(2, 3)] = rec[uidx(0, 4)];
            rec[uidx(2, 4)] = rec[uidx(1, 3)];
            // ---- fit, Eq. 42 backward, b bar = M^-1 p bar ----
            typename std::conditional<FIT == FIT_AUTO, LdltAuto, Ldlt<FIT>>::type fac;
            float p[5], bb[5];
            fac.factor(rec, m);
            if (fac.dim > 0) {
                fac.solve(rec + 15, p);
                const float A = p[0], B = p[1], C = p[2], H = p[3], I = p[4];
                const float w = 1.0f + H * H + I * I;
                const float rw = rsqrtf(w);
                const float iD = rw * rw * rw;                    // (1+H^2+I^2)^(-3/2)
                const float N = A * (I * I + 1.0f) + B * (H * H + 1.0f) - C * H * I;
                const float sg = sgn * gk * iD;
                float pbar[5];
                pbar[0] = sg * (I * I + 1.0f);
                pbar[1] = sg * (H * H + 1.0f);
                pbar[2] = -sg * H * I;
                pbar[3] = sg * (2.0f * B * H - C * I - 3.0f * H * N / w);
                pbar[4] = sg * (2.0f * A * I - C * H - 3.0f * I * N / w);
                fac.solve(pbar, bb);
                // ---- reverse pass over the points ----
                float xs[3] = {0.0f, 0.0f, 0.0f}, ys[3] = {0.0f, 0.0f, 0.0f}, zs[3] = {0.0f, 0.0f, 0.0f};
                float cs[3] = {0.0f, 0.0f, 0.0f}, d00b = 0.0f;    // centroid sums, sorted
                CellArea ar;
                ar.prepare(nx_, ny_, nz_);
#pragma unroll 1
                for (unsigned list = mask; list; list &= list - 1u) {
                    const int i = __ffs(list) - 1;
                    const float4 f = tab.ef[i];
                    const float d0 = row[i];
                    const float x = f.x * bxx + f.y * bxy + f.z * bxz;
                    const float y = f.x * byx + f.y * byy + f.z * byz;
                    const float z = f.x * nx_ + f.y * ny_ + f.z * nz_ + (d0 - d00);
                    const float Q[5] = {x * x, y * y, x * y, x, y};
                    float pQ = 0.0f, bQ = 0.0f;
#pragma unroll
                    for (int a = 0; a < 5; ++a) {
                        pQ = fmaf(p[a], Q[a], pQ);
                        bQ = fmaf(bb[a], Q[a], bQ);
                    }
                    const float res = z - pQ;
                    float Qb[5];
#pragma unroll
                    for (int a = 0; a < 5; ++a) Qb[a] = bb[a] * res - p[a] * bQ;
                    const float xb = 2.0f * x * Qb[0] + y * Qb[2] + Qb[3];
                    const float yb = 2.0f * y * Qb[1] + x * Qb[2] + Qb[4];
                    xs[0] += xb * f.x; xs[1] += xb * f.y; xs[2] += xb * f.z;
                    ys[0] += yb * f.x; ys[1] += yb * f.y; ys[2] += yb * f.z;
                    zs[0] += bQ * f.x; zs[1] += bQ * f.y; zs[2] += bQ * f.z;
                    d00b -= bQ;
                    // d0_i = d0(phi_i, n): dd0/dphi = 1/A_i, dd0/dn = c_i
                    float Ai, cc[3];
                    const bool cut = ar.eval(d0, Ai, cc);
                    row[i] = cut ? bQ / Ai : 0.0f;
#pragma unroll
                    for (int a = 0; a < 3; ++a) cs[a] += cut ? bQ * cc[a] : 0.0f;
                }
                {   // the centre's d0 = d0(phi_0, n)
                    float A0, cc[3];
                    if (ar.eval(d00, A0, cc)) {
                        row[0] = d00b / A0;
#pragma unroll
                        for (int a = 0; a < 3; ++a) cs[a] += d00b * cc[a];
                    }
                }
                float nbx, nby, nbz, tx, ty, tz;
                ar.unsort(cs, nbx, nby, nbz);
                nbx += zs[0]; nby += zs[1]; nbz += zs[2];
                // ---- frame backward: b_x = b_y x n ----
                cross3(xs[0], xs[1], xs[2], byx, byy, byz, tx, ty, tz);  // nbar += bxbar x b_y
                nbx += tx; nby += ty; nbz += tz;
                cross3(nx_, ny_, nz_, xs[0], xs[1], xs[2], tx, ty, tz);  // bybar += n x bxbar
                const float bybx = ys[0] + tx, byby = ys[1] + ty, bybz = ys[2] + tz;
                // b_y = u/|u|, u = n x r
                const float dp = byx * bybx + byy * byby + byz * bybz;
                const float ubx = (bybx - byx * dp) * iu, uby = (byby - byy * dp) * iu,
                            ubz = (bybz - byz * dp) * iu;
                cross3(rx, ry, rz, ubx, uby, ubz, tx, ty, tz);           // nbar += r x ubar
                nbx += tx; nby += ty; nbz += tz;
                // ---- normal backward: n = -g/|g| ----
                const float s = nx_ * nbx + ny_ * nby + nz_ * nbz;
                gbx = (nbx - nx_ * s) * inv; gby = (nby - ny_ * s) * inv; gbz = (nbz - nz_ * s) * inv;
            } else {
#pragma unroll
                for (int i = 0; i < 27; ++i) row[i] = 0.0f;
            }
        }
        // ---- Parker-Youngs backward: the entry's 27 partial derivatives ----
        for_e27<1>([&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int p = E27Table::v[i];
            constexpr int ex = p % 3 - 1, ey = (p / 3) % 3 - 1, ez = p / 9 - 1;
            constexpr int e2 = ex * ex + ey * ey + ez * ez;
            const float wi = cm ? 1.0f : (e2 == 1 ? 4.0f : (e2 == 2 ? 2.0f : 1.0f));
            row[i] += wi * ((float)ex * gbx + (float)ey * gby + (float)ez * gbz);
        });
        __syncthreads();
        const int cnt = (int)(lim - k0 < CB_THREADS ? lim - k0 : CB_THREADS) * 27;
        for (int t = threadIdx.x; t < cnt; t += CB_THREADS) contrib[k0 * 27 + t] = rows[t];
        __syncthreads();
    }
}

// g_phi[j] = sum over the 27 offsets o of contrib[slot[j - e_o]][o] (when cell
// j - e_o is in the list), in the fixed order o = 0..26, for the marked cells j;
// 0 for all others.  A block takes GATHER_RUNS runs of 1024 cells: its warps
// read the runs' marks and clear the runs, then the block lists the marked cells
// in shared memory (GATHER_LIST at a time) and gives one to each thread: the
// look-ups are a chain of dependent loads, so the block needs cells enough for
// all its threads (marked cells are a percent of a field, and crowd where the
// interface lies along x; 42 M cells: one warp taking those of its own run 84 us,
// a block of eight runs 78 us, of 32 47.5 us; all 27 look-ups of a cell in flight
// instead of nine, at more registers, 64 us).  A listed cell has its whole stencil
// in the field, so j - e_o is a listed cell only where it lies in the field beside j.
constexpr int GATHER_RUNS = 32, GATHER_LIST = 4096, GATHER_PER = GATHER_RUNS / 8;

__global__ void __launch_bounds__(256, 4)
k_curv_gather(const int32_t* __restrict__ idx, int64_t n, const int64_t* __restrict__ d_n,
              const int32_t* __restrict__ slot, const float* __restrict__ contrib, int nx, int ny,
              int64_t cells, float* __restrict__ g_phi, int vec) {
    __shared__ unsigned short list[GATHER_LIST];     // cell - first cell of the block's runs
    __shared__ int s_total[8];
    int64_t lim = n;
    if (d_n) {
        const int64_t dn = *d_n;
        lim = dn < n ? dn : n;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nxy = nx * ny;
    const unsigned ncell = (unsigned)cells;
    const int64_t nrun = (cells + RUN - 1) / RUN;
    for (int64_t r0 = (int64_t)blockIdx.x * GATHER_RUNS; r0 < nrun; r0 += (int64_t)gridDim.x * GATHER_RUNS) {
        // warp w has runs w, w + 8, ..; lane l the l-th word of each
        unsigned w[GATHER_PER];
        int cnt = 0;
#pragma unroll
        for (int i = 0; i < GATHER_PER; ++i) {
            const int64_t c = (r0 + 8 * i + warp) * RUN + 32 * lane;
            w[i] = c < cells ? *mark_word(g_phi, (unsigned)c) : 0u;
            cnt += __popc(w[i]);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < GATHER_PER; ++i) {
            const int64_t j0 = (r0 + 8 * i + warp) * RUN;
            if (vec && j0 + RUN <= cells) {
#pragma unroll
                for (int u = 0; u < RUN / 128; ++u)
                    reinterpret_cast<float4*>(g_phi + j0)[32 * u + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            } else {
                for (int64_t j = j0 + lane; j < j0 + RUN && j < cells; j += 32) g_phi[j] = 0.0f;
            }
        }
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) s_total[warp] = incl;
        __syncthreads();                             // (and the clears before the sums)
        int first = incl - cnt, total = 0;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            first += v < warp ? s_total[v] : 0;
            total += s_total[v];
        }
        for (int base = 0; base < total; base += GATHER_LIST) {
            int at = first - base;
#pragma unroll
            for (int i = 0; i < GATHER_PER; ++i)
                for (unsigned b = w[i]; b; b &= b - 1u, ++at)
                    if (at >= 0 && at < GATHER_LIST)
                        list[at] = (unsigned short)(RUN * (8 * i + warp) + 32 * lane + __ffs(b) - 1);
            __syncthreads();
            const int part = total - base < GATHER_LIST ? total - base : GATHER_LIST;
            for (int t = threadIdx.x; t < part; t += 256) {
                const unsigned j = (unsigned)(r0 * RUN) + list[t];
                float acc = 0.0f;
                // nine map entries, then their list entries, then the partial
                // derivatives, each nine loads in flight
                for_range<0, 3>([&](auto bc) {
                    constexpr int b = 9 * decltype(bc)::value;
                    unsigned src[9], sl[9];
                    int li[9];
                    float v[9];
                    for_range<0, 9>([&](auto ic) {
                        constexpr int i = decltype(ic)::value;
                        int ex, ey, ez;
                        e_of_c<b + i>(ex, ey, ez);
                        src[i] = j - (unsigned)(ex + ey * nx + ez * nxy);
                        sl[i] = src[i] < ncell ? (unsigned)__ldg(slot + src[i]) : 0xffffffffu;
                    });
    #pragma unroll
                    for (int i = 0; i < 9; ++i) li[i] = sl[i] < lim ? __ldg(idx + sl[i]) : -1;
    #pragma unroll
                    for (int i = 0; i < 9; ++i)
                        v[i] = sl[i] < lim && (unsigned)li[i] == src[i] ? __ldg(contrib + (int64_t)sl[i] * 27 + b + i)
                                                                        : 0.0f;
    #pragma unroll
                    for (int i = 0; i < 9; ++i) acc += v[i];
                });
                g_phi[j] = acc;
            }
            __syncthreads();                         // the list is used again
        }
        __syncthreads();                             // and the totals
    }
}

template <int METHOD>
static const void* pick_vjp(int fit) {
    switch (fit) {
        case FIT_FP32: return reinterpret_cast<const void*>(&k_vof_curvature_vjp<METHOD, FIT_FP32>);
        case FIT_DF32: return reinterpret_cast<const void*>(&k_vof_curvature_vjp<METHOD, FIT_DF32>);
        case FIT_FP64: return reinterpret_cast<const void*>(&k_vof_curvature_vjp<METHOD, FIT_FP64>);
        default: return reinterpret_cast<const void*>(&k_vof_curvature_vjp<METHOD, FIT_AUTO>);
    }
}

}  // namespace plic

extern "C" size_t plic_curv_bwd_workspace_bytes(int64_t cells, int64_t n_iface) {
    if (cells < 0 || n_iface < 0) return 0;
    const size_t a = ((size_t)cells * sizeof(int32_t) + 255) / 256 * 256;
    const size_t b = ((size_t)n_iface * 27 * sizeof(float) + 255) / 256 * 256;
    return a + b;
}

extern "C" plic_status vof_curvature_backward(const float* phi, int nx, int ny, int nz,
                                              const int32_t* idx, int64_t n_iface,
                                              const int64_t* d_n_iface, const float* g_kappa,
                                              float* g_phi, plic_method m, uint32_t flags,
                                              void* workspace, size_t ws_bytes, void* stream) {
    using namespace plic;
    if (nx < 3 || ny < 3 || nz < 3 || n_iface < 0) return PLIC_ERR_ARG;
    if ((int)m < 0 || (int)m > 4) return PLIC_ERR_ARG;
    const uint32_t known = PLIC_FLAG_POINT_CENTROID | PLIC_FLAG_KAPPA_PAPER_SIGN |
                           PLIC_FLAG_FIT_FP32 | PLIC_FLAG_FIT_DF32 | PLIC_FLAG_FIT_FP64 |
                           PLIC_FLAG_NORMAL_CM | PLIC_FLAG_NEIGHBOR_NORMAL;
    const uint32_t fitf = flags & (PLIC_FLAG_FIT_FP32 | PLIC_FLAG_FIT_DF32 | PLIC_FLAG_FIT_FP64);
    if ((flags & ~known) || (fitf & (fitf - 1u))) return PLIC_ERR_ARG;
    if (flags & (PLIC_FLAG_POINT_CENTROID | PLIC_FLAG_NEIGHBOR_NORMAL)) return PLIC_ERR_UNSUPPORTED;
    const int64_t cells = (int64_t)nx * ny * nz;
    if (cells > 2147483647LL) return PLIC_ERR_ARG;
    if (!phi || !g_phi || (n_iface > 0 && (!idx || !g_kappa)) || !workspace) return PLIC_ERR_ARG;
    if (ws_bytes < plic_curv_bwd_workspace_bytes(cells, n_iface)) return PLIC_ERR_ARG;
    if (!aligned(phi, 4) || !aligned(g_phi, 4) || (idx && !aligned(idx, 4)) ||
        (g_kappa && !aligned(g_kappa, 4)) || !aligned(workspace, 256) ||
        (d_n_iface && !aligned(d_n_iface, 8)))
        return PLIC_ERR_ALIGN;
    cudaStream_t s = as_stream(stream);
    char* ws = reinterpret_cast<char*>(workspace);
    int32_t* slot = reinterpret_cast<int32_t*>(ws);
    float* contrib = reinterpret_cast<float*>(ws + ((size_t)cells * sizeof(int32_t) + 255) / 256 * 256);
    if (n_iface == 0) {
        const cudaError_t e = cudaMemsetAsync(g_phi, 0, (size_t)cells * sizeof(float), s);
        if (e != cudaSuccess) { set_last_error("vof_curvature_backward", e); return PLIC_ERR_CUDA; }
        return check_launch("vof_curvature_backward");
    }
    const int cg = stride_grid(reinterpret_cast<const void*>(&k_curv_clear_marks), 256, (cells + 31) / 32);
    // the reverse pass reads phi and g_kappa: marks in g_phi before or during it only where
    // they lie elsewhere
    auto inside = [&](const float* p, int64_t count) {
        const uintptr_t a = (uintptr_t)p, g = (uintptr_t)g_phi;
        return a < g + (uintptr_t)cells * sizeof(float) && g < a + (uintptr_t)count * sizeof(float);
    };
    const bool in_place = inside(phi, cells) || inside(g_kappa, n_iface);
    float* marks = in_place ? nullptr : g_phi;
    if (marks) k_curv_clear_marks<<<cg, 256, 0, s>>>(marks, cells);
    // the same fit policy as the forward call: adaptive unless a FIT flag is given
    const int fit = (flags & PLIC_FLAG_FIT_DF32) ? FIT_DF32 : (flags & PLIC_FLAG_FIT_FP32) ? FIT_FP32
                  : (flags & PLIC_FLAG_FIT_FP64) ? FIT_FP64 : FIT_AUTO;
    const void* k = nullptr;
    switch (m) {
        case PLIC_ANALYTIC: k = pick_vjp<M_ANALYTIC>(fit); break;
        case PLIC_SZ_ORIG: k = pick_vjp<M_SZ_ORIG>(fit); break;
        case PLIC_SZ_OPT: k = pick_vjp<M_SZ_OPT>(fit); break;
        case PLIC_NEWTON: k = pick_vjp<M_NEWTON>(fit); break;
        case PLIC_NESTED: k = pick_vjp<M_NESTED>(fit); break;
    }
    const int grid = stride_grid(k, CB_THREADS, n_iface);
    void* args[] = {(void*)&phi, (void*)&nx, (void*)&ny, (void*)&idx, (void*)&n_iface,
                    (void*)&d_n_iface, (void*)&g_kappa, (void*)&contrib, (void*)&slot, (void*)&marks,
                    (void*)&flags};
    const cudaError_t e = cudaLaunchKernel(k, dim3(grid), dim3(CB_THREADS), args, 0, s);
    if (e != cudaSuccess) { set_last_error("vof_curvature_backward", e); return PLIC_ERR_CUDA; }
    if (in_place) {
        k_curv_clear_marks<<<cg, 256, 0, s>>>(g_phi, cells);
        const int mg = stride_grid(reinterpret_cast<const void*>(&k_curv_mark), 256, n_iface);
        k_curv_mark<<<mg, 256, 0, s>>>(idx, n_iface, d_n_iface, nx, nx * ny, g_phi);
    }
    const int vec = aligned(g_phi, 16);
    const int gg = stream_grid(reinterpret_cast<const void*>(&k_curv_gather), 256, (cells + RUN - 1) / RUN * 256 / GATHER_RUNS + 255);
    k_curv_gather<<<gg, 256, 0, s>>>(idx, n_iface, d_n_iface, slot, contrib, nx, ny, cells, g_phi, vec);
    return check_launch("vof_curvature_backward");
}
