// vof_curvature_tpc.cu -- the curvature step (Sec. 4.2, Appendix B) with one
// thread per interface cell, for long interface lists.
//
// The eight-lane layout of vof_curvature_coop.cuh shortens the dependent
// chain of a cell (it wins when the list is too short to fill the GPU), but
// every lane of a group repeats the normal, the frame and the per-normal
// solver constants, and the group reductions add shuffles.  With enough
// cells to fill every warp slot many times over (the batched workload), the
// instruction count decides instead, and one thread per cell does each step
// once:
//   - the 27 stencil values with compile-time offsets, the Parker-Youngs (or
//     centre-of-mass) sums in registers and the list of the interface neighbours in
//     shared memory;
//   - normal, frame, centre offset d0(phi_0, n) and the per-normal constants
//     of the solver once;
//   - a loop over that list only (Eq. 36), two neighbours per trip: their
//     offsets are solved together (paired FP32
//     instructions for the optimised SZ solution), their points accumulated
//     into the normal equations in registers;
//   - the 5x5 solve of the fit precision and Eq. 42, as in the lane phase of
//     the eight-lane layout (co_solve).
// The results equal those of the eight-lane layout up to the summation order
// of the stencil sums and of the normal equations.
#include "host_common.h"
#include "vof_curvature_coop.cuh"
#include "vof_curvature_pair.cuh"

namespace plic {

// kappa (sign per flags) of interface cell c of a field, one thread.  sv: the
// thread's column of 28 entries in shared memory, TPC_THREADS apart.  The prologue
// lists the interface neighbours there as it reads them, each with its value and the
// byte offset of its direction in tab.ef (one 8-byte word per lane, conflict-free), and
// the loop takes two entries per trip.  Reading each value from the field again through
// a table of integer directions cost the address arithmetic and a load of five or six
// wavefronts: batch of 64 fields, 2.6 M cells, 216.5 us; all 27 values in the
// column and the neighbours from the bits of a mask 200.3; this list 198.1 (1 GiB
// field with its compaction 215.5 -> 212).
template <int METHOD, int FIT>
__device__ __forceinline__ float tpc_kappa(const float* __restrict__ phi, int nx, int64_t nxy,
                                           int64_t c, uint32_t flags, const E27Shared& tab, float2* sv) {
    const bool cm = (flags & PLIC_FLAG_NORMAL_CM) != 0;
    const float* p0 = phi + c;
    // offsets within the field in 32 bits (list entries are int32 cell indices)
    const int nxy32 = (int)nxy;
    // 1. stencil: normal sums (Eq. 38 weights or all 1) and the interface neighbours
    float gx = 0.0f, gy = 0.0f, gz = 0.0f;
    const float phi0 = __ldg(p0);
    float2* tail = sv;
    for_e27<1>([&](auto I) {
        constexpr int i = decltype(I)::value;
        constexpr int p = E27Table::v[i];
        constexpr int ex = p % 3 - 1, ey = (p / 3) % 3 - 1, ez = p / 9 - 1;
        constexpr int e2 = ex * ex + ey * ey + ez * ez;
        constexpr float wpy = e2 == 1 ? 4.0f : (e2 == 2 ? 2.0f : 1.0f);
        const float v = __ldg(p0 + (ex + ey * nx + ez * nxy32));
        const float w = cm ? 1.0f : wpy;
        if (ex != 0) gx = fmaf(w * (float)ex, v, gx);
        if (ey != 0) gy = fmaf(w * (float)ey, v, gy);
        if (ez != 0) gz = fmaf(w * (float)ez, v, gz);
        // 0 < v < 1 as one unsigned compare of the bits: the positive floats
        // below 1.0f are the patterns 1 .. 0x3F7FFFFF
        if (__float_as_uint(v) - 1u < 0x3F7FFFFFu) {
            *tail = make_float2(v, __int_as_float((int)sizeof(float4) * i));
            tail += TPC_THREADS;
        }
    });
    // 2. normal and frame (Sec. 4.2)
    const float gl2 = gx * gx + gy * gy + gz * gz;
    if (!(gl2 > 0.0f)) return 0.0f;                    // undefined normal: kappa = 0
    const float inv = -rsqrtf(gl2);
    const float nx_ = gx * inv, ny_ = gy * inv, nz_ = gz * inv;
    float rx = 0.56270900f, ry = 0.32704452f, rz = 0.75921047f;
    float byx = ny_ * rz - nz_ * ry, byy = nz_ * rx - nx_ * rz, byz = nx_ * ry - ny_ * rx;
    float bl = byx * byx + byy * byy + byz * byz;
    if (!(bl > 1e-12f)) {
        rx = 0.32704452f; ry = 0.75921047f; rz = 0.56270900f;
        byx = ny_ * rz - nz_ * ry; byy = nz_ * rx - nx_ * rz; byz = nx_ * ry - ny_ * rx;
        bl = byx * byx + byy * byy + byz * byz;
    }
    const float ib = rsqrtf(bl);
    byx *= ib; byy *= ib; byz *= ib;
    const float bxx = byy * nz_ - byz * ny_, bxy = byz * nx_ - byx * nz_, bxz = byx * ny_ - byy * nx_;
    // 3. centre offset and, for centroid points, the centre centroid
    CellPlic<METHOD> pl;
    pl.prepare(nx_, ny_, nz_);
    const float d00 = pl.offset(phi0);
    const bool centroid = (flags & PLIC_FLAG_POINT_CENTROID) != 0;
    float c0x = 0.0f, c0y = 0.0f, c0z = 0.0f;
    if (centroid) {
        float A;
        area_centroid<float>(nx_, ny_, nz_, d00, A, c0x, c0y, c0z);
    }
    // 4. interface neighbours (Eq. 36): points and normal equations
    float rec[21];
#pragma unroll
    for (int q = 0; q < 20; ++q) rec[q] = 0.0f;
    rec[20] = (float)((int)(tail - sv) / TPC_THREADS);
    *tail = make_float2(0.5f, __int_as_float(0));
    // two neighbours per trip (in ascending order; an odd last one pairs with
    // the zero point behind the list, which adds nothing: its fill is 1/2, not phi0,
    // which the caller's list may have outside [0, 1], where the paired solve is NaN)
#pragma unroll 1
    for (const float2* r = sv; r < tail; r += 2 * TPC_THREADS) {
        const float2 r1 = r[0], r2 = r[TPC_THREADS];
        const int i1 = __float_as_int(r1.y), i2 = __float_as_int(r2.y);
        const float4 f1 = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(tab.ef) + i1);
        const float4 f2 = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(tab.ef) + i2);
        const p2::f2 d0i = offset_two<METHOD>(pl, make_float2(r1.x, r2.x));
        float qx[2] = {f1.x, f2.x}, qy[2] = {f1.y, f2.y};
        float qz[2] = {f1.z, f2.z}, z[2];
        const float dd[2] = {d0i.x, d0i.y};
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (centroid) {
                float A, cx, cy, cz;
                area_centroid<float>(nx_, ny_, nz_, dd[j], A, cx, cy, cz);
                qx[j] += cx - c0x; qy[j] += cy - c0y; qz[j] += cz - c0z;
                z[j] = qx[j] * nx_ + qy[j] * ny_ + qz[j] * nz_;
                if (j == 1 && i2 == 0) qx[j] = qy[j] = qz[j] = 0.0f;   // d00's rounding in the pair
            } else {
                z[j] = qx[j] * nx_ + qy[j] * ny_ + qz[j] * nz_ + (dd[j] - d00);
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float x = qx[j] * bxx + qy[j] * bxy + qz[j] * bxz;
            const float y = qx[j] * byx + qy[j] * byy + qz[j] * byz;
            const float zz = z[j];
            const float Q[5] = {x * x, y * y, x * y, x, y};
            // the 12 distinct moments of the normal matrix: the entries
            // (xy, xy), (xy, x), (xy, y) equal (x^2, y^2), (x^2, y), (y^2, x)
            // and are copied after the loop
#pragma unroll
            for (int a = 0; a < 5; ++a) {
#pragma unroll
                for (int b = a; b < 5; ++b)
                    if (a != 2) rec[uidx(a, b)] = fmaf(Q[a], Q[b], rec[uidx(a, b)]);
                rec[15 + a] = fmaf(zz, Q[a], rec[15 + a]);
            }
        }
    }
    rec[uidx(2, 2)] = rec[uidx(0, 1)];
    rec[uidx(2, 3)] = rec[uidx(0, 4)];
    rec[uidx(2, 4)] = rec[uidx(1, 3)];
    // 5. fit and Eq. 42
    return co_solve<FIT>(rec, flags);
}

// Single field: thread per list entry, grid-stride.
template <int METHOD, int FIT>
__global__ void __launch_bounds__(TPC_THREADS)
k_vof_curvature_tpc(const float* __restrict__ phi, int nx, int ny, const int32_t* __restrict__ idx,
                    int64_t n, const int64_t* __restrict__ d_n, float* __restrict__ kappa,
                    uint32_t flags, float scale) {
    pdl_wait();                  // a kernel before it (the compaction) has completed
    int64_t lim = n;
    if (d_n) {
        const int64_t dn = *d_n;
        lim = dn < n ? dn : n;
    }
    __shared__ E27Shared tab;
    __shared__ float2 sv[28 * TPC_THREADS];
    tab.fill();
    const int64_t nxy = (int64_t)nx * ny;
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < lim;
         k += (int64_t)gridDim.x * blockDim.x)
        kappa[k] = scale * tpc_kappa<METHOD, FIT>(phi, nx, nxy, (int64_t)__ldg(idx + k), flags, tab, sv + threadIdx.x);
    pdl_trigger();
}

// Persistent batched kernel: each warp claims tickets of `chunk` cells (a
// multiple of 32) of the concatenated lists and gives one cell to each lane.
// Five blocks per SM for the optimised SZ (95 registers; the compiler's 118 leave four).
template <int METHOD, int FIT>
__global__ void __launch_bounds__(TPC_THREADS, METHOD == M_SZ_OPT ? 5 : 0)
k_vof_curvature_batched_tpc(const vof_field* __restrict__ fields, const int64_t* __restrict__ prefix,
                            int n_fields, int64_t total, int chunk,
                            unsigned long long* __restrict__ ticket, uint32_t flags) {
    const int lane = threadIdx.x & 31;
    __shared__ E27Shared tab;
    __shared__ float2 sv[28 * TPC_THREADS];
    tab.fill();
    pdl_wait();                  // the tables are written
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(ticket, (unsigned long long)chunk);
        const int64_t start = (int64_t)__shfl_sync(0xffffffffu, t, 0);
        if (start >= total) break;
        const int64_t end = start + chunk < total ? start + chunk : total;
        // the field of the ticket's first cell, found once per ticket (lane 0,
        // binary search over the list prefix); each lane then steps forward
        // from it to its own cell's field (the lists are long: rarely a step)
        int f0 = 0;
        if (lane == 0) {
            int lo = 0, hi = n_fields - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (__ldg(prefix + mid) <= start) lo = mid; else hi = mid - 1;
            }
            f0 = lo;
        }
        f0 = __shfl_sync(0xffffffffu, f0, 0);
        for (int64_t gi = start + lane; gi < end; gi += 32) {
            int lo = f0;
            while (lo + 1 < n_fields && __ldg(prefix + lo + 1) <= gi) ++lo;
            const int64_t kk = gi - __ldg(prefix + lo);
            const vof_field& F = fields[lo];
            const float k = tpc_kappa<METHOD, FIT>(F.phi, F.nx, (int64_t)F.nx * F.ny,
                                                   (int64_t)__ldg(F.idx + kk), flags, tab, sv + threadIdx.x);
            F.kappa[kk] = k;
        }
    }
}

template <int METHOD>
static const void* pick_tpc(bool batched, int fit) {
#define PLIC_TPC(K) \
    {reinterpret_cast<const void*>(&K<METHOD, FIT_FP64>), reinterpret_cast<const void*>(&K<METHOD, FIT_FP32>), \
     reinterpret_cast<const void*>(&K<METHOD, FIT_DF32>), reinterpret_cast<const void*>(&K<METHOD, FIT_AUTO>)}
    static const void* single[4] = PLIC_TPC(k_vof_curvature_tpc);
    static const void* many[4] = PLIC_TPC(k_vof_curvature_batched_tpc);
#undef PLIC_TPC
    return batched ? many[fit] : single[fit];
}

const void* select_tpc(bool batched, plic_method m, int fit) {
    if (fit < 0 || fit > 3) return nullptr;
    switch (m) {
        case PLIC_ANALYTIC: return pick_tpc<M_ANALYTIC>(batched, fit);
        case PLIC_SZ_ORIG: return pick_tpc<M_SZ_ORIG>(batched, fit);
        case PLIC_SZ_OPT: return pick_tpc<M_SZ_OPT>(batched, fit);
        case PLIC_NEWTON: return pick_tpc<M_NEWTON>(batched, fit);
        case PLIC_NESTED: return pick_tpc<M_NESTED>(batched, fit);
    }
    return nullptr;
}

}  // namespace plic
