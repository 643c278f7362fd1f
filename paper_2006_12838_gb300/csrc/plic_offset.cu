// plic_offset.cu -- batched PLIC inversion d0(V0, n) (Sec. 2, Eq. 1) with the
// five solvers of Sec. 2.3-2.5, and the C entry point plic_offset().
//
// Layout: structure of arrays nx, ny, nz, V0 -> d0.  One thread handles one
// 16-byte vector of each array per step of a grid-stride loop (4 cells in FP32,
// 2 in FP64), so every warp issues fully coalesced 512-byte loads; the grid is
// up to 16 waves of resident blocks (stream_grid: measured faster than one
// persistent wave).  Loads and the store are streaming (evict-first): every
// byte is touched once.
//
// Roofline: 20 B/cell in FP32 (16 in, 4 out), 40 B/cell in FP64.  The closed-form
// FP32 solvers run at the HBM rate (k_plic_offset_pair); in FP64 the optimised SZ and
// the analytic solution are bound by instruction issue (k_plic_offset_fx), the other
// methods by the FP64 pipe.
#include "host_common.h"
#include "plic_fx.cuh"
#include "plic_pair.cuh"
#include "plic_solvers.cuh"

namespace plic {

template <typename T> struct Vec16;
template <> struct Vec16<float> { typedef float4 type; static constexpr int W = 4; };
template <> struct Vec16<double> { typedef double2 type; static constexpr int W = 2; };

template <typename V> __device__ __forceinline__ V ld_stream(const V* p) { return __ldcs(p); }
template <typename V> __device__ __forceinline__ void st_stream(V* p, V v) { __stcs(p, v); }

__device__ __forceinline__ void to_arr(float4 v, float* a) { a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w; }
__device__ __forceinline__ void to_arr(double2 v, double* a) { a[0] = v.x; a[1] = v.y; }
__device__ __forceinline__ float4 from_arr(const float* a) { return make_float4(a[0], a[1], a[2], a[3]); }
__device__ __forceinline__ double2 from_arr(const double* a) { return make_double2(a[0], a[1]); }

__device__ __forceinline__ void count_invalid(int bad, unsigned long long* counter) {
    if (counter == nullptr) return;
    const unsigned mask = __activemask();
    const int tot = __reduce_add_sync(mask, bad);
    const int leader = __ffs(mask) - 1;
    if ((int)(threadIdx.x & 31) == leader && tot > 0) atomicAdd(counter, (unsigned long long)tot);
}

template <int METHOD, typename T, bool POLISH, bool FAITHFUL>
__global__ void __launch_bounds__(256)
k_plic_offset(const T* __restrict__ nx, const T* __restrict__ ny, const T* __restrict__ nz,
              const T* __restrict__ V0, T* __restrict__ d0, int64_t n, int vec_ok,
              unsigned long long* invalid, void* /* round trip: not fused here */) {
    typedef typename Vec16<T>::type VT;
    constexpr int W = Vec16<T>::W;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int bad = 0;
    const int64_t nvec = vec_ok ? n / W : 0;
    for (int64_t i = tid; i < nvec; i += stride) {
        T a[W], b[W], c[W], v[W], r[W];
        to_arr(ld_stream(reinterpret_cast<const VT*>(nx) + i), a);
        to_arr(ld_stream(reinterpret_cast<const VT*>(ny) + i), b);
        to_arr(ld_stream(reinterpret_cast<const VT*>(nz) + i), c);
        to_arr(ld_stream(reinterpret_cast<const VT*>(V0) + i), v);
#pragma unroll
        for (int j = 0; j < W; ++j) r[j] = offset_cell<METHOD, T, POLISH, FAITHFUL>(a[j], b[j], c[j], v[j], bad);
        st_stream(reinterpret_cast<VT*>(d0) + i, from_arr(r));
    }
    for (int64_t i = nvec * W + tid; i < n; i += stride)
        d0[i] = offset_cell<METHOD, T, POLISH, FAITHFUL>(nx[i], ny[i], nz[i], V0[i], bad);
    count_invalid(bad, invalid);
}

// Work-compacted form of k_plic_offset for the default (non-literal) forms of the
// iterative solvers and, in FP64, of Kawano's SZ:
// the warp runs the symmetry front end and the closed-form cases (Eqs. 24-25)
// on its 32 x W cells, then gathers the cells that need the heavy part (the
// trigonometric root of cases (3)/(4), or the Newton / nested-interval
// iterations) into a dense per-warp task list -- one warp vote per cell slot
// and a popcount prefix give each task its place -- and runs the heavy part
// on those tasks only, 32 at a time; the owners then take their results
// back.  Without this every lane of the warp would pass through the heavy
// part whenever any lane needed it (about every time: 40-60 % of random cells
// are in cases (3)/(4)), and lanes with closed-form cells would idle through
// it.  The task list lives in shared memory (4 values per task).
// The symmetry front end of Sec. 2.1 for one double cell on the bit patterns:
// the FP64 kernels are bound by the FP64 pipe, so the sort of |n| (the order
// of non-negative doubles is that of their bits; a NaN sorts last and makes L
// NaN), the validity tests and the choice V = V0 or 1 - V0 (exact) run as
// integer instructions; L keeps the FP64 sum |nx| + |ny| + |nz| in that order.
__device__ __forceinline__ bool front_bits(double nx, double ny, double nz, double V0, double& n1,
                                           double& n2, double& n3, double& L, double& V) {
    const unsigned long long S = 0x8000000000000000ull;
    const unsigned long long ux = (unsigned long long)__double_as_longlong(nx) & ~S;
    const unsigned long long uy = (unsigned long long)__double_as_longlong(ny) & ~S;
    const unsigned long long uz = (unsigned long long)__double_as_longlong(nz) & ~S;
    const unsigned long long lo = ux < uy ? ux : uy, hi = ux < uy ? uy : ux;
    const unsigned long long b1 = lo < uz ? lo : uz, b3 = hi > uz ? hi : uz;
    n1 = __longlong_as_double((long long)b1);
    n3 = __longlong_as_double((long long)b3);
    n2 = __longlong_as_double((long long)(ux ^ uy ^ uz ^ b1 ^ b3));
    L = (__longlong_as_double((long long)ux) + __longlong_as_double((long long)uy)) +
        __longlong_as_double((long long)uz);
    const unsigned long long bv = (unsigned long long)__double_as_longlong(V0), va = bv & ~S;
    const unsigned long long bl = (unsigned long long)__double_as_longlong(L);
    // 0 <= V0 <= 1 (-0 accepted, NaN refused) and 0 < L <= 3
    const bool ok = ((bv >> 63) == 0ull || va == 0ull) && va <= 0x3FF0000000000000ull && bl != 0ull &&
                    bl <= 0x4008000000000000ull;
    V = va <= 0x3FE0000000000000ull ? __longlong_as_double((long long)va) : 1.0 - V0;
    return ok;
}

// |h| with the sign of V0 - 1/2 (+ for V0 >= 1/2), on the bits.
__device__ __forceinline__ double sign_of_side(double h, double V0) {
    const unsigned long long S = 0x8000000000000000ull;
    const unsigned long long va = (unsigned long long)__double_as_longlong(V0) & ~S;
    const unsigned long long m = (unsigned long long)__double_as_longlong(h) & ~S;
    return __longlong_as_double((long long)(va >= 0x3FE0000000000000ull ? m : (m | S)));
}

template <int METHOD, typename T, bool POLISH>
__global__ void __launch_bounds__(256)
k_plic_offset_compact(const T* __restrict__ nx, const T* __restrict__ ny, const T* __restrict__ nz,
                      const T* __restrict__ V0, T* __restrict__ d0, int64_t n, int vec_ok,
                      unsigned long long* invalid, void* /* round trip: not fused here */) {
    typedef typename Vec16<T>::type VT;
    constexpr int W = Vec16<T>::W;
    constexpr bool SZ = METHOD == M_SZ_ORIG;
    typedef Solver<METHOD, T, false> S;
    // FP64: one task list for the block's 8 warps (heavy parts long enough
    // to repay the barriers; only the block's last round is partly empty);
    // FP32: one list per warp, no barriers
    constexpr bool POOL = sizeof(T) == 8;
    // FP64: the front end on the bit patterns (front_bits), except for nested
    // intervals (4-5 % faster for the others, 3 % slower there)
    constexpr bool BITS = sizeof(T) == 8 && METHOD != M_NESTED;
    __shared__ T task[8][32 * W][4];
    __shared__ int wtot[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t wstride = (int64_t)gridDim.x * blockDim.x;
    int bad = 0;
    const int64_t nvec = vec_ok ? n / W : 0;
    // the loop bound is the same for the 32 lanes of a warp (votes below),
    // and with POOL for the whole block (barriers)
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (POOL ? 0 : warp * 32); i0 < nvec;
         i0 += wstride) {
        const int64_t i = i0 + (POOL ? threadIdx.x : lane);
        const bool have = i < nvec;
        T a[W], b[W], c[W], v[W];
        if (have) {
            to_arr(ld_stream(reinterpret_cast<const VT*>(nx) + i), a);
            to_arr(ld_stream(reinterpret_cast<const VT*>(ny) + i), b);
            to_arr(ld_stream(reinterpret_cast<const VT*>(nz) + i), c);
            to_arr(ld_stream(reinterpret_cast<const VT*>(V0) + i), v);
        }
        // front end (Sec. 2.1) and the closed-form cases
        T red[W][4], scale[W], res[W];
        unsigned need = 0u;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            res[j] = T(0);
            scale[j] = T(0);
            if (!have) continue;
            T n1, n2, n3, L, V;
            bool ok;
            if constexpr (BITS) {
                ok = front_bits(a[j], b[j], c[j], v[j], n1, n2, n3, L, V);
            } else {
                reduce_normal<T, false>(a[j], b[j], c[j], n1, n2, n3);
                L = fabs(a[j]) + fabs(b[j]) + fabs(c[j]);
                ok = (v[j] >= T(0)) && (v[j] <= T(1)) && (L > T(0)) && (L <= T(3));
            }
            if (!ok) {
                bad += 1;
                res[j] = T(NAN);
                continue;
            }
            if constexpr (!BITS) V = reduce_volume<T, false>(v[j]);
            if (SZ) {
                const T il = Fm<T>::rcp_(L);
                n1 *= il;
                n3 *= il;
                n2 = Fm<T>::fdim_(T(1), n1 + n3);
                scale[j] = L;
            } else {
                scale[j] = BITS ? L : T(1);             // with BITS, L/2 is the offset's origin
            }
            red[j][0] = V; red[j][1] = n1; red[j][2] = n2; red[j][3] = n3;
            T d;
            if (S::easy(V, n1, n2, n3, d)) res[j] = d;
            else need |= 1u << j;
        }
        // the heavy part on the packed task list of the warp (of the block)
        unsigned m[W];
        int pre[W + 1];
        pre[0] = 0;
#pragma unroll
        for (int j = 0; j < W; ++j) {
            m[j] = __ballot_sync(0xffffffffu, (need >> j) & 1u);
            pre[j + 1] = pre[j] + __popc(m[j]);
        }
        if constexpr (POOL) {
            T (*flat)[4] = &task[0][0];
            if (lane == 0) wtot[warp] = pre[W];
            __syncthreads();
            int base = 0, total = 0;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const int x = wtot[w];
                base += w < warp ? x : 0;
                total += x;
            }
#pragma unroll
            for (int j = 0; j < W; ++j)
                if ((need >> j) & 1u) {
                    T* q = flat[base + pre[j] + __popc(m[j] & lt)];
                    q[0] = red[j][0]; q[1] = red[j][1]; q[2] = red[j][2]; q[3] = red[j][3];
                }
            __syncthreads();
            for (int t = threadIdx.x; t < total; t += blockDim.x) {
                T* q = flat[t];
                q[0] = S::hard(q[0], q[1], q[2], q[3]);
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < W; ++j)
                if ((need >> j) & 1u) res[j] = flat[base + pre[j] + __popc(m[j] & lt)][0];
            __syncthreads();
        } else {
#pragma unroll
            for (int j = 0; j < W; ++j)
                if ((need >> j) & 1u) {
                    T* q = task[warp][pre[j] + __popc(m[j] & lt)];
                    q[0] = red[j][0]; q[1] = red[j][1]; q[2] = red[j][2]; q[3] = red[j][3];
                }
            __syncwarp();
            for (int t = lane; t < pre[W]; t += 32) {
                T* q = task[warp][t];
                q[0] = S::hard(q[0], q[1], q[2], q[3]);
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < W; ++j)
                if ((need >> j) & 1u) res[j] = task[warp][pre[j] + __popc(m[j] & lt)][0];
            __syncwarp();
        }
        // polish and the symmetry back to d0 (Eqs. 5-8)
        T r[W];
#pragma unroll
        for (int j = 0; j < W; ++j) {
            if (!(scale[j] > T(0))) {
                r[j] = res[j];                       // invalid cell: NaN
                continue;
            }
            T x = res[j];
            if (POLISH) x = polish<T>(x, red[j][0], red[j][1], red[j][2], red[j][3]);
            if constexpr (BITS) {
                // the sign of V0 - 1/2 on the bits (no FP64 subtraction)
                r[j] = sign_of_side(SZ ? scale[j] * (T(0.5) - x) : T(0.5) * scale[j] - x, v[j]);
            } else {
                if (SZ) r[j] = scale[j] * copysign(T(0.5) - x, v[j] - T(0.5));
                else r[j] = copysign(T(0.5) * (red[j][1] + red[j][2] + red[j][3]) - x, v[j] - T(0.5));
            }
        }
        if (have) st_stream(reinterpret_cast<VT*>(d0) + i, from_arr(r));
    }
    for (int64_t i = nvec * W + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += wstride)
        d0[i] = offset_cell<METHOD, T, POLISH, false>(nx[i], ny[i], nz[i], V0[i], bad);
    count_invalid(bad, invalid);
}

// The optimised SZ, Kawano's SZ and the analytic solution in FP32 on paired
// FP32 instructions: each thread takes 4 cells per step as two pairs, so every
// cell sees identical arithmetic wherever it lies.  VEC (every array on a
// 16-byte boundary): consecutive cells through one 16-byte load per array.
// Otherwise (an odd row of a (3, n) tensor, a slice): cells 32 apart, a run of
// 128 cells per warp, four loads per array in flight.  The cells left over (n mod 4, n
// mod 1024) take one lane each, the cell in both lanes of the pair; all unaligned cells
// that way took 88 us for 10 M cells of the analytic solution, 40 us this way (aligned
// arrays: 35; 64 M: 222 and 193, with cells 256 apart 227, whose neighbouring warps
// fetch the sector between their lines twice; 16-byte loads of the enclosing
// vectors, shifted across the lanes: 249).
// With ROUNDTRIP the forward volume of each stored d0 is written to vrt in
// the same pass (plic_offset_roundtrip); COUNT (an invalid-cell counter was
// given) keeps the per-cell count of invalid inputs, which otherwise costs
// instructions for nothing.
// Bound: HBM (20 B per cell, 24 with the round trip).  With the arcsine, the
// sine and a Newton step on Eq. 10 in d these kernels were issue bound (131
// instructions per cell in the round trip); with the depressed cubic
// (p2::centre_distance), 2^26 cells: optimised SZ 265 -> 205 us, analytic
// 320 -> 200 us (0.985 of the copy rate); round trip of 2^28 cells 1240 ->
// 1000 us (0.945).  Residency of these two: five blocks per SM (48 registers)
// without and four (64 registers) with the round trip is the fastest measured
// (205 against 212 us at the compiler's 51 registers, 995 against 1004 us at 56).
constexpr int pair_blocks(int method, bool roundtrip) {
    return method == M_SZ_ORIG ? 0 : roundtrip ? 4 : 5;
}

template <int METHOD, bool POLISH, bool ROUNDTRIP, bool COUNT, bool VEC>
__global__ void __launch_bounds__(256, pair_blocks(METHOD, ROUNDTRIP))
k_plic_offset_pair(const float* __restrict__ nx, const float* __restrict__ ny,
                   const float* __restrict__ nz, const float* __restrict__ V0,
                   float* __restrict__ d0, int64_t n, int /* vec_ok: VEC */,
                   unsigned long long* invalid, float* __restrict__ vrt) {
    int bad[2] = {0, 0}, bad1[2] = {0, 0};           // per lane of the pair; bad1: a cell in both lanes
    float2 w0, w1;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t tail;                                    // the cells from here on go one at a time
    if constexpr (VEC) {
        const int64_t nvec = n / 4;
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += stride) {
            const float4 a = __ldcs(reinterpret_cast<const float4*>(nx) + i);
            const float4 b = __ldcs(reinterpret_cast<const float4*>(ny) + i);
            const float4 c = __ldcs(reinterpret_cast<const float4*>(nz) + i);
            const float4 v = __ldcs(reinterpret_cast<const float4*>(V0) + i);
            const float2 r0 = p2::offset_pair<METHOD, POLISH, ROUNDTRIP, COUNT>(
                make_float2(a.x, a.y), make_float2(b.x, b.y), make_float2(c.x, c.y), make_float2(v.x, v.y),
                bad, &w0);
            const float2 r1 = p2::offset_pair<METHOD, POLISH, ROUNDTRIP, COUNT>(
                make_float2(a.z, a.w), make_float2(b.z, b.w), make_float2(c.z, c.w), make_float2(v.z, v.w),
                bad, &w1);
            __stcs(reinterpret_cast<float4*>(d0) + i, make_float4(r0.x, r0.y, r1.x, r1.y));
            if (ROUNDTRIP) __stcs(reinterpret_cast<float4*>(vrt) + i, make_float4(w0.x, w0.y, w1.x, w1.y));
        }
        tail = nvec * 4;
    } else {
        tail = n & ~(int64_t)1023;
        for (int64_t i0 = (int64_t)blockIdx.x * 1024; i0 < tail; i0 += 4 * stride) {
            const int64_t i = i0 + ((threadIdx.x & ~31u) * 4u + (threadIdx.x & 31u));
            float a[4], b[4], c[4], v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                a[j] = __ldcs(nx + i + 32 * j);
                b[j] = __ldcs(ny + i + 32 * j);
                c[j] = __ldcs(nz + i + 32 * j);
                v[j] = __ldcs(V0 + i + 32 * j);
            }
#pragma unroll
            for (int j = 0; j < 4; j += 2) {
                const float2 r = p2::offset_pair<METHOD, POLISH, ROUNDTRIP, COUNT>(
                    make_float2(a[j], a[j + 1]), make_float2(b[j], b[j + 1]), make_float2(c[j], c[j + 1]),
                    make_float2(v[j], v[j + 1]), bad, &w0);
                __stcs(d0 + i + 32 * j, r.x);
                __stcs(d0 + i + 32 * (j + 1), r.y);
                if (ROUNDTRIP) {
                    __stcs(vrt + i + 32 * j, w0.x);
                    __stcs(vrt + i + 32 * (j + 1), w0.y);
                }
            }
        }
    }
    for (int64_t i = tail + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float2 r = p2::offset_pair<METHOD, POLISH, ROUNDTRIP, COUNT>(
            make_float2(nx[i], nx[i]), make_float2(ny[i], ny[i]), make_float2(nz[i], nz[i]),
            make_float2(V0[i], V0[i]), bad1, &w0);
        d0[i] = r.x;
        if (ROUNDTRIP) vrt[i] = w0.x;
    }
    if (COUNT) count_invalid(bad[0] + bad[1] + bad1[0], invalid);
}

// The optimised SZ and the analytic solution in PLIC_FP64 and
// PLIC_FP64_REFINED: the scheme of plic_fx.cuh, and for the cells that the kernel below
// leaves over the same scheme on the rescaled normal, one thread per cell, or the closed
// forms in FP64 (a call, to keep their registers out of the loop).  2^24 cells: normals of
// unit L1 length 452 us, of length 0.3 630 and 1.2 583 (all or half of the cells outside the
// range; by the closed forms, called as the cells were read, 4880, 4820 and 4190; packed
// closed forms 3165, double-float steps 585).  The rescaled cells packed by case as well
// came to 450, 440 and 510, but the unaligned arrays' loop then to 194 us per 10 M cells of
// unit normals, against 184.
template <int METHOD>
__device__ __noinline__ fx::u64 fx_rest(double nx, double ny, double nz, double V0, int& bad) {
    fx::u64 d0;
    if (fx::offset(fx::bits(nx), fx::bits(ny), fx::bits(nz), fx::bits(V0), d0)) return d0;
    int b = 0;
    d0 = fx::bits(offset_cell<METHOD, double, false, false>(nx, ny, nz, V0, b));
    bad += b;
    return d0;
}

// Both methods and precisions are this kernel.  The cases are packed: FX_CELLS cells
// per block and trip; every thread reads its four cells and settles case (5); the others
// leave their task in shared memory and their place in the
// list of their case, or in list 0 where the scheme does not take them as they are (lanes
// of one list share a counter's increment; the order in a
// list does not matter); the warps take 32 cells of one list at a time, list 0 last;
// every thread stores its own cells.  The arrays are read as integers: of the bits of a double in
// a register the compiler makes |x| an operation on the FP64 pipe (three per cell:
// 396 against 317 us).
// Bound: instruction issue (470 warp instructions per 32 cells, 71 % of the slots; ALU
// pipe 68 % busy) beside the FP64 pipe (7 instructions, 67 %).  2^24 cells: closed forms 3200 us (optimised
// SZ, FP64 pipe 85 % busy) and 4490 us (analytic); this scheme with one thread running
// each of its cells through its case 379 us (every case of the warp in turn, 18.8 lanes
// on) and with the tests in fixed point too; packed 284 us (27 lanes on).  16 M
// cells FP64_REFINED 555 (double-float steps) -> 273 us.  256 threads and 1024 cells per
// block 295 us, 64 and 256 295 us; ten blocks per SM (48 registers) 285, eight 287 us.
// Below 2^15 cells 8.2 us at any shape (closed forms 18-22 us).
constexpr int FX_THREADS = 128, FX_CELLS = 4 * FX_THREADS;

template <int METHOD, bool VEC>
__global__ void __launch_bounds__(FX_THREADS, 10)
k_plic_offset_fx(const double* __restrict__ nx, const double* __restrict__ ny,
                        const double* __restrict__ nz, const double* __restrict__ V0,
                        double* __restrict__ d0, int64_t n, int /* vec_ok: VEC */,
                        unsigned long long* invalid, void* /* round trip: not fused here */) {
    typedef fx::u64 u64;
    typedef fx::i64 i64;
    // a cell's task: b1 (with V0 < 1/2 in its sign), b2 and a, y; its d0 then in hi.y
    __shared__ ulonglong2 lo[FX_CELLS], hi[FX_CELLS];
    __shared__ unsigned short list[5][FX_CELLS];        // the cells of cases (1) to (4); 0: the others
    __shared__ int count[5];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int bad = 0;
    for (int64_t i0 = (int64_t)blockIdx.x * FX_CELLS; i0 < n; i0 += (int64_t)gridDim.x * FX_CELLS) {
        const int cells = (int)(n - i0 < FX_CELLS ? n - i0 : FX_CELLS);
        const bool vec = VEC && cells == FX_CELLS;
        if (threadIdx.x < 5) count[threadIdx.x] = 0;
        __syncthreads();
        auto place = [&](int j) { return vec ? 2 * (FX_THREADS * (j >> 1) + (int)threadIdx.x) + (j & 1)
                                             : FX_THREADS * j + (int)threadIdx.x; };
        auto one = [&](int i, u64 ax, u64 ay, u64 az, u64 v) {
            int code = 5;
            if (i < cells) {
                u64 b1 = ax & fx::ABS, b2 = ay & fx::ABS, b3 = az & fx::ABS;
                const u64 va = v & fx::ABS, sign = va < fx::HALF ? fx::TOP : 0ull;
                fx::sort(b1, b2, b3);
                code = 0;
                if (fx::in_range(b1, b3, v)) {
                    fx::Task t;
                    u64 s;
                    code = fx::classify(b1, b2, b3, va, t, s);
                    if (code != 5) {
                        lo[i] = make_ulonglong2(t.b1 | sign, t.b2);
                        hi[i].x = t.a;
                        s = t.y;
                    } else {
                        s |= sign;
                    }
                    hi[i].y = s;
                }
            }
            const unsigned same = __match_any_sync(0xffffffffu, code);
            const int first = __ffs(same) - 1;
            int at = 0;
            if (lane == first && code != 5) at = atomicAdd(&count[code], __popc(same));
            at = __shfl_sync(0xffffffffu, at, first) + __popc(same & ((1u << lane) - 1u));
            if (code != 5) list[code][at] = (unsigned short)i;
        };
        if (vec) {
#pragma unroll 1
            for (int k = 0; k < 2; ++k) {
                const int64_t q = i0 / 2 + FX_THREADS * k + threadIdx.x;
                const ulonglong2 a = __ldcs(reinterpret_cast<const ulonglong2*>(nx) + q);
                const ulonglong2 b = __ldcs(reinterpret_cast<const ulonglong2*>(ny) + q);
                const ulonglong2 c = __ldcs(reinterpret_cast<const ulonglong2*>(nz) + q);
                const ulonglong2 d = __ldcs(reinterpret_cast<const ulonglong2*>(V0) + q);
                one(place(2 * k), a.x, b.x, c.x, d.x);
                one(place(2 * k + 1), a.y, b.y, c.y, d.y);
            }
        } else {
#pragma unroll 1
            for (int j = 0; j < 4; ++j) {
                const int i = place(j);
                const int64_t q = i0 + (i < cells ? i : 0);
                one(i, __ldcs(reinterpret_cast<const u64*>(nx) + q), __ldcs(reinterpret_cast<const u64*>(ny) + q),
                    __ldcs(reinterpret_cast<const u64*>(nz) + q), __ldcs(reinterpret_cast<const u64*>(V0) + q));
            }
        }
        __syncthreads();
        // 32 cells of a case at a time, the longest roots first
        const int c1 = count[1], c2 = count[2], c3 = count[3], c4 = count[4];
        const int t4 = (c4 + 31) >> 5, t3 = t4 + ((c3 + 31) >> 5), t1 = t3 + ((c1 + 31) >> 5),
                  t2 = t1 + ((c2 + 31) >> 5);
        for (int t = warp; t < t2; t += FX_THREADS / 32) {
            const int code = t < t4 ? 4 : t < t3 ? 3 : t < t1 ? 1 : 2;
            const int k = 32 * (t - (t < t4 ? 0 : t < t3 ? t4 : t < t1 ? t3 : t1)) + lane;
            if (k < (code == 4 ? c4 : code == 3 ? c3 : code == 1 ? c1 : c2)) {
                const int i = list[code][k];
                const ulonglong2 p = lo[i], q = hi[i];
                const fx::Task c = {p.x & fx::ABS, p.y, q.x, q.y};
                u64 s;
                bool ok;
                if (code == 2) ok = fx::root_square(c, s);
                else if (code == 3) ok = fx::root_cubic(c, false, false, s);
                else if (code == 4) ok = fx::root_cubic(c, false, true, s);
                else ok = fx::root_cubic(c, true, false, s);
                hi[i].y = fx::round_s(s, (i64)p.x < 0);
                if (!ok) list[0][atomicAdd(&count[0], 1)] = (unsigned short)i;
            }
        }
        __syncthreads();
        const int rest = count[0];
        if (rest > 0) {
            for (int k = threadIdx.x; k < rest; k += FX_THREADS) {
                const int i = list[0][k];
                const int64_t q = i0 + i;
                hi[i].y = fx_rest<METHOD>(nx[q], ny[q], nz[q], V0[q], bad);
            }
            __syncthreads();
        }
        if (vec) {
#pragma unroll
            for (int k = 0; k < 2; ++k)
                __stcs(reinterpret_cast<double2*>(d0) + i0 / 2 + FX_THREADS * k + threadIdx.x,
                       make_double2(fx::asd(hi[place(2 * k)].y), fx::asd(hi[place(2 * k + 1)].y)));
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (place(j) < cells) __stcs(d0 + i0 + place(j), fx::asd(hi[place(j)].y));
        }
        // (the next trip writes the tasks behind its first barrier)
    }
    count_invalid(bad, invalid);
}

// PLIC_FP64_REFINED: double in/out, FP32 solve + two FP64 Newton steps.
template <int METHOD>
__global__ void __launch_bounds__(256)
k_plic_offset_refined(const double* __restrict__ nx, const double* __restrict__ ny,
                      const double* __restrict__ nz, const double* __restrict__ V0,
                      double* __restrict__ d0, int64_t n, int vec_ok,
                      unsigned long long* invalid, void* /* round trip: not fused here */) {
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int bad = 0;
    const int64_t nvec = vec_ok ? n / 2 : 0;
    for (int64_t i = tid; i < nvec; i += stride) {
        const double2 a = __ldcs(reinterpret_cast<const double2*>(nx) + i);
        const double2 b = __ldcs(reinterpret_cast<const double2*>(ny) + i);
        const double2 c = __ldcs(reinterpret_cast<const double2*>(nz) + i);
        const double2 v = __ldcs(reinterpret_cast<const double2*>(V0) + i);
        const double r0 = offset_cell_refined<METHOD>(a.x, b.x, c.x, v.x, bad);
        const double r1 = offset_cell_refined<METHOD>(a.y, b.y, c.y, v.y, bad);
        __stcs(reinterpret_cast<double2*>(d0) + i, make_double2(r0, r1));
    }
    for (int64_t i = nvec * 2 + tid; i < n; i += stride)
        d0[i] = offset_cell_refined<METHOD>(nx[i], ny[i], nz[i], V0[i], bad);
    count_invalid(bad, invalid);
}

template <int METHOD, typename T, bool POLISH, bool FAITHFUL>
static const void* kptr() {
    return reinterpret_cast<const void*>(&k_plic_offset<METHOD, T, POLISH, FAITHFUL>);
}

template <int METHOD, typename T, bool POLISH>
static const void* cptr() {
    return reinterpret_cast<const void*>(&k_plic_offset_compact<METHOD, T, POLISH>);
}

// The default solvers run work-compacted (k_plic_offset_compact); the
// paper-literal ones keep one cell after the other per lane.
// In FP32 the optimised SZ, Kawano's SZ and the analytic solution take the
// paired kernel (k_plic_offset_pair, chosen in offset_entry); Kawano's SZ in
// FP32 is packed in no form here: its heavy part (one arccosine and one
// cosine on the FP32 pipes) is too short to repay the packing (measured 102
// against 130 G solves/s one cell after the other, on 2^26 cells), and only
// its faithful form reaches this function in FP32.  In FP64, and for the
// iterative solvers, packing wins (e.g. nested intervals FP32 27 -> 40 G solves/s).
template <int METHOD>
static const void* pick(plic_precision p, bool faithful, bool vec) {
    if constexpr (METHOD == M_SZ_OPT || METHOD == M_ANALYTIC) {
        if (!faithful && (p == PLIC_FP64 || p == PLIC_FP64_REFINED))
            return vec ? reinterpret_cast<const void*>(&k_plic_offset_fx<METHOD, true>)
                       : reinterpret_cast<const void*>(&k_plic_offset_fx<METHOD, false>);
        // in FP32 these two come here in their faithful forms only (pick_pair)
        return p == PLIC_FP64 ? kptr<METHOD, double, false, true>()
             : p == PLIC_FP32_POLISHED ? kptr<METHOD, float, true, true>() : kptr<METHOD, float, false, true>();
    } else {
        if (p == PLIC_FP64_REFINED) return reinterpret_cast<const void*>(&k_plic_offset_refined<METHOD>);
        if (p == PLIC_FP64)
            return faithful ? kptr<METHOD, double, false, true>() : cptr<METHOD, double, false>();
        if constexpr (METHOD == M_SZ_ORIG)           // its default form is paired (pick_pair)
            return p == PLIC_FP32_POLISHED ? kptr<METHOD, float, true, true>() : kptr<METHOD, float, false, true>();
        else if (p == PLIC_FP32_POLISHED)
            return faithful ? kptr<METHOD, float, true, true>() : cptr<METHOD, float, true>();
        else
            return faithful ? kptr<METHOD, float, false, true>() : cptr<METHOD, float, false>();
    }
}

// The paired FP32 kernels (optimised SZ, Kawano's SZ, analytic); *fused is set
// when the round-trip volume comes out of the same kernel.  The optimised SZ
// and the analytic root end with their Newton step in either precision, so
// FP32 and FP32_POLISHED are one kernel there.
template <int METHOD, bool POLISH, bool VEC>
static const void* pick_pair_k(bool roundtrip, bool count) {
    if (roundtrip)
        return count ? reinterpret_cast<const void*>(&k_plic_offset_pair<METHOD, POLISH, true, true, VEC>)
                     : reinterpret_cast<const void*>(&k_plic_offset_pair<METHOD, POLISH, true, false, VEC>);
    return count ? reinterpret_cast<const void*>(&k_plic_offset_pair<METHOD, POLISH, false, true, VEC>)
                 : reinterpret_cast<const void*>(&k_plic_offset_pair<METHOD, POLISH, false, false, VEC>);
}

template <int METHOD>
static const void* pick_pair(bool polish, bool roundtrip, bool count, bool vec, bool* fused) {
    *fused = roundtrip;
    constexpr bool ONE = METHOD != M_SZ_ORIG;
    if (polish || ONE)
        return vec ? pick_pair_k<METHOD, true, true>(roundtrip, count)
                   : pick_pair_k<METHOD, true, false>(roundtrip, count);
    return vec ? pick_pair_k<METHOD, ONE, true>(roundtrip, count)
               : pick_pair_k<METHOD, ONE, false>(roundtrip, count);
}

static plic_status offset_entry(const void* nx, const void* ny, const void* nz, const void* V0,
                                void* d0, void* vrt, int64_t n, plic_method m, plic_precision p,
                                uint32_t flags, int64_t* d_invalid_count, void* stream,
                                bool* fused, const char* who) {
    *fused = false;
    if (n < 0) return PLIC_ERR_ARG;
    if ((int)m < 0 || (int)m > 4 || (int)p < 0 || (int)p > 3) return PLIC_ERR_ARG;
    if (flags & ~(uint32_t)PLIC_FLAG_FAITHFUL) return PLIC_ERR_ARG;
    if (p == PLIC_FP64_REFINED && (flags & PLIC_FLAG_FAITHFUL)) return PLIC_ERR_UNSUPPORTED;
    if (n == 0) return PLIC_OK;
    if (!nx || !ny || !nz || !V0 || !d0) return PLIC_ERR_ARG;
    const bool dbl = p == PLIC_FP64 || p == PLIC_FP64_REFINED;
    const size_t es = dbl ? 8 : 4;
    if (!aligned(nx, es) || !aligned(ny, es) || !aligned(nz, es) || !aligned(V0, es) ||
        !aligned(d0, es) || (vrt && !aligned(vrt, es)) ||
        (d_invalid_count && !aligned(d_invalid_count, 8)))
        return PLIC_ERR_ALIGN;
    const int vec_ok = aligned(nx, 16) && aligned(ny, 16) && aligned(nz, 16) && aligned(V0, 16) &&
                       aligned(d0, 16) && (!vrt || aligned(vrt, 16));
    const bool faithful = (flags & PLIC_FLAG_FAITHFUL) != 0;
    const bool pair = !dbl && !faithful && (m == PLIC_ANALYTIC || m == PLIC_SZ_ORIG || m == PLIC_SZ_OPT);
    const bool fx = dbl && !faithful && (m == PLIC_ANALYTIC || m == PLIC_SZ_OPT);
    const void* k = nullptr;
    switch (m) {
        case PLIC_ANALYTIC:
            k = pair ? pick_pair<M_ANALYTIC>(p == PLIC_FP32_POLISHED, vrt != nullptr,
                                                            d_invalid_count != nullptr, vec_ok != 0, fused)
                                    : pick<M_ANALYTIC>(p, faithful, vec_ok != 0);
            break;
        case PLIC_SZ_ORIG:
            k = pair ? pick_pair<M_SZ_ORIG>(p == PLIC_FP32_POLISHED, vrt != nullptr,
                                                           d_invalid_count != nullptr, vec_ok != 0, fused)
                                    : pick<M_SZ_ORIG>(p, faithful, vec_ok != 0);
            break;
        case PLIC_SZ_OPT:
            k = pair ? pick_pair<M_SZ_OPT>(p == PLIC_FP32_POLISHED, vrt != nullptr,
                                                          d_invalid_count != nullptr, vec_ok != 0, fused)
                                    : pick<M_SZ_OPT>(p, faithful, vec_ok != 0);
            break;
        case PLIC_NEWTON: k = pick<M_NEWTON>(p, faithful, vec_ok != 0); break;
        case PLIC_NESTED: k = pick<M_NESTED>(p, faithful, vec_ok != 0); break;
    }
    const int threads = fx ? FX_THREADS : 256;
    const int W = dbl && !fx ? 2 : 4;
    // 4 cells per thread also where the paired and the packed FP64 kernels read
    // unaligned arrays
    const int64_t work = vec_ok || pair || fx ? (n + W - 1) / W : n;
    const int grid = stream_grid(k, threads, work);
    unsigned long long* inv = reinterpret_cast<unsigned long long*>(d_invalid_count);
    void* args[] = {(void*)&nx, (void*)&ny, (void*)&nz, (void*)&V0, (void*)&d0,
                    (void*)&n, (void*)&vec_ok, (void*)&inv, (void*)&vrt};
    cudaError_t e = cudaLaunchKernel(k, dim3(grid), dim3(threads), args, 0, as_stream(stream));
    if (e != cudaSuccess) {
        set_last_error(who, e);
        return PLIC_ERR_CUDA;
    }
    return PLIC_OK;
}

}  // namespace plic

extern "C" plic_status plic_offset(const void* nx, const void* ny, const void* nz,
                                   const void* V0, void* d0, int64_t n, plic_method m,
                                   plic_precision p, uint32_t flags, int64_t* d_invalid_count,
                                   void* stream) {
    bool fused;
    return plic::offset_entry(nx, ny, nz, V0, d0, nullptr, n, m, p, flags, d_invalid_count, stream,
                              &fused, "plic_offset");
}

extern "C" plic_status plic_offset_roundtrip(const void* nx, const void* ny, const void* nz,
                                             const void* V0, void* d0, void* V0_rt, int64_t n,
                                             plic_method m, plic_precision p, uint32_t flags,
                                             int64_t* d_invalid_count, void* stream) {
    if (n > 0 && !V0_rt) return PLIC_ERR_ARG;
    bool fused;
    plic_status s = plic::offset_entry(nx, ny, nz, V0, d0, V0_rt, n, m, p, flags, d_invalid_count,
                                       stream, &fused, "plic_offset_roundtrip");
    if (s != PLIC_OK || fused || n == 0) return s;
    const plic_precision vp = (p == PLIC_FP64 || p == PLIC_FP64_REFINED) ? PLIC_FP64 : PLIC_FP32;
    return plic_volume(nx, ny, nz, d0, V0_rt, n, vp, stream);
}
