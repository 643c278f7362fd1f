// vof_compact.cu -- interface-cell compaction (Sec. 4.1, Eq. 33): the ordered
// list of interior cells with 0 < phi < 1, and plic_workspace_bytes().
//
// Two launches, no atomics on global memory and no inter-block waiting, so the
// list is in ascending cell order and identical run to run.  The field is
// taken as one flat run of cells (the planes z = 0 and z = nz - 1 left out),
// whatever its rows: a chunk is 32 lanes x 4 U cells, a tile CT_WARPS x K chunks.
//   1. k_compact_count : reads the field once.  A warp first asks whether its
//                        chunk holds any value in (0, 1) at all -- one fused
//                        multiply-add v - v^2 and half a three-way maximum
//                        per cell, one vote per chunk -- and goes on only
//                        where it does (a quarter of the chunks of a field of
//                        droplets): there it tests the cells exactly, drops
//                        those on the field's boundary (the only place where
//                        x, y and z are needed) and stores the chunk's bits, one
//                        word per 32 cells.  Per tile it writes the count and a
//                        mask of the chunks that hold cells, and per block of
//                        S tiles the sum of their counts.
//   2. k_compact_emit  : one warp per tile sums the counts before it and writes
//                        the indices from the stored bits of the marked
//                        chunks, or (no bits: the allocation-free entry) from
//                        the field again, marked chunks only.
// Bound: HBM, 4 B per field cell read once (+ 1/8 B of bits for marked chunks,
// + 4 B per interface cell).  Times of the two passes (fields read from HBM),
// against a row-wise pass that packed every cell's test into bits: 64^3 14.2 +
// 5.6 -> 5.9 + 5.3 us; 301 x 203 x 257 (rows that are not whole 16-byte
// vectors, read cell by cell before) 42.9 + 10.0 -> 13.7 + 6.7 us; 256^3 15.1 +
// 6.2 -> 15.0 + 6.8 us (in L2, with the curvature after it: 29.0 -> 24.1 us);
// 1 GiB 170.7 + 24.8 (with a scan launch between) -> 153.4 + 18.7 us, the
// plain read being 149.
#include <mutex>
#include <stdio.h>

#include "host_common.h"
#include "workspace.h"

namespace plic {

constexpr int CT_THREADS = 256;
constexpr int CT_WARPS = CT_THREADS / 32;
// The interface test 0 < phi < 1 on the float's bits: the positive floats
// below 1.0f are exactly the bit patterns 1 .. 0x3F7FFFFF (zero, negative
// values, 1.0f and above, infinities and NaNs all fall outside).
__device__ __forceinline__ bool iface_bits(float v) { return __float_as_uint(v) - 1u < 0x3F7FFFFFu; }

// Positive exactly for 0 < v < 1 (v - v^2 rounded once: its sign is that of
// v (1 - v), and it does not underflow to 0, since v - v^2 >= 2^-149 there);
// NaN for a NaN and for +inf - inf, which the maxima below skip.
__device__ __forceinline__ float inside(float v) { return fmaf(-v, v, v); }
__device__ __forceinline__ float max3(float a, float b, float c) { return fmaxf(fmaxf(a, b), c); }

// Division of 0 <= n < 2^31 by a divisor fixed per launch: with l =
// ceil(log2 d) and m = floor(2^(31 + l) / d) + 1 (m < 2^32), floor(n m / 2^(31 + l))
// is the quotient (Granlund and Montgomery 1994: m d - 2^(31 + l) <= d <= 2^l).
struct Divider {
    unsigned d, m, s;
    explicit Divider(unsigned divisor) : d(divisor) {
        int l = 0;
        while ((1ull << l) < divisor) ++l;
        m = (unsigned)((1ull << (31 + l)) / divisor + 1ull);
        s = (unsigned)(l > 0 ? l - 1 : 0);
        if (l == 0) m = 0u;                          // d = 1: n itself (div() below)
    }
    __device__ __forceinline__ unsigned div(unsigned n) const { return m ? __umulhi(n, m) >> s : n; }
};

// Field geometry for the boundary test of single cells.
struct Geometry {
    Divider nx, ny;
    unsigned nz;
    // Of the cells c + step j whose bit j is set in m (j < 4), those interior.
    template <int STEP>
    __device__ __forceinline__ unsigned interior(unsigned c, unsigned m) const {
        unsigned row = nx.div(c), x = c - row * nx.d, z = ny.div(row), y = row - z * ny.d;
        if (STEP == 1 && x + 3u < nx.d) {            // four cells of one row
            const bool in = y - 1u < ny.d - 2u && z - 1u < nz - 2u;
            if (x == 0u) m &= ~1u;
            if (x + 4u == nx.d) m &= ~8u;
            return in ? m : 0u;
        }
        unsigned k = 0u;
        for (int j = 0; j < 4; ++j) {
            const unsigned cj = c + (unsigned)(STEP * j);
            row = nx.div(cj); x = cj - row * nx.d; z = ny.div(row); y = row - z * ny.d;
            if (x - 1u < nx.d - 2u && y - 1u < ny.d - 2u && z - 1u < nz - 2u) k |= 1u << j;
        }
        return m & k;
    }
};

// The values of a chunk: ALIGNED (16-byte aligned field): component k of v[u]
// is cell c0 + 128 u + 4 lane + k; otherwise v[u] holds cells c0 + 128 u + 32 k
// + lane.  Cells from `end` on read as 0.
template <int U, bool ALIGNED>
__device__ __forceinline__ void load_chunk(const float* __restrict__ phi, int64_t c0, int64_t end,
                                           float4 (&v)[U]) {
    const int lane = threadIdx.x & 31;
    if (c0 + 128 * U <= end) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (ALIGNED) {
                v[u] = __ldg(reinterpret_cast<const float4*>(phi + c0) + 32 * u + lane);
            } else {
                const float* p = phi + c0 + 128 * u + lane;
                v[u] = make_float4(__ldg(p), __ldg(p + 32), __ldg(p + 64), __ldg(p + 96));
            }
        }
    } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t c = c0 + 128 * u + (ALIGNED ? 4 * lane : lane);
            constexpr int step = ALIGNED ? 1 : 32;
            v[u].x = c < end ? __ldg(phi + c) : 0.0f;
            v[u].y = c + step < end ? __ldg(phi + c + step) : 0.0f;
            v[u].z = c + 2 * step < end ? __ldg(phi + c + 2 * step) : 0.0f;
            v[u].w = c + 3 * step < end ? __ldg(phi + c + 3 * step) : 0.0f;
        }
    }
}

// The four-bit interface mask of a lane's component of a chunk, boundary
// cells dropped: bit k for component k of v (see load_chunk), c its first cell.
template <bool ALIGNED>
__device__ __forceinline__ unsigned mask4(float4 v, unsigned c, const Geometry& g) {
    unsigned m = (unsigned)iface_bits(v.x) | ((unsigned)iface_bits(v.y) << 1) |
                 ((unsigned)iface_bits(v.z) << 2) | ((unsigned)iface_bits(v.w) << 3);
    return m ? g.interior<ALIGNED ? 1 : 32>(c, m) : 0u;
}

// Pass 1 (see the head of this file).  info[t]: the tile's count and, from bit
// 16, its chunk mask (K * CT_WARPS bits; a count is at most 8192); super[b]:
// the block's count (not written for S = 1).  Every chunk of a tile is loaded
// before any is used (K U 16-byte loads per lane in flight).
template <int U, int K, bool ALIGNED>
__global__ void __launch_bounds__(CT_THREADS)
k_compact_count(const float* __restrict__ phi, Geometry geo, int64_t base, int64_t cells, int64_t ntiles,
                int S, int* __restrict__ info, int* __restrict__ super, unsigned* __restrict__ bits) {
    constexpr int CHUNK = 128 * U, TILE = CT_WARPS * K * CHUNK;
    __shared__ unsigned s_info[64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 64) s_info[threadIdx.x] = 0u;
    __syncthreads();
    pdl_wait();                                     // the kernel that wrote the field complete
    const int64_t t0 = (int64_t)blockIdx.x * S, end = base + cells;
    const int nt = (int)(t0 + S < ntiles ? S : ntiles - t0);
    for (int i = 0; i < nt; ++i) {
        const int64_t first = base + (t0 + i) * TILE;
        float4 v[K][U];
#pragma unroll
        for (int q = 0; q < K; ++q) load_chunk<U, ALIGNED>(phi, first + (q * CT_WARPS + warp) * CHUNK, end, v[q]);
#pragma unroll
        for (int q = 0; q < K; ++q) {
            float in[U], any = 0.0f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                in[u] = max3(inside(v[q][u].x), inside(v[q][u].y), inside(v[q][u].z));
                in[u] = fmaxf(in[u], inside(v[q][u].w));
                any = fmaxf(any, in[u]);
            }
            if (!__any_sync(0xffffffffu, any > 0.0f)) continue;
            const int64_t c0 = first + (q * CT_WARPS + warp) * CHUNK;
            unsigned* wp = bits ? bits + ((c0 - base) >> 5) : nullptr;
            int cnt = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                unsigned m = 0u, w = 0u;
                const bool some = __any_sync(0xffffffffu, in[u] > 0.0f);
                if (some) m = mask4<ALIGNED>(v[q][u], (unsigned)(c0 + 128 * u + (ALIGNED ? 4 * lane : lane)), geo);
                cnt += __popc(m);
                if (!wp) continue;
                if (ALIGNED) {
                    if (some) {
                        // the nibbles of 8 lanes make one word
                        w = m << (4 * (lane & 7));
                        w |= __shfl_xor_sync(0xffffffffu, w, 1);
                        w |= __shfl_xor_sync(0xffffffffu, w, 2);
                        w |= __shfl_xor_sync(0xffffffffu, w, 4);
                    }
                    if ((lane & 7) == 0) wp[4 * u + (lane >> 3)] = w;
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        w = __ballot_sync(0xffffffffu, (m >> k) & 1u);
                        if (lane == 0) wp[4 * u + k] = w;
                    }
                }
            }
            cnt = __reduce_add_sync(0xffffffffu, cnt);
            if (lane == 0 && cnt)
                atomicAdd(&s_info[i], (unsigned)cnt | (0x10000u << (q * CT_WARPS + warp)));
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int sum = 0;
        for (int i = threadIdx.x; i < nt; i += 32) {
            info[t0 + i] = (int)s_info[i];
            sum += (int)(s_info[i] & 0xffffu);
        }
        if (S > 1) {
            sum = __reduce_add_sync(0xffffffffu, sum);
            if (threadIdx.x == 0) super[blockIdx.x] = sum;
        }
    }
    pdl_trigger();                                  // the next pass may be scheduled
}

// Pass 2: one warp per tile and trip, CT_WARPS * TPW consecutive tiles per
// block (`tpw` trips; a block without cells returns at once).  The tile's first
// slot is the sum of the counts before it: the block sums those of the blocks of
// pass 1 before its first tile's (at most CT_MAX_SUPERS, eight 16-byte loads per
// thread issued together), each warp adds those of the tiles from there to
// its own.  With bits, the block lists the non-zero words of its eight tiles in
// shared memory with their first slots (lane l of a tile's warp takes the words
// W l .., W = TILE / 1024; words of unmarked chunks, never written, count as
// 0; one warp scan), and then all its warps go through the list, lane q writing
// bit q's cell: a short coalesced store per word, in parallel however the
// cells crowd in one tile (a lane looping over the bits of its own words:
// 836 k warp instructions on the 256^3 field; a warp going through its own
// tile's words one after the other: 14 us).  Without bits the marked chunks are
// read from the field again.  The warp of the last tile writes the total.
template <int U, int K, bool ALIGNED, bool BITS>
__global__ void __launch_bounds__(CT_THREADS)
k_compact_emit(const float* __restrict__ phi, Geometry geo, int64_t base, int64_t cells, int64_t ntiles,
               int S, int tpw, const int* __restrict__ info, const int* __restrict__ super,
               const unsigned* __restrict__ bits, int32_t* __restrict__ idx, int64_t cap,
               int64_t* __restrict__ d_count) {
    constexpr int CHUNK = 128 * U, TILE = CT_WARPS * K * CHUNK, W = TILE / 1024;
    __shared__ int s_part[CT_WARPS], s_words[CT_WARPS];
    __shared__ uint2 s_list[BITS ? CT_WARPS * 32 * W : 1];
    __shared__ unsigned short s_word[BITS ? CT_WARPS * 32 * W : 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nblk = CT_WARPS * tpw;                 // tiles of a block, at most 32
    const int64_t t0 = (int64_t)blockIdx.x * nblk;
    pdl_wait();                                     // pass 1 complete
    // every warp holds the infos of the block's tiles, lane l tile t0 + l
    const unsigned mine = (lane < nblk && t0 + lane < ntiles) ? (unsigned)__ldg(info + t0 + lane) : 0u;
    const bool last = t0 + nblk >= ntiles;
    if (!last && __all_sync(0xffffffffu, (mine & 0xffffu) == 0u)) return;
    // the words of tile t0 + i of this warp (those of its marked chunks): lane l
    // takes W of them, which lie in one chunk
    static_assert((4 * U) % W == 0, "words and chunks nest");
    unsigned b[W];
    auto words = [&](int i) {
        const unsigned marked = i < nblk ? __shfl_sync(0xffffffffu, mine, i) >> 16 : 0u;
        const unsigned* tb = bits + (t0 + i) * (TILE / 32) + W * lane;
        const bool on = (marked >> (W * lane / (4 * U))) & 1u;
#pragma unroll
        for (int k = 0; k < W; ++k) b[k] = on ? __ldg(tb + k) : 0u;
    };
    if constexpr (BITS) words(warp);                // one round trip with the sums below
    // the block's first tile lies in pass-1 block b0 = t0 / S; the tiles from
    // there to t0 are summed one by one (S and nblk are powers of two)
    const int64_t b0 = t0 / S, r0 = b0 * S;
    const int* head = S > 1 ? super : info;
    const unsigned keep = S > 1 ? 0xffffffffu : 0xffffu;
    unsigned part = 0u;                              // counts of fewer than 2^31 cells
    {
        const int n4 = (int)(b0 >> 2);
        int4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int q = threadIdx.x + u * CT_THREADS;
            v[u] = q < n4 ? __ldg(reinterpret_cast<const int4*>(head) + q) : make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            part += (v[u].x & keep) + (v[u].y & keep) + (v[u].z & keep) + (v[u].w & keep);
        if (threadIdx.x < (int)(b0 & 3)) part += __ldg(head + 4 * n4 + threadIdx.x) & keep;
        if (threadIdx.x < (int)(t0 - r0)) part += __ldg(info + r0 + threadIdx.x) & 0xffff;
    }
    part = __reduce_add_sync(0xffffffffu, part);
    if (lane == 0) s_part[warp] = (int)part;
    __syncthreads();
    unsigned before = 0u;
#pragma unroll
    for (int w = 0; w < CT_WARPS; ++w) before += (unsigned)s_part[w];
    if (last && warp == 0) {
        const unsigned total = before + __reduce_add_sync(0xffffffffu, mine & 0xffffu);
        if (lane == 0) *d_count = (int64_t)total;
    }
    for (int i = warp; i < nblk; i += CT_WARPS) {
        const unsigned own = __shfl_sync(0xffffffffu, mine, i);
        int64_t pos = before + __reduce_add_sync(0xffffffffu, lane < i ? mine & 0xffffu : 0u);
        const int64_t first = base + (t0 + i) * TILE;
        if constexpr (BITS) {
            // nothing in the eight tiles of this trip (the same for every warp)
            if (!__any_sync(0xffffffffu, (lane & ~(CT_WARPS - 1)) == i - warp && mine != 0u)) {
                words(i + CT_WARPS);
                continue;
            }
            int c = 0;                               // cells, and non-zero words from bit 16
#pragma unroll
            for (int k = 0; k < W; ++k) c += __popc(b[k]) + (b[k] ? 0x10000 : 0);
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += u;
            }
            if (lane == 31) s_words[warp] = incl >> 16;
            __syncthreads();
            int at = (incl - c) >> 16, total = 0;
#pragma unroll
            for (int w = 0; w < CT_WARPS; ++w) {
                at += w < warp ? s_words[w] : 0;
                total += s_words[w];
            }
            unsigned p = (unsigned)pos + (unsigned)((incl - c) & 0xffff);
#pragma unroll
            for (int k = 0; k < W; ++k)
                if (b[k]) {
                    s_list[at] = make_uint2(b[k], p);
                    s_word[at] = (unsigned short)(32 * W * warp + W * lane + k);
                    p += __popc(b[k]);
                    ++at;
                }
            __syncthreads();
            if (i + CT_WARPS < nblk) words(i + CT_WARPS);     // of the next trip
            const unsigned cell0 = (unsigned)(base + (t0 + (i - warp)) * TILE) + lane;
            const unsigned lt = (1u << lane) - 1u;
#pragma unroll 4
            for (int e = warp; e < total; e += CT_WARPS) {
                const uint2 x = s_list[e];
                const unsigned slot = x.y + __popc(x.x & lt);
                if (((x.x >> lane) & 1u) && slot < cap) idx[slot] = (int32_t)(cell0 + 32u * s_word[e]);
            }
            __syncthreads();                         // the list is used again
        } else {
            if ((own & 0xffffu) == 0u) continue;
            for (unsigned todo = own >> 16; todo; todo &= todo - 1u) {
                const int64_t c0 = first + (__ffs(todo) - 1) * CHUNK;
                float4 v[U];
                load_chunk<U, ALIGNED>(phi, c0, base + cells, v);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t c = c0 + 128 * u + (ALIGNED ? 4 * lane : lane);
                    unsigned m = mask4<ALIGNED>(v[u], (unsigned)c, geo);
                    if (ALIGNED) {
                        int incl = __popc(m);
                        const int n = incl;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const int x = __shfl_up_sync(0xffffffffu, incl, o);
                            if (lane >= o) incl += x;
                        }
                        int64_t p = pos + incl - n;
                        for (; m; m &= m - 1u, ++p)
                            if (p < cap) idx[p] = (int32_t)(c + __ffs(m) - 1);
                        pos += __shfl_sync(0xffffffffu, incl, 31);
                    } else {
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const unsigned w = __ballot_sync(0xffffffffu, (m >> k) & 1u);
                            const int64_t p = pos + __popc(w & ((1u << lane) - 1u));
                            if (((m >> k) & 1u) && p < cap) idx[p] = (int32_t)(c + 32 * k);
                            pos += __popc(w);
                        }
                    }
                }
            }
        }
    }
    pdl_trigger();                                  // (sooner: 1-4 us slower in all)
}

// Both passes as programmatic dependent launches (launch_after): each waits
// for the kernel before it on the stream, the first for the one that wrote
// the field.  info: p.tiles ints, then (S > 1) p.supers ints from the next 16-byte
// boundary; bits: one word per 32 of p.cells, whole tiles, or null.
template <int U, int K, bool ALIGNED>
static cudaError_t launch_compact(const float* phi, const Geometry& g, const CompactPlan& p, int* info,
                                  unsigned* bits, int32_t* idx, int64_t cap, int64_t* d_count,
                                  cudaStream_t s) {
    Geometry geo = g;
    int64_t base = p.base, cells = p.cells, tiles = p.tiles;
    // two trips per block once the prefix is long (1 GiB: 224 us with the curvature
    // after it, 226.5 with one trip, 225.4 with four)
    int S = p.S, tpw = p.S > 1 ? 2 : 1;
    int* super = info + (p.tiles + 3) / 4 * 4;
    void* a1[] = {(void*)&phi, (void*)&geo, (void*)&base, (void*)&cells, (void*)&tiles,
                  (void*)&S, (void*)&info, (void*)&super, (void*)&bits};
    cudaError_t e = launch_after(reinterpret_cast<const void*>(&k_compact_count<U, K, ALIGNED>),
                                 dim3((unsigned)p.supers), dim3(CT_THREADS), a1, s);
    if (e != cudaSuccess) return e;
    void* a2[] = {(void*)&phi, (void*)&geo, (void*)&base, (void*)&cells, (void*)&tiles, (void*)&S, (void*)&tpw,
                  (void*)&info, (void*)&super, (void*)&bits, (void*)&idx, (void*)&cap, (void*)&d_count};
    const void* k = bits ? reinterpret_cast<const void*>(&k_compact_emit<U, K, ALIGNED, true>)
                         : reinterpret_cast<const void*>(&k_compact_emit<U, K, ALIGNED, false>);
    return launch_after(k, dim3((unsigned)((p.tiles + CT_WARPS * tpw - 1) / (CT_WARPS * tpw))), dim3(CT_THREADS), a2, s);
}

template <bool ALIGNED>
static cudaError_t launch_compact(const float* phi, const Geometry& g, const CompactPlan& p, int* info,
                                  unsigned* bits, int32_t* idx, int64_t cap, int64_t* d_count,
                                  cudaStream_t s) {
    if (p.tile == 8192) return launch_compact<4, 2, ALIGNED>(phi, g, p, info, bits, idx, cap, d_count, s);
    if (p.tile == 4096) return launch_compact<4, 1, ALIGNED>(phi, g, p, info, bits, idx, cap, d_count, s);
    return launch_compact<1, 1, ALIGNED>(phi, g, p, info, bits, idx, cap, d_count, s);
}

static cudaError_t compact_passes(const float* phi, int nx, int ny, int nz, const CompactPlan& p, int* info,
                                  unsigned* bits, int32_t* idx, int64_t cap, int64_t* d_count,
                                  cudaStream_t s) {
    const Geometry g = {Divider((unsigned)nx), Divider((unsigned)ny), (unsigned)nz};
    return aligned(phi, 16) ? launch_compact<true>(phi, g, p, info, bits, idx, cap, d_count, s)
                            : launch_compact<false>(phi, g, p, info, bits, idx, cap, d_count, s);
}

}  // namespace plic

extern "C" size_t plic_workspace_bytes(int op, int64_t arg) {
    if (arg < 0) return 0;
    switch (op) {
        case PLIC_WS_COMPACT: return plic::compact_workspace(arg);
        case PLIC_WS_BATCHED: return plic::batch_workspace((size_t)arg);
        default: return 0;
    }
}

extern "C" plic_status vof_interface_compact(const float* phi, int nx, int ny, int nz,
                                             int32_t* idx, int64_t idx_capacity, int64_t* d_count,
                                             void* workspace, size_t ws_bytes, void* stream) {
    using namespace plic;
    if (nx < 0 || ny < 0 || nz < 0 || idx_capacity < 0) return PLIC_ERR_ARG;
    const int64_t ncell = (int64_t)nx * ny * nz;
    if (ncell > 2147483647LL) return PLIC_ERR_ARG;
    if (!d_count) return PLIC_ERR_ARG;
    if (!aligned(d_count, 8)) return PLIC_ERR_ALIGN;
    cudaStream_t s = as_stream(stream);
    if (nx < 3 || ny < 3 || nz < 3) {        // no cell has all 26 neighbours inside
        cudaError_t e = cudaMemsetAsync(d_count, 0, sizeof(int64_t), s);
        if (e != cudaSuccess) { set_last_error("vof_interface_compact", e); return PLIC_ERR_CUDA; }
        return PLIC_OK;
    }
    if (!phi || (!idx && idx_capacity > 0) || !workspace) return PLIC_ERR_ARG;
    if (ws_bytes < plic_workspace_bytes(PLIC_WS_COMPACT, ncell)) return PLIC_ERR_ARG;
    if (!aligned(phi, 4) || (idx && !aligned(idx, 4)) || !aligned(workspace, 256)) return PLIC_ERR_ALIGN;
    const CompactPlan p = compact_plan(nx, ny, nz);
    int* info = reinterpret_cast<int*>(workspace);
    if (compact_bytes(p) > ws_bytes) return PLIC_ERR_ARG;
    unsigned* bits = reinterpret_cast<unsigned*>(reinterpret_cast<char*>(workspace) + compact_bits(p));
    const cudaError_t e = compact_passes(phi, nx, ny, nz, p, info, bits, idx, idx_capacity, d_count, s);
    if (e != cudaSuccess) { set_last_error("vof_interface_compact", e); return PLIC_ERR_CUDA; }
    return check_launch("vof_interface_compact");
}

// ---------------------------------------------------------------------------
// Allocation-free variant.  The scratch of the two passes (tile infos and block
// sums, no bits) lives in a file-scope device array instead of a caller-provided
// workspace.  Every GPU that loads the library holds these 256 KiB until the
// process exits.
// ---------------------------------------------------------------------------
namespace plic {

// a field of at most PLIC_NOALLOC_MAX_CELLS cells has at most that many / 8192
// tiles and CT_MAX_SUPERS block sums
constexpr int64_t kNoAllocInts = 2 * (PLIC_NOALLOC_MAX_CELLS / 8192) + 1;

static __device__ __align__(256) int g_noalloc_tiles[kNoAllocInts];

// Device address of g_noalloc_tiles, looked up once per device (with that
// device current) and cached; host code must not pass the symbol itself.
static int* noalloc_scratch(plic_status* st) {
    static std::mutex mu;
    static int* addr[256] = {nullptr};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 256) {
        set_last_error("vof_interface_compact_noalloc: cudaGetDevice", e);
        *st = PLIC_ERR_CUDA;
        return nullptr;
    }
    std::lock_guard<std::mutex> lk(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_tiles);
        if (e != cudaSuccess || !p) {
            set_last_error("vof_interface_compact_noalloc: cudaGetSymbolAddress", e);
            *st = PLIC_ERR_CUDA;
            return nullptr;
        }
        addr[dev] = reinterpret_cast<int*>(p);
    }
    return addr[dev];
}

}  // namespace plic

extern "C" plic_status vof_interface_compact_noalloc(const float* phi, int nx, int ny, int nz,
                                                     int32_t* idx, int64_t idx_capacity,
                                                     int64_t* d_count, void* stream) {
    using namespace plic;
    if (nx < 0 || ny < 0 || nz < 0 || idx_capacity < 0 || !d_count) return PLIC_ERR_ARG;
    const int64_t ncell = (int64_t)nx * ny * nz;
    if (ncell > (int64_t)PLIC_NOALLOC_MAX_CELLS) {
        set_limit_error(ncell);
        return PLIC_ERR_ARG;
    }
    if (ncell > 0 && (!phi || (!idx && idx_capacity > 0))) return PLIC_ERR_ARG;
    if (!aligned(d_count, 8) || (phi && !aligned(phi, 4)) || (idx && !aligned(idx, 4)))
        return PLIC_ERR_ALIGN;
    plic_status st = PLIC_OK;
    int* tiles = noalloc_scratch(&st);
    if (!tiles) return st;
    cudaStream_t s = as_stream(stream);
    if (nx < 3 || ny < 3 || nz < 3) {        // no cell has all 26 neighbours inside
        cudaError_t e = cudaMemsetAsync(d_count, 0, sizeof(int64_t), s);
        if (e != cudaSuccess) { set_last_error("vof_interface_compact_noalloc", e); return PLIC_ERR_CUDA; }
        return PLIC_OK;
    }
    // every tile entry that a pass reads is written earlier in the same call,
    // so the contents left by a previous call need no clearing
    const CompactPlan p = compact_plan(nx, ny, nz);
    if (info_ints(p) > kNoAllocInts) {
        set_limit_error(ncell);
        return PLIC_ERR_ARG;
    }
    const cudaError_t e = compact_passes(phi, nx, ny, nz, p, tiles, nullptr, idx, idx_capacity, d_count, s);
    if (e != cudaSuccess) { set_last_error("vof_interface_compact_noalloc", e); return PLIC_ERR_CUDA; }
    return check_launch("vof_interface_compact_noalloc");
}
