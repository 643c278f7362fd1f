// vof_curvature.cu -- curvature over interface-cell lists (Sec. 4.2), for one
// field (vof_curvature, vof_laplace_pressure) and for many fields in one
// persistent launch (vof_curvature_batched).
//
// Two layouts of the per-cell work: one thread per interface cell
// (vof_curvature_tpc.cu; every single-field call and the batched default)
// and eight lanes per cell (vof_curvature_coop.cuh; a batched tuning
// option).  Measured on GB300: 2.69 M cells of 64 fields in 0.22 ms with one
// thread per cell against 0.90 ms with eight lanes; the 56 478-cell list of the
// 256^3 curvature field in 8.0 us (eight lanes, at an earlier stage: 33.3 against
// 12.5).  The single-field entry keeps one layout for every
// list length, so that a cell's kappa does not depend on the list (or the
// buffer) it comes in.
#include "host_common.h"
#include "workspace.h"
#include "vof_curvature_coop.cuh"

namespace plic {

constexpr int CO_THREADS = 128;       // 4 warps per block
constexpr int CO_WARPS = CO_THREADS / 32;
static_assert(TPC_THREADS == CO_THREADS, "one block shape for both layouts");
// Layout of the batched kernel when the tuning leaves it open (lanes per cell).
constexpr int BATCHED_DEFAULT_LANES = 1;

// Persistent batched kernel: each warp claims tickets of `chunk` cells (a
// multiple of 32) of the concatenated interface lists from a device counter
// and stops when the tickets pass the total; no warp waits for another.
template <int METHOD, int FIT>
__global__ void __launch_bounds__(CO_THREADS)
k_vof_curvature_batched(const vof_field* __restrict__ fields, const int64_t* __restrict__ prefix,
                        int n_fields, int64_t total, int chunk,
                        unsigned long long* __restrict__ ticket, uint32_t flags) {
    __shared__ float smem[CO_WARPS][CO_BATCH * CO_VALS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    pdl_wait();                  // the tables are written
    for (;;) {
        unsigned long long t = 0;
        if (lane == 0) t = atomicAdd(ticket, (unsigned long long)chunk);
        const int64_t start = (int64_t)__shfl_sync(0xffffffffu, t, 0);
        if (start >= total) break;
        const int64_t end = start + chunk < total ? start + chunk : total;
        for (int64_t b0 = start; b0 < end; b0 += CO_BATCH) {
            // lane l locates entry b0 + l: field (binary search on the prefix)
            // and position in that field's list
            const int64_t gi = b0 + lane;
            int f = 0;
            int64_t kk = 0;
            if (gi < end) {
                int lo = 0, hi = n_fields - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (__ldg(prefix + mid) <= gi) lo = mid; else hi = mid - 1;
                }
                f = lo;
                kk = gi - __ldg(prefix + lo);
            }
            auto fetch = [&](int slot) {
                const int fs = __shfl_sync(0xffffffffu, f, slot);
                const long long ks = __shfl_sync(0xffffffffu, (long long)kk, slot);
                const vof_field& F = fields[fs];
                CoCell c;
                c.phi = F.phi; c.nx = F.nx; c.nxy = (int64_t)F.nx * F.ny;
                c.valid = b0 + slot < end;
                c.c = c.valid ? (int64_t)__ldg(F.idx + ks) : 0;
                c.out = F.kappa + ks;
                return c;
            };
            co_warp_batch<METHOD, FIT>(fetch, CO_BATCH, flags, 1.0f, smem[warp]);
        }
    }
}

// The batch's tables, passed by value: a kernel writes them to the workspace and clears
// the ticket; the batch's kernel is launched behind it (pdl_wait).  Two copies from
// pageable memory and a memset in its place: 213.6 instead of 205 us per call of
// the 64-field batch, and a captured call read the host's tables, long gone,
// at each replay.  Up to 64 fields go in one launch of 3.6 KB of parameters, more in
// launches of 512 (28.7 KB; a launch takes at most 32 KB), a block of 64 threads per 64
// fields.  Whole calls, lists of 607 cells (in brackets: launches of 64; the copies): 65
// fields 12.4 us (14.7; 22.4), 300 21.0 (37.2; 30.0), 1000 52 (111; 61), 10 000 425 (982; 467).
constexpr int TABLE_THREADS = 64;
template <int N>
struct BatchTable {
    vof_field f[N];
    int64_t prefix[N];                   // list entries before each field
    int first, count;
};

template <int N>
__global__ void __launch_bounds__(TABLE_THREADS)
k_batch_table(const __grid_constant__ BatchTable<N> t, vof_field* __restrict__ fields, int64_t* __restrict__ prefix,
              unsigned long long* __restrict__ ticket) {
    const int i = blockIdx.x * TABLE_THREADS + threadIdx.x;
    if (i < t.count) {
        fields[t.first + i] = t.f[i];
        prefix[t.first + i] = t.prefix[i];
    }
    if (i == 0) *ticket = 0ull;
    pdl_trigger();
}

// Fields [first, first + count) of a batch, count <= N; `before`: the list entries before
// them, moved on.
template <int N>
static cudaError_t launch_table(const vof_field* fields, size_t first, int count, int64_t& before, vof_field* d_fields,
                                int64_t* d_pre, unsigned long long* d_ticket, cudaStream_t s) {
    BatchTable<N> t;
    t.first = (int)first;
    t.count = count;
    for (int j = 0; j < count; ++j) {
        t.f[j] = fields[first + j];
        t.prefix[j] = before;
        before += t.f[j].n_iface;
    }
    void* args[] = {(void*)&t, (void*)&d_fields, (void*)&d_pre, (void*)&d_ticket};
    return cudaLaunchKernel(reinterpret_cast<const void*>(&k_batch_table<N>),
                            dim3((unsigned)((count + TABLE_THREADS - 1) / TABLE_THREADS)), dim3(TABLE_THREADS), args, 0, s);
}

#define PLIC_FIT_TABLE(K, M) \
    static const void* K##_tab[4] = { \
        reinterpret_cast<const void*>(&K<M, FIT_FP64>), reinterpret_cast<const void*>(&K<M, FIT_FP32>), \
        reinterpret_cast<const void*>(&K<M, FIT_DF32>), reinterpret_cast<const void*>(&K<M, FIT_AUTO>)};

template <int METHOD>
static const void* pick_batched(int fit) {
    PLIC_FIT_TABLE(k_vof_curvature_batched, METHOD)
    return k_vof_curvature_batched_tab[fit];
}

// Fit precision from the flags: one of FIT_FP32 / FIT_DF32 / FIT_FP64, or the
// adaptive default; -1 when more than one is set.
static int fit_mode(uint32_t flags) {
    const uint32_t f = flags & (PLIC_FLAG_FIT_FP32 | PLIC_FLAG_FIT_DF32 | PLIC_FLAG_FIT_FP64);
    if (f == 0) return FIT_AUTO;
    if (f == PLIC_FLAG_FIT_FP32) return FIT_FP32;
    if (f == PLIC_FLAG_FIT_DF32) return FIT_DF32;
    if (f == PLIC_FLAG_FIT_FP64) return FIT_FP64;
    return -1;
}

// The eight-lane batched kernel for a method and fit mode.
static const void* select_coop(plic_method m, int fit) {
    switch (m) {
        case PLIC_ANALYTIC: return pick_batched<M_ANALYTIC>(fit);
        case PLIC_SZ_ORIG: return pick_batched<M_SZ_ORIG>(fit);
        case PLIC_SZ_OPT: return pick_batched<M_SZ_OPT>(fit);
        case PLIC_NEWTON: return pick_batched<M_NEWTON>(fit);
        case PLIC_NESTED: return pick_batched<M_NESTED>(fit);
    }
    return nullptr;
}

static const uint32_t kCurvFlags = PLIC_FLAG_POINT_CENTROID | PLIC_FLAG_KAPPA_PAPER_SIGN |
                                   PLIC_FLAG_FIT_FP32 | PLIC_FLAG_FIT_DF32 | PLIC_FLAG_FIT_FP64 |
                                   PLIC_FLAG_NORMAL_CM | PLIC_FLAG_NEIGHBOR_NORMAL;

// vof_curvature and vof_laplace_pressure: out[k] = scale * kappa[k]
static plic_status curvature_entry(const float* phi, int nx, int ny, int nz, const int32_t* idx,
                                   int64_t n_iface, const int64_t* d_n_iface, float* out,
                                   plic_method m, uint32_t flags, float scale, void* stream,
                                   const char* who) {
    // fields of at most 2^31 - 1 cells (int32 list entries; 32-bit stencil offsets)
    if (nx < 3 || ny < 3 || nz < 3 || n_iface < 0 || (int64_t)nx * ny * nz > 2147483647LL)
        return PLIC_ERR_ARG;
    if ((int)m < 0 || (int)m > 4 || (flags & ~kCurvFlags) || fit_mode(flags) < 0) return PLIC_ERR_ARG;
    if (n_iface == 0) return PLIC_OK;
    if (!phi || !idx || !out) return PLIC_ERR_ARG;
    if (!aligned(phi, 4) || !aligned(idx, 4) || !aligned(out, 4) || (d_n_iface && !aligned(d_n_iface, 8)))
        return PLIC_ERR_ALIGN;
    if (flags & PLIC_FLAG_NEIGHBOR_NORMAL)
        return launch_curvature_nn(phi, nx, ny, nz, idx, n_iface, d_n_iface, out, m, flags,
                                   fit_mode(flags), scale, stream, who);
    const void* k = select_tpc(false, m, fit_mode(flags));
    if (!k) return PLIC_ERR_ARG;
    const int grid = stride_grid(k, TPC_THREADS, n_iface);
    void* args[] = {(void*)&phi, (void*)&nx, (void*)&ny, (void*)&idx, (void*)&n_iface,
                    (void*)&d_n_iface, (void*)&out, (void*)&flags, (void*)&scale};
    // a programmatic dependent launch: the list usually comes from the
    // compaction launched just before on the same stream
    cudaError_t e = launch_after(k, dim3(grid), dim3(TPC_THREADS), args, as_stream(stream));
    if (e != cudaSuccess) { set_last_error(who, e); return PLIC_ERR_CUDA; }
    return PLIC_OK;
}

}  // namespace plic

extern "C" plic_status vof_curvature(const float* phi, int nx, int ny, int nz, const int32_t* idx,
                                     int64_t n_iface, const int64_t* d_n_iface, float* kappa,
                                     plic_method m, uint32_t flags, void* stream) {
    return plic::curvature_entry(phi, nx, ny, nz, idx, n_iface, d_n_iface, kappa, m, flags, 1.0f,
                                 stream, "vof_curvature");
}

extern "C" plic_status vof_laplace_pressure(const float* phi, int nx, int ny, int nz,
                                            const int32_t* idx, int64_t n_iface,
                                            const int64_t* d_n_iface, float sigma, float* dp,
                                            plic_method m, uint32_t flags, void* stream) {
    if (!(sigma == sigma)) return PLIC_ERR_ARG;
    return plic::curvature_entry(phi, nx, ny, nz, idx, n_iface, d_n_iface, dp, m, flags,
                                 2.0f * sigma, stream, "vof_laplace_pressure");
}

extern "C" plic_status vof_curvature_batched(const vof_field* fields, int n_fields,
                                             const vof_tuning* tuning, plic_method m,
                                             uint32_t flags, void* workspace, size_t ws_bytes,
                                             void* stream) {
    using namespace plic;
    if (n_fields < 0 || (int)m < 0 || (int)m > 4 || (flags & ~kCurvFlags) || fit_mode(flags) < 0)
        return PLIC_ERR_ARG;
    if (flags & PLIC_FLAG_NEIGHBOR_NORMAL) return PLIC_ERR_UNSUPPORTED;
    if (n_fields == 0) return PLIC_OK;
    if (!fields || !workspace) return PLIC_ERR_ARG;
    if (ws_bytes < plic_workspace_bytes(PLIC_WS_BATCHED, n_fields)) return PLIC_ERR_ARG;
    if (!aligned(workspace, 256)) return PLIC_ERR_ALIGN;
    int threads = CO_THREADS, chunk = 0, bps = 0, lanes = 0;
    if (tuning) {
        threads = tuning->block_threads;
        chunk = tuning->cells_per_chunk;
        bps = tuning->blocks_per_sm;
        lanes = tuning->lanes_per_cell;
        if (threads < 32 || threads > 1024 || (threads & 31) || chunk < 1 || bps < 0 ||
            (lanes != 0 && lanes != 1 && lanes != 8))
            return PLIC_ERR_ARG;
        if (threads != CO_THREADS) return PLIC_ERR_UNSUPPORTED;   // built for 4 warps per block
    }
    if (lanes == 0) lanes = BATCHED_DEFAULT_LANES;
    // argument checks and the total of the list lengths
    const size_t nf = (size_t)n_fields;
    int64_t total = 0;
    for (size_t i = 0; i < nf; ++i) {
        const vof_field& F = fields[i];
        if (F.nx < 3 || F.ny < 3 || F.nz < 3 || F.n_iface < 0 ||
            (int64_t)F.nx * F.ny * F.nz > 2147483647LL ||
            (F.n_iface > 0 && (!F.phi || !F.idx || !F.kappa)))
            return PLIC_ERR_ARG;
        if (!aligned(F.phi, 4) || !aligned(F.idx, 4) || !aligned(F.kappa, 4)) return PLIC_ERR_ALIGN;
        total += F.n_iface;
    }
    if (total == 0) return PLIC_OK;
    const void* k = lanes == 1 ? select_tpc(true, m, fit_mode(flags)) : select_coop(m, fit_mode(flags));
    if (!k) return PLIC_ERR_ARG;
    const int occ = blocks_per_sm(k, threads, 0);
    const int per_sm = bps > 0 ? (bps < occ ? bps : occ) : occ;
    int64_t grid = (int64_t)sm_count() * per_sm;
    // Cells per ticket when the tuning leaves them open: 128, or as few as 32 where
    // the resident warps would get fewer than four tickets each, since the last ones
    // then set the time (0.4 M cells 43.6 us with 128, 37.6 with 32; 1.2 M cells 99 with
    // 128 or 64, 101 with 32; 2.7 M cells 228 and 238).
    if (chunk == 0)
        for (chunk = 128; chunk > CO_BATCH && total < 4 * chunk * grid * CO_WARPS;) chunk /= 2;
    chunk = (chunk + CO_BATCH - 1) / CO_BATCH * CO_BATCH;     // whole warp batches
    char* ws = reinterpret_cast<char*>(workspace);
    const BatchLayout at = batch_layout(nf);
    vof_field* d_fields = reinterpret_cast<vof_field*>(ws);
    int64_t* d_pre = reinterpret_cast<int64_t*>(ws + at.prefix);
    unsigned long long* d_ticket = reinterpret_cast<unsigned long long*>(ws + at.ticket);
    cudaStream_t s = as_stream(stream);
    cudaError_t e = cudaSuccess;
    int64_t before = 0;
    for (size_t i = 0; i < nf && e == cudaSuccess; i += 512)
        e = nf - i <= 64 ? launch_table<64>(fields, i, (int)(nf - i), before, d_fields, d_pre, d_ticket, s)
                         : launch_table<512>(fields, i, (int)(nf - i < 512 ? nf - i : 512), before, d_fields, d_pre,
                                             d_ticket, s);
    if (e != cudaSuccess) { set_last_error("vof_curvature_batched", e); return PLIC_ERR_CUDA; }
    const int64_t need = ((total + chunk - 1) / chunk + CO_WARPS - 1) / CO_WARPS;
    if (grid > need) grid = need;
    if (grid < 1) grid = 1;
    int n_f = n_fields;
    void* args[] = {(void*)&d_fields, (void*)&d_pre, (void*)&n_f, (void*)&total, (void*)&chunk,
                    (void*)&d_ticket, (void*)&flags};
    e = launch_after(k, dim3((unsigned)grid), dim3(threads), args, s);
    if (e != cudaSuccess) { set_last_error("vof_curvature_batched", e); return PLIC_ERR_CUDA; }
    return PLIC_OK;
}
