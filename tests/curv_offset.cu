// curv_offset.cu -- the offsets of the curvature step's neighbour solves (optimised
// SZ), paired and one at a time, for given normals and volumes.
#include "../paper_2006_12838_gb300/csrc/host_common.h"
#include "../paper_2006_12838_gb300/csrc/vof_curvature_pair.cuh"

__global__ void k_offsets(const float* nx, const float* ny, const float* nz, const float* V0, float* pair,
                          float* single, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    plic::CellPlic<plic::M_SZ_OPT> pl;
    pl.prepare(nx[i], ny[i], nz[i]);
    pair[i] = plic::offset_two<plic::M_SZ_OPT>(pl, make_float2(0.5f, V0[i])).y;
    single[i] = pl.offset(V0[i]);
}

extern "C" int curv_offsets(const float* nx, const float* ny, const float* nz, const float* V0, float* pair,
                            float* single, int64_t n) {
    k_offsets<<<(unsigned)((n + 127) / 128), 128>>>(nx, ny, nz, V0, pair, single, n);
    return (int)cudaDeviceSynchronize();
}
