// workspace.h -- what lies where in the callers' workspaces, in one place for the
// entries that use them and the size query that callers allocate by.
// No CUDA: tests/workspace_host.cpp compiles it for the host.
#pragma once
#include <stddef.h>
#include <stdint.h>

#include "../../include/plic.h"

namespace plic {

inline size_t round256(size_t b) { return (b + 255) / 256 * 256; }

// vof_curvature_batched: the descriptors, the list entries before each field, and the
// ticket counter on a line of its own (every warp's atomicAdd goes there).
struct BatchLayout {
    size_t prefix, ticket, end;
};
inline BatchLayout batch_layout(size_t n_fields) {
    BatchLayout l;
    l.prefix = n_fields * sizeof(vof_field);
    l.ticket = round256(l.prefix + n_fields * sizeof(int64_t));
    l.end = l.ticket + sizeof(unsigned long long);
    return l;
}

// The size query's answer for n_fields fields: callers hold workspaces of this size,
// so the layout fits into it and not the other way round.
inline size_t batch_workspace(size_t n_fields) {
    return round256(n_fields * (sizeof(vof_field) + sizeof(int64_t)) + 2 * sizeof(int64_t)) + 256;
}

// tiles or blocks of tiles whose counts the write pass sums in front of each block
constexpr int64_t CT_MAX_SUPERS = 8192;

// How a field is cut: cells [base, base + cells) of the flat field (base a
// multiple of 32 cells), tiles of `tile` cells, S tiles per block of pass 1.
struct CompactPlan {
    int64_t base, cells, tiles, supers;
    int tile, S;
};

// Tile sizes: 8192 cells (16 loads of 16 bytes per lane in flight) where that
// fills the chip more than twice (2560 blocks and up), smaller tiles below, where
// the last blocks and, smaller still, a single block set the time (64^3: 248 tiles
// of 1024 cells 5.9 us, 32 tiles of 8192 14 us; with the curvature after it, 256^3
// 24.0 us with 8192 cells and 23.6 with 4096, 301 x 203 x 257 24.0 and 23.7,
// 1 GiB 215 and 219).  S grows once the write pass would have to sum more
// than CT_MAX_SUPERS counts (above 67 M cells; one scan launch in between took
// 11 us on 1 GiB).
inline CompactPlan compact_plan(int nx, int ny, int nz) {
    CompactPlan p;
    const int64_t nxy = (int64_t)nx * ny;
    p.base = nxy & ~(int64_t)31;
    p.cells = nxy * (nz - 1) - p.base;
    p.tile = p.cells >= (int64_t)20 << 20 ? 8192 : p.cells >= (int64_t)1 << 20 ? 4096 : 1024;
    p.tiles = (p.cells + p.tile - 1) / p.tile;
    p.S = 1;
    while ((p.tiles + p.S - 1) / p.S > CT_MAX_SUPERS) p.S *= 2;
    p.supers = (p.tiles + p.S - 1) / p.S;
    return p;
}

// Ints of scratch before the bits: tile infos and block sums.
inline int64_t info_ints(const CompactPlan& p) {
    return (p.tiles + 3) / 4 * 4 + (p.S > 1 ? p.supers : 0);
}

// vof_interface_compact: the infos and sums, then one word of bits per 32 cells, whole
// chunks (512 cells): where the bits begin, and the end of all.
inline size_t compact_bits(const CompactPlan& p) { return round256((size_t)info_ints(p) * sizeof(int)); }
inline size_t compact_bytes(const CompactPlan& p) { return compact_bits(p) + (size_t)((p.cells + 511) / 512) * 64; }

// The size query's answer for a field of n cells of any shape: two words per 8192 cells and
// one per 16 (the infos and sums take at most one word per 819 cells).
inline size_t compact_workspace(int64_t n) {
    return round256((size_t)((n + 8191) / 8192 * 2 + 1) * sizeof(int)) + round256((size_t)(n / 16 + 1) * sizeof(unsigned));
}

}  // namespace plic
