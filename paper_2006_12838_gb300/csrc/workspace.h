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

}  // namespace plic
