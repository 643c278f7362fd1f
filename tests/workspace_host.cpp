// workspace_host.cpp -- csrc/workspace.h on the host: the parts of the batched call's and of
// the compaction's workspaces lie in order, aligned and inside the sizes that the query
// answers.  Prints how many counts of fields and how many field shapes fail, then the
// sizes for 0 .. 3000 fields.
#include <cmath>
#include <cstdio>
#include <random>

#include "../paper_2006_12838_gb300/csrc/workspace.h"

int main() {
    long bad = 0;
    for (size_t n = 1; n <= 3000; ++n) {
        const plic::BatchLayout l = plic::batch_layout(n);
        bad += l.prefix < n * sizeof(vof_field) || l.prefix % 8 || l.ticket < l.prefix + n * sizeof(int64_t) ||
               l.ticket % 8 || l.end < l.ticket + 8 || l.end > plic::batch_workspace(n);
    }
    printf("%ld\n", bad);
    // shapes around the thresholds of the tile size and of the block sums, thin and long
    // ones, and random ones up to 2^31 - 1 cells
    bad = 0;
    std::mt19937_64 r(1);
    auto check = [&](long nx, long ny, long nz) {
        if (nx < 3 || ny < 3 || nz < 3 || nx * ny > 2147483647L / nz) return;
        const plic::CompactPlan p = plic::compact_plan((int)nx, (int)ny, (int)nz);
        const long n = nx * ny * nz;
        bad += p.base % 32 || p.base > nx * ny || p.base + p.cells != nx * ny * (nz - 1) || p.tiles * p.tile < p.cells ||
               p.supers > plic::CT_MAX_SUPERS || p.supers * p.S < p.tiles || p.S > 32 ||
               plic::compact_bits(p) < (size_t)plic::info_ints(p) * 4 || plic::compact_bytes(p) > plic::compact_workspace(n) ||
               (n <= PLIC_NOALLOC_MAX_CELLS && plic::info_ints(p) > 2 * (PLIC_NOALLOC_MAX_CELLS / 8192) + 1);
    };
    for (long at : {1L << 20, 20L << 20, 8192L * 8192L, 2 * 8192L * 8192L, 4 * 8192L * 8192L, 1L << 28, 2147483647L})
        for (long a : {3L, 4L, 31L, 32L, 33L, 301L, 1024L})
            for (long b : {3L, 5L, 64L, 203L, 512L})
                for (long d = -2; d <= 2; ++d) {
                    check(a, b, at / (a * b) + d);
                    check(a, at / (a * b) + d, b);
                    check(at / (a * b) + d, a, b);
                }
    for (int i = 0; i < 200000; ++i) {
        long e[3];
        for (long& x : e) x = (long)std::exp2(1.5 + 12 * (r() >> 11) * 0x1p-53);
        check(e[0], e[1], e[2]);
    }
    printf("%ld\n", bad);
    for (size_t n = 0; n <= 3000; ++n) printf("%zu\n", plic::batch_workspace(n));
    return 0;
}
