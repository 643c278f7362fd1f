// workspace_host.cpp -- csrc/workspace.h on the host: the batched call's parts lie in
// order, aligned and inside the size that the query answers.  Prints how many counts
// of fields fail, then the sizes for 0 .. 3000 fields.
#include <cstdio>

#include "../paper_2006_12838_gb300/csrc/workspace.h"

int main() {
    long bad = 0;
    for (size_t n = 1; n <= 3000; ++n) {
        const plic::BatchLayout l = plic::batch_layout(n);
        bad += l.prefix < n * sizeof(vof_field) || l.prefix % 8 || l.ticket < l.prefix + n * sizeof(int64_t) ||
               l.ticket % 8 || l.end < l.ticket + 8 || l.end > plic::batch_workspace(n);
    }
    printf("%ld\n", bad);
    for (size_t n = 0; n <= 3000; ++n) printf("%zu\n", plic::batch_workspace(n));
    return 0;
}
