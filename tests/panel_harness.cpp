// Test harness for the size rules of the eliminations by panels
// (paper_2605_19254_gb300/csrc/panel.h, compiled for the host): reads lines
// "n L most" and writes the panel's width, the shared memory of that panel and of
// one twice as wide, the limit, and the words of a row.
#include <stdio.h>

#include "panel.h"

int main() {
    long long n;
    int L, most;
    while (scanf("%lld %d %d", &n, &L, &most) == 3) {
        const int C = smf::panel_cluster(n), w = smf::panel_width(n, L, most), x = w ? 2 * w : 1;
        const long long rows = (n + C - 1) / C;
        printf("%d %zu %zu %zu %d\n", w, w ? smf::panel_smem(rows, (long long)w * L, w) : 0,
               smf::panel_smem((n + 15) / 16, (long long)x * L, x), smf::panel_smem_limit(L), smf::panel_stride((w ? w : 1) * L));
    }
    return 0;
}
