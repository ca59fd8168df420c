// Test harness for csrc/pool_book.h: reads the number of workers and the budget,
// then lines "s w in_use" (worker w starts a job; writes the workers whose pools are
// trimmed and what idle pools keep in all) and "f w bytes" (it ends).
#include <stdio.h>

#include "pool_book.h"

int main() {
    int n, w;
    size_t budget, v;
    char op;
    if (scanf("%d %zu", &n, &budget) != 2) return 1;
    smf::PoolBook b;
    b.kept.assign(n, 0);
    while (scanf(" %c %d %zu", &op, &w, &v) == 3) {
        if (op == 'f') {
            b.finish(w, v);
            continue;
        }
        b.start(w, v, budget, [](int i) { printf("%d ", i); });
        size_t sum = 0;
        for (size_t k : b.kept) sum += k;
        printf("| %zu\n", sum);
    }
    return 0;
}
