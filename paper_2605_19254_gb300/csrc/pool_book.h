// What the memory pools of a server's idle workers keep, so that they and the
// running jobs stay within the server's budget.  Called with the server's lock
// held: a worker with kept bytes is idle, and its pool has nothing in flight.
#pragma once

#include <stddef.h>

#include <vector>

namespace smf {

struct PoolBook {
    std::vector<size_t> kept;  // bytes worker i's pool keeps while it is idle

    // Worker w starts a job that brings the running jobs to in_use bytes (its own
    // pool's are among them): idle pools are given back, the largest first, until
    // what is left fits the budget.  trim(i) empties the pool of worker i.
    template <class Trim>
    void start(int w, size_t in_use, size_t budget, Trim trim) {
        kept[w] = 0;
        for (;;) {
            size_t sum = 0;
            int big = 0;
            for (size_t i = 0; i < kept.size(); i++) {
                sum += kept[i];
                if (kept[i] > kept[big]) big = (int)i;
            }
            if (sum == 0 || in_use + sum <= budget) return;
            trim(big);
            kept[big] = 0;
        }
    }
    void finish(int w, size_t bytes) { kept[w] = bytes; }
};

}  // namespace smf
