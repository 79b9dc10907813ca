// Test harness (host only): the runs that launch_runs (pv_runs.h) cuts items into.
#include "pv_runs.h"

// x, y: the items' extents. runs = (first, count, x, y) of each launch, at most max_runs; a launch numbered fail_at
// returns 7. Returns what launch_runs returned; *n_runs launches were made.
extern "C" int cut_runs(int first, int n, const long long* x, const long long* y, int fail_at, long long* runs, int max_runs,
                        int* n_runs) {
    *n_runs = 0;
    return pv::launch_runs(first, n, [&](int i) { return pv::RunExtent{x[i], y[i]}; },
                           [&](int at, int m, pv::RunExtent most) {
                               if (*n_runs < max_runs) {
                                   long long* r = runs + 4 * *n_runs;
                                   r[0] = at;
                                   r[1] = m;
                                   r[2] = most.x;
                                   r[3] = most.y;
                               }
                               return (*n_runs)++ == fail_at ? 7 : 0;
                           });
}
