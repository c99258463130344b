// Host-side driver for gf_coop.h, for the CPU tests: a launch that takes at most
// `fits` CTAs, or fails with `error` whatever the grid.
#include "gf_coop.h"

// tried[0 .. return): the grids launched; *err: what coop_launch returned;
// *recorded: the error still on the record, as cudaGetLastError would give it
extern "C" int coop_run(int grid, int fits, int error, int *tried, int *err, int *recorded)
{
    const int REFUSED = 720;
    int n = 0;
    *recorded = 0;
    *err = gf::coop_launch(
        grid, REFUSED,
        [&](int g) {
            tried[n++] = g;
            const int e = error ? error : (g > fits ? REFUSED : 0);
            if (e) *recorded = e;
            return e;
        },
        [&] { *recorded = 0; });
    return n;
}
