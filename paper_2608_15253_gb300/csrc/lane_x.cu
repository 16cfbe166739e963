// X passes of FP32 rows (lane_x.cuh): shapes by half length M = G * Q.  One
// GB300, forward pass with the RK45 stage formed in it, mean of the stages:
//   512x512x64  239 us against 380 for a row per warp in radix-8 passes
//   250x250x40  52 us against 71;  256x256x16 24 us against 32
//   1024x1024   22 us plain, 30 with the stage, against 51 plus 15 (16 threads of 64 values a
//   row; 32 of 32 leave half of them idle in the split: c2r 19 against 15 us on cached rows)
//   150x150x24 with a region map 20 us against 43 plus 10 for the stage state
//   formed by a kernel of its own
// inverse: 150x150x24 11.5 us against 29, 250x250x40 35 against 39, 1024x1024 20 against 41.
// The straight-line code of a row is long; the kernels are kept to one body
// per kind of row without branches in the split (with a body per stage and
// the general rows in the same kernel: 285, 63 and 33 us, half of a small
// grid's time in instruction fetches).
#include "lane.h"
#include "lane_x.cuh"

namespace mm {

template <> XLane<float> lane_x<float>(int M) {
    switch (M) {
#define MM_CASE(m, g, q, rows) \
    case m: return {{lane_r2c_kernel<float, m, g, q, rows, X_PLAIN>, lane_r2c_kernel<float, m, g, q, rows, X_STAGE>, lane_r2c_any_f(m)}, \
                    lane_c2r_kernel<float, m, g, q, rows>, g, rows, XSplit<m, g, q>::LINE * sizeof(lcx<float>)};
        MM_XLANE_SHAPES(MM_CASE)
        MM_XLANE_LONG(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
