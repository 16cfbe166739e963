// X passes of FP64 rows (lane_x.cuh): shapes by half length M = G * Q.  One
// GB300: 64x64x16 21 / 20 us (forward / inverse) against 43 / 48 for the
// runtime-planned shared-memory passes; 128x32 (a row per warp) 12.4 / 10.2
// against 17.4 plus 6.1 for the stage state, and 16.4.
#include "lane.h"
#include "lane_x.cuh"

namespace mm {

template <> XLane<double> lane_x<double>(int M) {
    switch (M) {
#define MM_CASE(m, g, q, rows) \
    case m: return {{lane_r2c_kernel<double, m, g, q, rows, X_PLAIN>, lane_r2c_kernel<double, m, g, q, rows, X_STAGE>, lane_r2c_any_d(m)}, \
                    lane_c2r_kernel<double, m, g, q, rows>, g, rows, XSplit<m, g, q>::LINE * sizeof(lcx<double>), \
                    fine_r2c_kernel<double, m>, fine_c2r_kernel<double, m>, fine_line(m) * sizeof(lcx<double>)};
        MM_XLANE_SHAPES(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
