// X passes of FP32 rows (lane_x.cuh): shapes by half length M = G * Q.  One
// GB300, forward pass with the RK45 stage formed in it, mean of the stages:
//   512x512x64  285 us against 380 for a row per warp in radix-8 passes
//               (6.4 TB/s: what the slopes and the spectrum cost)
//   250x250x40  63 us against 71;  150x150x24 with a region map 20 us against
//               43 plus 10 for the stage state formed by a kernel of its own
// inverse: 150x150x24 11.4 us against 29, 250x250x40 35 against 39.
#include "lane.h"
#include "lane_x.cuh"

namespace mm {

template <> XLane<float> lane_x<float>(int M) {
    switch (M) {
#define MM_CASE(m, g, q, rows) \
    case m: return {lane_r2c_kernel<float, m, g, q, rows>, lane_c2r_kernel<float, m, g, q, rows>, g, rows, XSplit<m, g, q>::LINE * sizeof(lcx<float>)};
        MM_XLANE_SHAPES(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
