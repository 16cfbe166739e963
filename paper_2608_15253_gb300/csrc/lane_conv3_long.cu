// Middle pass of FP32 3-D grids of many layers (conv_lane.cuh,
// lane_conv_kernel): shapes by line length.  One GB300, one evaluation of
// 128x128 columns of L/2 points:
//   L = 162   70 us    192   78 us    216   96 us    256  107 us
//       324  170 us    432  206 us    512  227 us   1024  698 us
// against 1.4 to 3.8 ms for the runtime-planned passes and, in the same order,
// 282, 81, 362, 108, 574, 815, 436 and 1861 us for lines split over threads of
// one column or whole in shared memory.  36 bytes of shared memory a point and
// column (exchange and tensor) are what limits them: 8 columns a CTA where two
// CTAs fit an SM or one of 384 threads fills it.  Three groups of threads a
// column (a component each) hide the exchange better than one from 432 points
// on, where one CTA fits an SM; at 162 to 216 points the persistent form, which
// brings the next inputs meanwhile, wins (192: 78 against 89 us), and at 256
// and 324 one thread group for all components (107 against 127 us).
#include "conv_lane.cuh"
#include "lane.h"

namespace mm {

// (L, G, Q, TP, CS, MINB, persistent)
#define MM_CONV3_LONG(X) \
    X(162, 9, 18, 8, 3, 1, true) X(192, 12, 16, 16, 3, 1, true) X(216, 12, 18, 16, 3, 1, true) X(256, 16, 16, 8, 1, 2, false) \
    X(324, 18, 18, 8, 1, 2, false) X(432, 16, 27, 8, 3, 1, false) X(512, 16, 32, 8, 3, 1, false) X(1024, 16, 64, 4, 3, 1, false)
// Where persistent CTAs of 16 columns do not reach half of the SMs: 8 columns and
// one side each, four times as many (L = 192 / 216, 8x8 columns 15.9 / 18.1 -> 9.9 / 12.0 us, 32x32 16.0 / 18.2 -> 12.0 / 14.1).
#define MM_CONV3_FEW(X) X(192, 12, 16, 8, 3, 3, false) X(216, 12, 18, 8, 3, 3, false)

LaneKern<float> lane_conv3_long(int L, int columns) {
#define MM_CASE(l, g, q, tp, cs, mb, st) \
    case l: return {lane_conv_kernel<float, l, g, q, tp, cs, true, mb, st>, cs * g * tp, tp, lane_conv_smem<float, l, g, q, tp, 6, st>(), st};
    if (columns <= 8 * sm_count()) switch (L) {
        MM_CONV3_FEW(MM_CASE)
        default: break;
    }
    switch (L) {
        MM_CONV3_LONG(MM_CASE)
        default: return {};
    }
#undef MM_CASE
}

}  // namespace mm
