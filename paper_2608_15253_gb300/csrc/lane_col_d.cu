// Y passes of FP64 3-D grids (conv_lane.cuh, lane_col_kernel): shapes by line
// length.
#include "conv_lane.cuh"
#include "lane.h"

namespace mm {

#define MM_COL_D(X) \
    X(32, 4, 8, 16) X(36, 4, 9, 16) X(48, 6, 8, 16) X(54, 6, 9, 16) X(64, 8, 8, 8) X(72, 8, 9, 8) X(81, 9, 9, 8) X(96, 8, 12, 8) \
    X(108, 9, 12, 8) X(128, 8, 16, 8) X(144, 9, 16, 8) X(162, 9, 18, 8) X(192, 12, 16, 8) X(216, 12, 18, 8) X(243, 9, 27, 8) X(256, 16, 16, 8) \
    X(288, 16, 18, 8) X(324, 18, 18, 8) X(384, 24, 16, 8) X(432, 24, 18, 8) X(512, 32, 16, 8)

template <> LaneKern<double> lane_col<double>(int L, bool forward) {
    switch (L) {
#define MM_CASE(l, g, q, tp) \
    case l: return {forward ? lane_col_kernel<double, l, g, q, tp, 1, 1> : lane_col_kernel<double, l, g, q, tp, -1, 1>, g * tp, tp, \
                    lane_col_smem<double, l, g, q, tp>(), false};
        MM_COL_D(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
