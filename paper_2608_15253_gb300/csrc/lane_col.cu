// Y passes of FP32 3-D grids (conv_lane.cuh, lane_col_kernel): shapes by line
// length, two columns per lane.  One GB300, forward / inverse:
//   512x512x64 (L = 1024)  273 / 253 us against 309 / 317 for the
//                          shared-memory Stockham kernel (four passes)
//   250x250x40 (L = 512)   48 / 44 us against 50 / 51
//   150x150x24 (L = 324)   12.3 / 10.3 us against 20.3 / 20.1
// One exchange instead of a barrier per radix; the load latency of a CTA is
// what is left (half of the warps' cycles at L = 1024).
#include "conv_lane.cuh"
#include "lane.h"

namespace mm {

#define MM_COL_F(X) \
    X(32, 4, 8, 32, 1) X(36, 4, 9, 32, 1) X(48, 6, 8, 16, 1) X(54, 6, 9, 16, 1) X(64, 8, 8, 16, 1) X(72, 8, 9, 16, 1) X(81, 9, 9, 16, 1) \
    X(96, 8, 12, 16, 1) X(108, 9, 12, 16, 1) X(128, 8, 16, 16, 1) X(144, 9, 16, 16, 1) X(162, 9, 18, 8, 1) X(192, 12, 16, 8, 3) X(216, 12, 18, 8, 3) \
    X(243, 9, 27, 8, 1) X(256, 16, 16, 8, 3) X(288, 16, 18, 8, 3) X(324, 18, 18, 8, 3) X(384, 16, 24, 8, 2) X(432, 16, 27, 8, 2) \
    X(486, 18, 27, 8, 2) X(512, 16, 32, 8, 2) X(576, 24, 24, 4, 3) X(648, 24, 27, 4, 2) X(729, 27, 27, 4, 2) X(768, 24, 32, 4, 2) \
    X(864, 27, 32, 4, 2) X(972, 27, 36, 4, 2) X(1024, 32, 32, 4, 2)

template <> LaneKern<float> lane_col<float>(int L, bool forward) {
    switch (L) {
#define MM_CASE(l, g, q, tp, mb) \
    case l: return {forward ? lane_col_kernel<float2, l, g, q, tp, 1, mb> : lane_col_kernel<float2, l, g, q, tp, -1, mb>, g * tp, 2 * tp, \
                    lane_col_smem<float2, l, g, q, tp>(), false};
        MM_COL_F(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
