// Middle pass of 3-D grids (conv_lane.cuh, lane_conv_kernel): shapes by line
// length.  One GB300, one evaluation:
//   512x512x64 (L = 128)  570 us against 590 for one column per thread with
//                         the components in turn; 3.5 TB/s of the 2.02 GB
//   250x250x40 (L = 81)   111 us against 137
//   150x150x24 (L = 48)   22.6 us against 26.7
//   256x256x16 (L = 32)   30.4 us against 34.5 for whole lines in registers
// FP32 lines up to 108 points take one column per thread: half the registers
// of two columns (96 against 168) keep twice the warps on an SM, which hides
// the exchange better than packed arithmetic shortens it (L = 48: 22.6
// against 26.7 us).  At 128 points shared memory limits the warps, and two
// columns per thread with the inputs prefetched win (551 against 628 us by
// themselves, 570 in a step).
#include "conv_lane.cuh"
#include "lane.h"

namespace mm {

// (L, G, Q, TP, MINB), 16 columns or more per CTA
#define MM_CONV3_F(X) \
    X(18, 2, 9, 32, 1) X(24, 3, 8, 32, 1) X(27, 3, 9, 32, 1) X(32, 4, 8, 32, 5) X(36, 4, 9, 32, 4) X(48, 6, 8, 16, 6) \
    X(54, 6, 9, 16, 6) X(64, 8, 8, 16, 5) X(72, 8, 9, 16, 5) X(81, 9, 9, 16, 4) X(96, 8, 12, 16, 4) X(108, 12, 9, 16, 2)
#define MM_CONV3_D(X) \
    X(18, 2, 9, 16, 1) X(24, 3, 8, 16, 1) X(27, 3, 9, 16, 1) X(32, 4, 8, 16, 1) X(36, 4, 9, 16, 1) X(48, 6, 8, 8, 1) \
    X(54, 6, 9, 8, 1) X(64, 8, 8, 8, 1) X(72, 8, 9, 8, 1) X(81, 9, 9, 8, 1) X(96, 8, 12, 8, 1) X(128, 8, 16, 8, 1)

template <> LaneKern<float> lane_conv3<float>(int L, int columns) {
    switch (L) {
#define MM_CASE(l, g, q, tp, mb) \
    case l: return {lane_conv_kernel<float, l, g, q, tp, 1, true, mb, false>, g * tp, tp, lane_conv_smem<float, l, g, q, tp, 6, false>(), false};
        MM_CONV3_F(MM_CASE)
#undef MM_CASE
        case 128: return {lane_conv_kernel<float2, 128, 8, 16, 8, 3, true, 2, true>, 192, 16, lane_conv_smem<float2, 128, 8, 16, 8, 6, true>(), true};
        default: return lane_conv3_long(L, columns);
    }
}

template <> LaneKern<double> lane_conv3<double>(int L, int) {
    switch (L) {
#define MM_CASE(l, g, q, tp, mb) \
    case l: return {lane_conv_kernel<double, l, g, q, tp, 1, true, mb, false>, g * tp, tp, lane_conv_smem<double, l, g, q, tp, 6, false>(), false};
        MM_CONV3_D(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
