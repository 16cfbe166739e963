// Y passes of FP32 3-D grids (conv_lane.cuh, lane_col_kernel): shapes by line
// length.  One GB300, forward / inverse:
//   512x512x64 (L = 1024)  241 / 258 us against 309 / 317 for the
//                          shared-memory Stockham kernel (four passes)
//   250x250x40 (L = 512)   42 / 45 us against 50 / 51
//   150x150x24 (L = 324)   14.7 / 13.3 us against 20.3 / 20.1
//   256x7x32 (L = 16)      6.1 / 6.3 us against 7.6 / 8.0
// One exchange instead of a barrier per radix; the load latency of a CTA is
// what is left.  Two columns per lane halve the instructions, one halves the
// registers and doubles the warps: forward, where half of a line is zeros and
// fewer loads are on their way, one column wins at most of the long lengths
// (L = 1024: 240 against 275 us, 648: 78 against 94, 512: 41 against 48); at 384, 486,
// 576 and 972 its registers do not allow more warps (576: 61 against 53).
// Inverse it wins at 729 and 768 alone (86 and 118 against 95 and 123 us; 1024: 290
// against 253).
#include "conv_lane.cuh"
#include "lane.h"

namespace mm {

// one column per lane
#define MM_COL_FWD1(X) \
    X(243, 9, 27, 8, 4) X(324, 18, 18, 16, 3) X(432, 16, 27, 8, 4) X(512, 16, 32, 8, 4) X(648, 24, 27, 8, 2) X(729, 27, 27, 8, 2) \
    X(768, 24, 32, 8, 2) X(864, 27, 32, 8, 2) X(1024, 32, 32, 8, 2)
#define MM_COL_INV1(X) X(729, 27, 27, 8, 2) X(768, 24, 32, 8, 2)
// two columns per lane
#define MM_COL_BOTH2(X) \
    X(16, 4, 4, 32, 1) X(32, 4, 8, 32, 1) X(36, 4, 9, 32, 1) X(48, 6, 8, 16, 1) X(54, 6, 9, 16, 1) X(64, 8, 8, 16, 1) X(72, 8, 9, 16, 1) X(81, 9, 9, 16, 1) \
    X(96, 8, 12, 16, 1) X(108, 9, 12, 16, 1) X(128, 8, 16, 16, 1) X(144, 9, 16, 16, 1) X(162, 9, 18, 8, 1) X(192, 12, 16, 8, 3) X(216, 12, 18, 8, 3) \
    X(256, 16, 16, 8, 3) X(288, 16, 18, 8, 3) X(384, 16, 24, 8, 2) X(486, 18, 27, 8, 2) X(576, 24, 24, 4, 3) X(972, 27, 36, 4, 2)
#define MM_COL_INV2(X) \
    X(243, 9, 27, 8, 1) X(324, 18, 18, 8, 3) X(432, 16, 27, 8, 2) X(512, 16, 32, 8, 2) X(648, 24, 27, 4, 2) X(864, 27, 32, 4, 2) X(1024, 32, 32, 4, 2)

template <> LaneKern<float> lane_col<float>(int L, bool forward) {
#define MM_CASE(N, DIR, l, g, q, tp, mb) \
    case l: return {lane_col_kernel<N, l, g, q, tp, DIR, mb>, g * tp, lane<N>::width * tp, lane_col_smem<N, l, g, q, tp>(), false};
#define MM_F1(l, g, q, tp, mb) MM_CASE(float, 1, l, g, q, tp, mb)
#define MM_F2(l, g, q, tp, mb) MM_CASE(float2, 1, l, g, q, tp, mb)
#define MM_I1(l, g, q, tp, mb) MM_CASE(float, -1, l, g, q, tp, mb)
#define MM_I2(l, g, q, tp, mb) MM_CASE(float2, -1, l, g, q, tp, mb)
    if (forward) switch (L) {
        MM_COL_FWD1(MM_F1)
        MM_COL_BOTH2(MM_F2)
        default: return {};
    }
    switch (L) {
        MM_COL_INV1(MM_I1)
        MM_COL_INV2(MM_I2)
        MM_COL_BOTH2(MM_I2)
        default: return {};
    }
#undef MM_F1
#undef MM_F2
#undef MM_I1
#undef MM_I2
#undef MM_CASE
}

}  // namespace mm
