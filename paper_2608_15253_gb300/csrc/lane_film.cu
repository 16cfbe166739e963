// Middle pass of one FP32 film (conv_lane.cuh, lane_film_kernel): shapes by
// line length.  One GB300, one evaluation: 512x512 10.4 us (49 us with the
// shared-memory Stockham kernel), 256x256 8.3 us (17.5 with three components
// per thread), 200x50 6.2 us (12.1).  Two columns per lane up to 512 points;
// one above, where two would need 240 registers (12.4 against 10.4 us).
#include "conv_lane.cuh"
#include "lane.h"

namespace mm {

#define MM_FILM_F2(X) \
    X(16, 4, 4) X(18, 6, 3) X(24, 6, 4) X(27, 9, 3) X(32, 8, 4) X(36, 9, 4) X(48, 8, 6) X(54, 9, 6) X(64, 8, 8) X(72, 9, 8) \
    X(81, 9, 9) X(96, 12, 8) X(108, 12, 9) X(128, 16, 8) X(144, 16, 9) X(162, 18, 9) X(192, 16, 12) X(216, 18, 12) \
    X(243, 27, 9) X(256, 16, 16) X(288, 18, 16) X(324, 18, 18) X(384, 16, 24) X(432, 18, 24) X(486, 18, 27) X(512, 16, 32)
#define MM_FILM_F1(X) X(576, 24, 24) X(648, 27, 24) X(729, 27, 27) X(768, 32, 24) X(864, 32, 27) X(972, 36, 27) X(1024, 32, 32)

template <> LaneKern<float> lane_film<float>(int L) {
    switch (L) {
#define MM_CASE(l, g, q) case l: return {lane_film_kernel<float2, l, g, q, 2>, 3 * g * 2, 4, lane_film_smem<float2, l, g, q, 2>(), false};
        MM_FILM_F2(MM_CASE)
#undef MM_CASE
#define MM_CASE(l, g, q) case l: return {lane_film_kernel<float, l, g, q, 4>, 3 * g * 4, 4, lane_film_smem<float, l, g, q, 4>(), false};
        MM_FILM_F1(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
