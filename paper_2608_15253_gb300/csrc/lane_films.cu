// Middle pass over the planes of many FP32 films (conv_lane.cuh,
// lane_conv_kernel without the z axis): shapes by line length.  Classes of
// the 1024-replica ensemble, one stage: 128^2 x 186 59.8 us (64.9 before),
// 96^2 x 213 41.3 (49.5), 64^2 x 200 18.4 (19.0), 48^2 x 207 14.6 (17.9),
// 32^2 x 218 8.2 (11.6).  FP64 ensembles do not exist.
#include "conv_lane.cuh"
#include "lane.h"

namespace mm {

#define MM_FILMS(X) \
    X(32, 4, 8, 32, 4) X(36, 4, 9, 32, 4) X(48, 6, 8, 16, 6) X(54, 6, 9, 16, 6) X(64, 8, 8, 16, 6) X(72, 8, 9, 16, 5) X(81, 9, 9, 16, 4) \
    X(96, 8, 12, 16, 4) X(108, 12, 9, 16, 4) X(128, 8, 16, 16, 3) X(144, 9, 16, 16, 2) X(162, 9, 18, 8, 4) X(192, 12, 16, 8, 4) \
    X(216, 12, 18, 8, 3) X(256, 16, 16, 8, 3)

template <> LaneKern<float> lane_films<float>(int L) {
    switch (L) {
#define MM_CASE(l, g, q, tp, mb) \
    case l: return {lane_conv_kernel<float, l, g, q, tp, 1, false, mb, false>, g * tp, tp, lane_conv_smem<float, l, g, q, tp, 4, false>(), false};
        MM_FILMS(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

template <> LaneKern<double> lane_films<double>(int) { return {}; }

}  // namespace mm
