// Middle pass of FP64 films (conv_lane.cuh, lane_film_kernel): shapes by
// line length, two columns per CTA so that the few columns of a film reach
// every SM's FP64 units (two fused multiply-adds per clock each).
#include "conv_lane.cuh"
#include "lane.h"
#include "lane_x.cuh"

namespace mm {

#define MM_FILM_D(X) \
    X(16, 4, 4) X(18, 6, 3) X(24, 6, 4) X(27, 9, 3) X(32, 8, 4) X(36, 9, 4) X(48, 8, 6) X(54, 9, 6) X(64, 8, 8) X(72, 9, 8) \
    X(81, 9, 9) X(96, 12, 8) X(108, 12, 9) X(128, 16, 8) X(144, 16, 9) X(162, 18, 9) X(192, 16, 12) X(216, 18, 12) \
    X(243, 27, 9) X(256, 16, 16) X(288, 18, 16) X(324, 18, 18) X(384, 24, 16) X(432, 24, 18) X(512, 32, 16)

template <> LaneKern<double> lane_film<double>(int L) {
    switch (L) {
#define MM_CASE(l, g, q) case l: return {lane_film_kernel<double, l, g, q, 2>, 3 * g * 2, 2, lane_film_smem<double, l, g, q, 2>(), false};
        MM_FILM_D(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

FineFilm fine_film(int L) {
    switch (L) {
#define MM_CASE(l, g, q) case l: return {fine_film_kernel<double, l>, 3 * fine_line(l) * sizeof(lcx<double>)};
        MM_FILM_D(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
