// Column kernels of conv_lane.cuh, looked up by line length: launch shape and
// entry point, or kern == nullptr where the length has none (the callers then
// take the runtime-planned path).  Each table lives in its own translation
// unit so that they compile in parallel.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace mm {

template <typename T> struct LaneArgs;

template <typename T>
struct LaneKern {
    void (*kern)(LaneArgs<T>) = nullptr;
    int threads = 0, cols = 0;      // per CTA
    size_t smem = 0;
    bool persistent = false;        // CTAs loop over the column tiles
};

template <typename T> LaneKern<T> lane_conv3(int L, int columns);   // middle pass of a 3-D grid, columns of one side
template <typename T> LaneKern<T> lane_film(int L);             // middle pass of one film
template <typename T> LaneKern<T> lane_films(int L);            // middle pass of many films
template <typename T> LaneKern<T> lane_col(int L, bool forward);    // Y passes of a 3-D grid

template <> LaneKern<float> lane_conv3<float>(int L, int columns);
template <> LaneKern<double> lane_conv3<double>(int L, int columns);
LaneKern<float> lane_conv3_long(int L, int columns);            // its lines of 162 points and more
template <> LaneKern<float> lane_film<float>(int L);
template <> LaneKern<double> lane_film<double>(int L);
template <> LaneKern<float> lane_films<float>(int L);
template <> LaneKern<double> lane_films<double>(int L);
template <> LaneKern<float> lane_col<float>(int L, bool forward);
template <> LaneKern<double> lane_col<double>(int L, bool forward);

// X passes of lane_x.cuh: `group` threads and `line` bytes of shared memory
// per row, at most `rows` rows per CTA.
template <typename T> struct XLaneArgs;

// FP32 rows of half length 1024, for the separate X passes alone
#define MM_XLANE_LONG(X) X(1024, 16, 64, 4)

template <typename T>
struct XLane {
    void (*r2c[3])(XLaneArgs<T>) = {};          // by XInput: plain rows, stage state, anything
    void (*c2r)(XLaneArgs<T>) = nullptr;
    int group = 0, rows = 0;
    size_t line = 0;
    void (*fine_r2c)(XLaneArgs<T>) = nullptr;   // a row per warp, `fine_line` bytes each (FP64)
    void (*fine_c2r)(XLaneArgs<T>) = nullptr;
    size_t fine_line = 0;
};

// Middle pass of one FP64 film in the row-per-warp passes (lane_x.cuh).
template <typename T> struct FineFilmArgs;
struct FineFilm {
    void (*kern)(FineFilmArgs<double>) = nullptr;
    size_t smem = 0;
};
FineFilm fine_film(int L);

// (M, G, Q, rows): the slots of a row, Q/2, fill its G threads evenly where
// the length allows it (Q = 2 G or a multiple), about 128 threads per CTA
#define MM_XLANE_SHAPES(X) \
    X(16, 2, 8, 64) X(18, 2, 9, 64) X(24, 4, 6, 32) X(27, 3, 9, 42) X(32, 4, 8, 32) X(36, 4, 9, 32) X(48, 4, 12, 32) X(54, 6, 9, 21) \
    X(64, 4, 16, 32) X(72, 6, 12, 21) X(81, 9, 9, 14) X(96, 8, 12, 16) X(108, 6, 18, 21) X(128, 8, 16, 16) X(144, 9, 16, 14) \
    X(162, 9, 18, 14) X(192, 8, 24, 16) X(216, 12, 18, 10) X(243, 9, 27, 14) X(256, 16, 16, 8) X(288, 12, 24, 10) X(324, 12, 27, 10) \
    X(384, 16, 24, 8) X(432, 16, 27, 8) X(486, 18, 27, 7) X(512, 16, 32, 8)

template <typename T> XLane<T> lane_x(int M);
// the third of the r2c kernels, in a translation unit of its own
void (*lane_r2c_any_f(int M))(XLaneArgs<float>);
void (*lane_r2c_any_d(int M))(XLaneArgs<double>);
template <> XLane<float> lane_x<float>(int M);
template <> XLane<double> lane_x<double>(int M);

}  // namespace mm
