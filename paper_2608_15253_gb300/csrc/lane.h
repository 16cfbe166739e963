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

template <typename T> LaneKern<T> lane_conv3(int L);            // middle pass of a 3-D grid
template <typename T> LaneKern<T> lane_film(int L);             // middle pass of one film
template <typename T> LaneKern<T> lane_films(int L);            // middle pass of many films
template <typename T> LaneKern<T> lane_col(int L, bool forward);    // Y passes of a 3-D grid

template <> LaneKern<float> lane_conv3<float>(int L);
template <> LaneKern<double> lane_conv3<double>(int L);
template <> LaneKern<float> lane_film<float>(int L);
template <> LaneKern<double> lane_film<double>(int L);
template <> LaneKern<float> lane_films<float>(int L);
template <> LaneKern<double> lane_films<double>(int L);
template <> LaneKern<float> lane_col<float>(int L, bool forward);
template <> LaneKern<double> lane_col<double>(int L, bool forward);

}  // namespace mm
