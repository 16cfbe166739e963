// Forward X pass of FP32 rows of any kind (lane_x.cuh, X_ANY), by half length.
#include "lane.h"
#include "lane_x.cuh"

namespace mm {

void (*lane_r2c_any_f(int M))(XLaneArgs<float>) {
    switch (M) {
#define MM_CASE(m, g, q, rows) case m: return lane_r2c_kernel<float, m, g, q, rows, X_ANY>;
        MM_XLANE_SHAPES(MM_CASE)
        MM_XLANE_LONG(MM_CASE)
#undef MM_CASE
        default: return nullptr;
    }
}

}  // namespace mm
