// Inverse X pass and corrector of stacked Heun films (stacked_x.cuh).
#include "stacked_x.cuh"

namespace mm {

StackedX stacked_x_heun2(int M) {
    switch (M) {
#define MM_CASE(m, g, q) case m: return {stacked_x_kernel<m, g, q, 2, false>, g, XSplit<m, g, q>::LINE * sizeof(lcx<float>)};
        MM_STACKED_X_SHAPES(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
