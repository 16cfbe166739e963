// Inverse X pass fused with the field kernel (field_x.cuh), by half length:
// one material with thermal field, spin torques and every stage update.  Two
// cells a thread: half the code, and instruction fetches bound these launches.
#include "field_x.cuh"

namespace mm {

FieldX field_x_full(int M) {
    switch (M) {
#define MM_CASE(m, g, q) \
    case m: return {{c2r_field_kernel<m, g, q, FX_FULL, 2>, c2r_field_kernel<m, g, q, FX_FULL, 2>}, g, \
                    XSplit<m, g, q>::LINE * sizeof(lcx<float>)};
        MM_FIELD_X_SHAPES(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
