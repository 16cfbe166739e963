// Inverse X pass fused with the field kernel (field_x.cuh), by half length:
// one material with the further local terms.
#include "field_x.cuh"

namespace mm {

FieldX field_x_ext(int M) {
    switch (M) {
#define MM_CASE(m, g, q) \
    case m: return {{c2r_field_kernel<m, g, q, FX_EXT, 2>, c2r_field_kernel<m, g, q, FX_EXT, 2>}, g, \
                    XSplit<m, g, q>::LINE * sizeof(lcx<float>)};
        MM_FIELD_X_SHAPES(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
