// Inverse X pass fused with the field kernel (field_x.cuh), by half length:
// one material, slopes only.  Four cells a thread where the row allows it: 16-byte
// accesses (512x512x64 256 us; with two, 355 against 293 before the CTAs were made
// smaller).
#include "field_x.cuh"

namespace mm {

FieldX field_x_quiet(int M) {
    switch (M) {
#define MM_CASE(m, g, q) \
    case m: return {{c2r_field_kernel<m, g, q, FX_QUIET, 2>, c2r_field_kernel<m, g, q, FX_QUIET, 4>}, g, \
                    XSplit<m, g, q>::LINE * sizeof(lcx<float>)};
        MM_FIELD_X_SHAPES(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
