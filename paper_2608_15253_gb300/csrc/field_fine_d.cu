// Inverse X pass fused with the slopes of small FP64 grids of one material (no
// thermal field, no spin torque, no further local terms): a row per CTA,
// three warps transform its components in the passes of fine_c2r_kernel while
// further warps form the local fields of its cells; the slopes follow when both
// are there.
//
// An FP64 instruction of a warp holds its scheduler for 64 clocks, and a few
// dozen rows leave most of the chip idle: so `parts` CTAs share a row, each
// repeats the three transforms (130 instructions a warp at M = 128, on idle
// schedulers) and owns a part of the cells, 32 of 128 on the fourth scheduler.
// 128x32: 12.4 us against 10.0 + 10.5 for the two kernels.
#include "field_cells.cuh"
#include "field_x.cuh"
#include "lane_x.cuh"

namespace mm {

template <int M>
__global__ void __launch_bounds__(kFineFieldThreads) fine_field_kernel(FieldArgs<double> a, FineSpec s) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dep_wait();
    if (a.gate && !a.st->active) return;
    const int nx = a.nx, row = blockIdx.x / s.parts, part = blockIdx.x % s.parts, z = row / a.ny, y = row - z * a.ny;
    const int per = (nx + s.parts - 1) / s.parts, x0 = part * per, x1 = min(nx, x0 + per);
    double* hd = reinterpret_cast<double*>(smem_raw) + 3 * 2 * fine_line(M);   // [3][nx]
    double* hl = hd + 3 * nx;                                                  // [3][per]
    const int c = threadIdx.x >> 5, cells = blockDim.x - 96;
    const long long N = a.N, i0 = (long long)row * nx;
    if (c < 3) {
        lcx<double>* sm = reinterpret_cast<lcx<double>*>(smem_raw) + c * fine_line(M);
        fine_c2r_row<double, M>(s.spec + ((long long)(c * a.nz + z) * s.PyA + y) * s.Wk, s.tw, sm, [&](int n, lcx<double> v) {
            if (2 * n < nx) hd[c * nx + 2 * n] = v.re;
            if (2 * n + 1 < nx) hd[c * nx + 2 * n + 1] = v.im;
        });
    } else {
        for (int x = x0 + (int)threadIdx.x - 96; x < x1; x += cells) {
            v3<double> H, k;
            cell_field<double, true, false, true>(a, x, y, z, i0 + x, 0, a.R0, ld3(a.m, N, i0 + x), nullptr, 0, H, k, false);
            hl[x - x0] = H.x;
            hl[per + x - x0] = H.y;
            hl[2 * per + x - x0] = H.z;
        }
    }
    __syncthreads();
    if (c < 3) return;
    double* o = a.out;
    if (!o) {
        const int kf = a.st->k_first;
        o = a.kptr[a.kstage == 0 ? kf : 6 - kf];
    }
    for (int x = x0 + (int)threadIdx.x - 96; x < x1; x += cells) {   // the cells this thread began
        const v3<double> H = mk3<double>(hl[x - x0] + hd[x], hl[per + x - x0] + hd[nx + x], hl[2 * per + x - x0] + hd[2 * nx + x]);
        st3(o, N, i0 + x, llg_slope(ld3(a.m, N, i0 + x), H, a.R0));
    }
}

FineField fine_field(int M) {
    switch (M) {
#define MM_CASE(m, g, q, rows) case m: return {fine_field_kernel<m>, fine_line(m) * sizeof(lcx<double>)};
        MM_XLANE_SHAPES(MM_CASE)
#undef MM_CASE
        default: return {};
    }
}

}  // namespace mm
