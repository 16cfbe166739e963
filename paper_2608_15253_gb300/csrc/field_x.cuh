#pragma once

#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "ctx.h"
#include "field_cells.cuh"
#include "lane.h"
#include "lane_x.cuh"

namespace mm {

// The last demag pass (inverse X, half spectrum -> real rows) fused with
// the field kernel: the first 3 G rows_per_cta threads of a CTA run the C2R of
// the three components of its rows (z, y), G threads each (lane_x.cuh), into
// shared memory over the exchange buffers; then every thread forms the field,
// torque and stage output of V cells at a time with the demag field read from
// there -- H_demag never goes through global memory.
struct C2RSpec {
    const float2* spec;     // [3][nz][PyA][Wk]
    const float2* tw;       // exp(-2 pi i q / Px)
    int PyA, Wk;
    int rpc;                // rows per CTA
};

// At most 160 threads a CTA and 128 registers a thread: 15 warps per SM in
// CTAs of 96 or 160 threads (192 threads with 160 registers, 12 warps: 293
// against 256 us at 512x512x64; 96 registers spill).
constexpr int kC2RThreads = 160;

// What the cells of one material have: slopes only without thermal field, spin
// torque and further local terms (QUIET); all but the further local terms
// (FULL); everything (EXT).
enum FieldXKind { FX_QUIET, FX_FULL, FX_EXT };

struct FieldX {
    void (*kern[2])(FieldArgs<float>, C2RSpec) = {};   // two or four cells a thread (QUIET; else both two)
    int group = 0;                                     // threads per row and component
    size_t line = 0;                                   // bytes of an exchange line
};
FieldX field_x_quiet(int M);
FieldX field_x_full(int M);
FieldX field_x_ext(int M);

// (M, G, Q): those of the X passes but for 256, where eight threads a row give
// 26.3 us at 256x256x16 against 32.7 with sixteen
#define MM_FIELD_X_SHAPES(X) \
    X(16, 2, 8) X(18, 2, 9) X(24, 4, 6) X(27, 3, 9) X(32, 4, 8) X(36, 4, 9) X(48, 4, 12) X(54, 6, 9) X(64, 4, 16) \
    X(72, 6, 12) X(81, 9, 9) X(96, 8, 12) X(108, 6, 18) X(128, 8, 16) X(144, 9, 16) X(162, 9, 18) X(192, 8, 24) \
    X(216, 12, 18) X(243, 9, 27) X(256, 8, 32) X(288, 12, 24) X(324, 12, 27) X(384, 16, 24) X(432, 16, 27) \
    X(486, 18, 27) X(512, 16, 32)

// threads that transform rpc rows, in whole warps, and the shared memory: their
// exchange lines, and the field rows over them
constexpr int field_x_fft(int group, int rpc) { return (3 * rpc * group + 31) / 32 * 32; }
inline size_t field_x_smem(int group, size_t line, int nx, int rpc) {
    const size_t tasks = (field_x_fft(group, rpc) + group - 1) / group;
    return std::max(tasks * line, (size_t)3 * rpc * nx * sizeof(float));
}

// rows per CTA: as many as 96 threads transform at once (at least one), fewer on
// small grids so that four CTAs per SM run (8 RK45 steps of a 512x512 film: 1326
// us against 1359 with two, whose last wave left half of the SMs one CTA short)
inline int c2r_rows(int G, long long rows) {
    const long long want = (rows + 4 * sm_count() - 1) / (4 * sm_count());
    return (int)std::max(1LL, std::min<long long>(96 / (3 * G), want));
}

// The same for small FP64 grids (field_fine_d.cu).
struct FineSpec {
    const double2* spec;    // [3][nz][PyA][Wk]
    const double2* tw;      // exp(-2 pi i q / Px)
    int PyA, Wk;
    int parts;              // CTAs per row
};
struct FineField {
    void (*kern)(FieldArgs<double>, FineSpec) = nullptr;
    size_t line = 0;        // bytes of a component's line
};
FineField fine_field(int M);
constexpr int kFineFieldThreads = 224;   // three warps of transforms, up to four of cells
inline size_t fine_field_smem(const FineField& f, int nx, int parts) {
    return 3 * f.line + 3 * sizeof(double) * (nx + (nx + parts - 1) / parts);
}

template <int M, int G, int Q, int KIND, int V>
__global__ void __launch_bounds__(kC2RThreads, 3) c2r_field_kernel(FieldArgs<float> a, C2RSpec s) {
    using S = XSplit<M, G, Q>;
    constexpr bool QUIET = KIND == FX_QUIET;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dep_wait();
    if (a.gate && !a.st->active) return;
    float* sH = reinterpret_cast<float*>(smem_raw);   // [rpc][3][nx], once the lines are in registers
    const int nx = a.nx, rpc = s.rpc, nrows = a.ny * a.nz;
    const int row0 = blockIdx.x * rpc, tpr = nx / V, fft = field_x_fft(G, rpc);
    constexpr bool EXT = KIND == FX_EXT;
    VecIn<V> in;
    auto cells = [&](int c, int& rl, int& x0, int& y, int& z) {   // the c-th V cells; false past the grid
        rl = c / tpr;
        x0 = V * (c - rl * tpr);
        z = (row0 + rl) / a.ny;
        y = row0 + rl - z * a.ny;
        return row0 + rl < nrows;
    };
    int rl, x0, y, z;
    if ((int)threadIdx.x < fft) {
        const int task = threadIdx.x / G, comp = task % 3, row = row0 + task / 3;
        const bool valid = task / 3 < rpc && row < nrows;
        rl = task / 3;
        z = valid ? row / a.ny : 0;
        y = valid ? row - z * a.ny : 0;
        const float2* X = s.spec + ((long long)(comp * a.nz + z) * s.PyA + y) * s.Wk;
        lcx<float>* line = reinterpret_cast<lcx<float>*>(smem_raw) + task * S::LINE;
        float* dst = sH + (rl * 3 + comp) * nx;
        lane_c2r_row<float, M, G, Q>(X, s.tw, line, threadIdx.x % G, valid, [] { __syncthreads(); }, [&](int n, float2 v) {
            if (valid && 2 * n < nx) *reinterpret_cast<float2*>(dst + 2 * n) = v;
        });
    } else {
        // threads without a row: their first cells meanwhile
        if (!QUIET && (int)threadIdx.x < rpc * tpr && cells(threadIdx.x, rl, x0, y, z))
            field_vec_load<V, EXT, QUIET>(a, x0, y, z, in);
        if (!S::WARP) __syncthreads();                // (the rows' own exchange)
        __syncthreads();
    }
    __syncthreads();
    for (int c = threadIdx.x; c < rpc * tpr; c += blockDim.x)
        if (cells(c, rl, x0, y, z)) {
            if (QUIET || c != (int)threadIdx.x || (int)threadIdx.x < fft) field_vec_load<V, EXT, QUIET>(a, x0, y, z, in);
            field_vec_finish<V, EXT, true, QUIET>(a, x0, y, z, in, sH + rl * 3 * nx + x0, nx);
        }
}

}  // namespace mm
