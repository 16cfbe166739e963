// The last demag pass of stacked films (inverse X) inside their field kernel,
// as c2r_field_kernel of field_x.cuh does it for a single grid: the demag field
// goes from the row transforms to the cells through shared memory.  Rows are
// counted through all films of the class.  One GB300, five classes of the
// 1024-replica ensemble, mean of a class: predictor 41.0 us, corrector 36.3
// against 15.3 for the inverse X pass and 31.9 / 26.9 for the field kernel.
// What bounds it: 520 instructions a cell in the predictor, the thermal draw among
// them, 340 in the corrector, and their loads; half of the issue slots are taken at
// the 12 warps an SM that 128 registers allow.  Rows of four cells a thread only
// (16-byte accesses), films of up to 256 columns.
#pragma once

#include <cuda_runtime.h>

#include "field_x.cuh"
#include "stacked_cells.cuh"

namespace mm {

struct StackedX {
    void (*kern)(StackArgs, C2RSpec, int) = nullptr;
    int group = 0;          // threads per row and component
    size_t line = 0;        // bytes of an exchange line
};
StackedX stacked_x_heun1(int M);
StackedX stacked_x_heun2(int M);
StackedX stacked_x_dm1(int M);
StackedX stacked_x_dm2(int M);

// (M, G, Q): the shapes of field_x.cuh for films of up to 256 columns
#define MM_STACKED_X_SHAPES(X) \
    X(16, 2, 8) X(18, 2, 9) X(24, 4, 6) X(27, 3, 9) X(32, 4, 8) X(36, 4, 9) X(48, 4, 12) X(54, 6, 9) X(64, 4, 16) \
    X(72, 6, 12) X(81, 9, 9) X(96, 8, 12) X(108, 6, 18) X(128, 8, 16) X(144, 9, 16) X(162, 9, 18) X(192, 8, 24) \
    X(216, 12, 18) X(243, 9, 27) X(256, 8, 32)

template <int M, int G, int Q, int STAGE, bool DM>
__global__ void __launch_bounds__(kC2RThreads, 3) stacked_x_kernel(StackArgs a, C2RSpec s, int nrows) {
    using S = XSplit<M, G, Q>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (!a.st->active) return;
    float* sH = reinterpret_cast<float*>(smem_raw);   // [rpc][3][nx], once the lines are in registers
    const int nx = a.nx, ny = a.ny, rpc = s.rpc, row0 = blockIdx.x * rpc;
    if ((int)threadIdx.x < field_x_fft(G, rpc)) {
        const int task = threadIdx.x / G, rl = task / 3, comp = task - 3 * rl, row = row0 + rl;
        const bool valid = rl < rpc && row < nrows;
        const int q = valid ? row / ny : 0, y = valid ? row - q * ny : 0;
        const float2* X = s.spec + ((long long)(q * 3 + comp) * s.PyA + y) * s.Wk;
        lcx<float>* line = reinterpret_cast<lcx<float>*>(smem_raw) + task * S::LINE;
        float* dst = sH + (rl * 3 + comp) * nx;
        lane_c2r_row<float, M, G, Q>(X, s.tw, line, threadIdx.x % G, valid, [] { __syncthreads(); }, [&](int n, float2 v) {
            if (valid && 2 * n < nx) *reinterpret_cast<float2*>(dst + 2 * n) = v;
        });
    } else {
        if (!S::WARP) __syncthreads();                // (the rows' own exchange)
        __syncthreads();
    }
    __syncthreads();
    const int tpr = nx / 4;
    for (int c = threadIdx.x; c < rpc * tpr; c += blockDim.x) {
        const int rl = c / tpr, x = 4 * (c - rl * tpr), row = row0 + rl;
        if (row < nrows) {
            const int q = row / ny;
            stacked_lean_cells<4, STAGE, DM, true>(a, q, x, row - q * ny, sH + rl * 3 * nx + x);
        }
    }
}

}  // namespace mm
