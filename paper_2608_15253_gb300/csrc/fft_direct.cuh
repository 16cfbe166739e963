// FFT building blocks that keep data in registers between global memory and
// the transform, used by the FP32 demag passes of 3-D grids:
//  * reg_dif / reg_dit: a whole power-of-two line in one thread's registers.
//    The forward transform (decimation in frequency) leaves the spectrum in
//    bit-reversed order and the inverse (decimation in time) takes it back
//    in that order, so a pointwise product between them needs no reordering.
#pragma once

#include "common.cuh"
#include "fft_ct.cuh"

namespace mm {

__host__ __device__ constexpr int ilog2_c(int n) {
    int b = 0;
    while ((1 << b) < n) ++b;
    return b;
}
__host__ __device__ constexpr int bitrev_c(int i, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b)
        if ((i >> b) & 1) r |= 1 << (bits - 1 - b);
    return r;
}

// exp(-2 pi i q / 32), q < 32, in constant memory (filled by the demag
// setup of the including translation unit): with a compile-time index it is
// read as an instruction operand.
static __constant__ float2 c_tw32[32];

// Multiply by the twiddle tw[q] = exp(-2 pi i q / L) (DIR > 0) or its
// conjugate; q is a compile-time constant after unrolling, so the exact
// cases q = 0 and q = L/4 (a swap and a sign) cost no multiplication.
// tw == nullptr (FP32, L dividing 32): the constant table c_tw32.
template <typename T, int DIR, int L, int TS = 1>
__device__ __forceinline__ cplx<T> twiddle_mul(cplx<T> v, int q, const cplx<T>* tw) {
    if (q == 0) return v;
    if (4 * q == L) return mul_mi<T, DIR>(v);
    cplx<T> w;
    if constexpr (sizeof(T) == 4 && 32 % (L * TS) == 0) {
        if (tw == nullptr) {
            const float2 c = c_tw32[q * TS * (32 / (L * TS))];
            w = mkc<T>(c.x, c.y);
        } else {
            w = tw[q * TS];
        }
    } else {
        w = tw[q * TS];
    }
    return DIR > 0 ? cmul<T>(v, w) : cmulc<T>(v, w);
}

// In-register forward DFT of length L (a power of two), natural order in,
// bit-reversed order out.  tw[q] = exp(-2 pi i q / L).  One template level
// per stage so that every register index is a compile-time constant.
// HALF: the upper half of the input is known to be zero (a zero-padded
// line), which removes the first stage's additions.
// TS: stride of tw (the table may belong to a length TS * L).
template <typename T, int L, bool HALF = false, int TS = 1, int S = 0>
__device__ __forceinline__ void reg_dif(cplx<T> (&v)[L], const cplx<T>* tw) {
    if constexpr ((L >> S) >= 2) {
        constexpr int len = L >> S, h = len >> 1;
#pragma unroll
        for (int q = 0; q < L / 2; ++q) {
            const int b = (q / h) * len, j = q % h;
            const cplx<T> u = v[b + j];
            if (HALF && S == 0) {
                v[b + j + h] = twiddle_mul<T, 1, L, TS>(u, j * (L / len), tw);
            } else {
                const cplx<T> t = v[b + j + h];
                v[b + j] = cadd<T>(u, t);
                v[b + j + h] = twiddle_mul<T, 1, L, TS>(csub<T>(u, t), j * (L / len), tw);
            }
        }
        reg_dif<T, L, HALF, TS, S + 1>(v, tw);
    }
}

// In-register inverse DFT (unnormalised, exp(+2 pi i k n / L)), bit-reversed
// order in, natural order out.  HALF: only the lower half of the output is
// used (the last stage skips the upper half).
template <typename T, int L, bool HALF = false, int TS = 1, int S = 0>
__device__ __forceinline__ void reg_dit_inv(cplx<T> (&v)[L], const cplx<T>* tw) {
    if constexpr ((2 << S) <= L) {
        constexpr int len = 2 << S, h = len >> 1;
        constexpr bool last = (2 << S) == L;
#pragma unroll
        for (int q = 0; q < L / 2; ++q) {
            const int b = (q / h) * len, j = q % h;
            const cplx<T> u = v[b + j];
            const cplx<T> t = twiddle_mul<T, -1, L, TS>(v[b + j + h], j * (L / len), tw);
            v[b + j] = cadd<T>(u, t);
            if (!(HALF && last)) v[b + j + h] = csub<T>(u, t);
        }
        reg_dit_inv<T, L, HALF, TS, S + 1>(v, tw);
    }
}

}  // namespace mm
