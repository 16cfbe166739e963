// Column passes of the demag convolution (Methods, "Physics and
// discretization": the zero-padded FFT convolution with the Newell tensor)
// on register FFTs over lanes (fft_lane.cuh).  A line of length L = G * Q is
// split over G threads of Q values, the four-step factorisation
//
//   X[k1 + Q k2] = sum_t W_G^(t k2) [ W_L^(t k1) sum_q x[q G + t] W_Q^(q k1) ]
//
// Columns are flattened (other-axis index, kx) positions, TP lanes of them
// (one column each, or two packed ones in FP32) per CTA.  Kernels: the middle pass of 3-D grids
// and of ensembles of films (lane_conv_kernel), the middle pass of single
// films (lane_film_kernel), and the Y passes of 3-D grids
// (lane_col_kernel).  Each kernel's comment gives its split.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "ctx.h"
#include "fft_lane.cuh"

namespace mm {

template <typename T>
struct LaneArgs {
    cplx<T>* base;            // spectrum
    long long comp_stride;    // between the three components
    long long line_stride;    // between consecutive points of a line
    long long o_stride;       // between consecutive other-axis indices
    int Wk, Kx;               // columns per other-axis index (row pitch), valid ones
    int n_o;                  // 3-D: Py (other-axis length); 2-D: number of film planes
    int n_cols;               // flattened columns (of side 0 in 3-D)
    int n_in, n_out;          // points per line read / written
    const T* khat;            // [ncomp][L/2+1][n_o/2+1 (3-D) or 1][Wk]
    long long kc, kk, ko;     // tensor strides: component, line frequency, other-axis frequency
    const cplx<T>* tw;        // exp(-2 pi i q / L)
};

// Exchange buffer: value (c, u, k1) of lane p at ((c G + u) US + k1 TP + p).
// US pads the G rows so that threads of neighbouring t write to different
// banks when the TP lanes of one row are narrower than 128 bytes.
template <typename N, int Q, int TP>
constexpr int lane_us() {
    const int sz = 2 * (int)sizeof(N), row = TP * sz;
    int us = Q * TP;
    if (row < 128)
        while ((us * sz) % 128 != row) ++us;
    return us;                                                    // a multiple of 16 bytes: TP sz is one
}

template <int SZ>
__device__ __forceinline__ void lane_async(void* smem, const void* gmem, bool in) {   // !in: zeros
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (SZ == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(in ? 16 : 0) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(in ? 8 : 0) : "memory");
}
__device__ __forceinline__ void lane_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int K>
__device__ __forceinline__ void lane_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(K) : "memory"); }

// exp(-2 pi i q / L) for runtime exponents, repeated over the lanes: (c, s)
template <typename N, int L, int NT>
__device__ __forceinline__ void lane_twiddles(lcx<N>* stw, const cplx<typename lane<N>::real>* tw) {
    for (int q = threadIdx.x; q < L; q += NT) {
        const cplx<typename lane<N>::real> w = __ldg(tw + q);
        stw[q] = {lane<N>::all(w.x), lane<N>::all(-w.y)};
    }
}
template <int DIR, typename N>
__device__ __forceinline__ lcx<N> lctws(lcx<N> v, lcx<N> w) {
    return lctw<DIR, N>(v, w.re, w.im, lmul(w.im, lane<N>::all(-1.0)));
}

// The CTA's tensor tile [NC][L/2+1][TP lanes] by cp.async: pieces of 16 bytes
// stay within one tensor row (the pitch Wk is a multiple of four columns).
template <typename N, int NC, int KZ, int TP, int NT, bool D3, typename T>
__device__ __forceinline__ void lane_tile(N* sk, const LaneArgs<T>& a, int pblk) {
    constexpr int CP = 16 / (int)sizeof(T);                       // columns per piece
    constexpr int NG = TP * (int)sizeof(N) / 16;                  // pieces per tile row
    static_assert(NG >= 1 && (TP * sizeof(N)) % 16 == 0, "tile rows of whole pieces");
    int o = 0, kx = 0;
    for (int e = threadIdx.x; e < NC * KZ * NG; e += NT) {
        const int grp = e % NG, row = e / NG, j = row / KZ, k = row - j * KZ;
        if (NT % NG != 0 || e == (int)threadIdx.x) {              // a thread keeps its group
            int p = pblk + CP * grp;
            if (p >= a.n_cols) p = 0;                             // past the end: any valid row
            o = p / a.Wk;
            kx = p - o * a.Wk;
        }
        const T* src = a.khat + j * a.kc + (long long)k * a.kk + (D3 ? (long long)o * a.ko : 0) + kx;
        lane_async<16>(reinterpret_cast<char*>(sk + (size_t)row * TP) + 16 * grp, src, true);
    }
}

// Tensor value at line frequency k1 + Q k2 (k1 < Q): the fold into the
// stored half range is a compile-time constant but on the one k2 where it
// depends on k1.
template <int L, int Q>
__device__ __forceinline__ bool lane_fold(int k1, int k2) {
    const int lo = 2 * Q * k2;                                    // 2 kz - 2 k1
    return lo > L ? true : (lo + 2 * (Q - 1) <= L ? false : 2 * k1 + lo > L);
}

// ---------------------------------------------------------------------------
// Middle pass, many columns: CS groups of G threads per lane.  Phase 1 (CS =
// 3: one component each): Q strided inputs from global memory, Q-point FFT,
// twiddle, one store to shared memory.  Phase 2: the item (k1, lane) takes
// the G values of the components that the tensor couples (3-D: all three;
// films: x and y together, z by itself), G-point DFT, H^ = K^ M^, inverse,
// back in place -- its slots belong to it alone.  Phase 3: phase 1 backwards,
// the un-padded outputs only.
//
// Persistent CTAs.  A thread brings its own next inputs by cp.async into
// slots that it alone reads, as soon as it has taken the present ones, so
// global memory works through all three phases; the tensor tile of the next
// columns follows when phase 2 is done with the present one.  In 3-D a CTA
// takes columns at ky, then those at Py - ky: both read the same stored
// tensor rows, which cross the bus once.  The parity sign of the second is
// diag(1, -1, 1) on both sides of the tensor: the y component changes sign
// on the way in and out.
// ---------------------------------------------------------------------------
// entries of the twiddle table: what follows it starts on a 16-byte boundary
template <int L> constexpr int lane_lt() { return (L + 1) / 2 * 2; }
template <int L> constexpr int lane_qin(int G) { return ((L + 1) / 2 + G - 1) / G; }   // 2 n_in - 1 <= L

template <typename N, int L, int G, int Q, int TP, int NC, bool ST>
constexpr size_t lane_conv_smem() {
    return (size_t)(3 * G * lane_us<N, Q, TP>() + (ST ? lane_lt<L>() + 3 * G * TP * lane_qin<L>(G) : 0)) * 2 * sizeof(N) +
           (size_t)NC * (L / 2 + 1) * TP * sizeof(N);
}

template <typename N, int L, int G, int Q, int TP, int CS, bool D3, int MINB, bool ST>
__global__ void __launch_bounds__(CS * G * TP, MINB) lane_conv_kernel(LaneArgs<typename lane<N>::real> a) {
    using T = typename lane<N>::real;
    static_assert(L == G * Q && (CS == 1 || CS == 3), "line split");
    constexpr int W = lane<N>::width, NT = CS * G * TP, NC = D3 ? 6 : 4, KZ = L / 2 + 1, SIDES = D3 ? 2 : 1;
    constexpr int QIN = lane_qin<L>(G);                           // slots that can hold inputs
    constexpr int US = lane_us<N, Q, TP>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lcx<N>* sm = reinterpret_cast<lcx<N>*>(smem_raw);
    lcx<N>* stw = sm + 3 * G * US;
    lcx<N>* sin = stw + lane_lt<L>() + threadIdx.x;               // this thread's input slots, NT apart
    N* sk = reinterpret_cast<N*>(stw + (ST ? lane_lt<L>() + 3 * G * TP * QIN : 0));
    if (ST) lane_twiddles<N, L, NT>(stw, a.tw);
    const int pr = threadIdx.x % TP, t = (threadIdx.x / TP) % G, c0 = CS == 3 ? threadIdx.x / (G * TP) : 0;
    const int ntile = (a.n_cols + TP * W - 1) / (TP * W);

    // column of this thread in tile w, side s; false if there is none
    auto column = [&](int w, int s, long long& off) {
        const int p = w * (TP * W) + pr * W;
        int o = p / a.Wk;
        const int kx = p - o * a.Wk;
        bool ok = w < ntile && p < a.n_cols && kx < a.Kx;
        if (D3 && s) {
            ok = ok && o != 0 && 2 * o != a.n_o;
            o = a.n_o - o;
        }
        off = ok ? (long long)o * a.o_stride + kx : 0;
        return ok;
    };
    auto fetch = [&](int w, int s) {
        long long off;
        const bool ok = column(w, s, off);
#pragma unroll
        for (int cc = 0; cc < 3 / CS; ++cc) {
            const cplx<T>* g = a.base + off + (c0 + cc) * a.comp_stride;
#pragma unroll
            for (int q = 0; q < QIN; ++q) {
                const int n = q * G + t;
                const bool in = ok && n < a.n_in;
                lane_async<2 * sizeof(N)>(sin + (cc * QIN + q) * NT, in ? g + n * a.line_stride : a.base, in);
            }
        }
        lane_commit();
    };
    int w = ST || !D3 ? blockIdx.x : blockIdx.x >> 1;             // !ST: one side of one tile per CTA
    if (ST) dep_wait();
    if (w >= ntile) return;
    if (ST) fetch(w, 0);
    lane_tile<N, NC, KZ, TP, NT, D3>(sk, a, w * (TP * W));        // (the tensor is older than any launch)
    lane_commit();
    if (!ST) dep_wait();
    for (; w < ntile; w += gridDim.x) {
#pragma unroll 1
        for (int s = !ST && D3 ? blockIdx.x & 1 : 0; s < SIDES; ++s) {
            // own inputs: the only later group is the tensor tile fetched with this tile's first side
            if (ST && s == 0) lane_wait<1>();
            else if (ST) lane_wait<0>();
            if (ST) __syncthreads();                              // the exchange buffer is free (and the twiddles stand)
            const N flip = lane<N>::all(D3 && s ? -1.0 : 1.0);
            long long off;
            const bool valid = column(w, s, off);
#pragma unroll
            for (int cc = 0; cc < 3 / CS; ++cc) {
                const int c = c0 + cc;
                lcx<N> v[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const int n = q * G + t;
                    if constexpr (ST) v[q] = q < QIN ? lmem<N>::load(reinterpret_cast<const cplx<T>*>(sin + (cc * QIN + q) * NT)) : lzero<N>();
                    else v[q] = q < QIN && valid && n < a.n_in ? lmem<N>::load(a.base + off + c * a.comp_stride + n * a.line_stride) : lzero<N>();
                }
                if (ST && cc == 3 / CS - 1) {
                    if (s + 1 < SIDES) fetch(w, s + 1);
                    else fetch(w + gridDim.x, 0);
                }
                if (D3 && c == 1) {
#pragma unroll
                    for (int q = 0; q < QIN; ++q) v[q] = {lmul(v[q].re, flip), lmul(v[q].im, flip)};
                }
                lfft<1, Q, N, QIN>(v);
#pragma unroll
                for (int k1 = 0; k1 < Q; ++k1) {
                    lcx<N> r = v[k1];
                    if (G > 1 && k1 > 0) r = ST ? lctws<1>(r, stw[t * k1]) : lctwr<1>(r, ltw_load<N>(a.tw, t * k1));
                    sm[(c * G + t) * US + k1 * TP + pr] = r;
                }
            }
            if (!ST || s == 0) lane_wait<ST ? 1 : 0>();                  // the tensor tile; the next inputs may be on their way
            __syncthreads();

            if constexpr (D3) {
#pragma unroll 1
                for (int it = threadIdx.x; it < Q * TP; it += NT) {
                    const int k1 = it / TP, pp = it % TP;
                    lcx<N> m[3][G];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
#pragma unroll
                        for (int u = 0; u < G; ++u) m[c][u] = sm[(c * G + u) * US + it];
                        lfft<1, G, N>(m[c]);
                    }
#pragma unroll
                    for (int k2 = 0; k2 < G; ++k2) {
                        const bool fold = lane_fold<L, Q>(k1, k2);
                        const int kz = k1 + Q * k2;
                        const N* K = sk + (fold ? L - kz : kz) * TP + pp;
                        const N kxx = K[0], kyy = K[KZ * TP], kzz = K[2 * KZ * TP], kxy = K[3 * KZ * TP];
                        N kxz = K[4 * KZ * TP], kyz = K[5 * KZ * TP];
                        if (!(2 * Q * k2 + 2 * (Q - 1) <= L)) {   // xz and yz are odd in kz
                            const N st = lane<N>::all(fold ? -1.0 : 1.0);
                            kxz = lmul(kxz, st);
                            kyz = lmul(kyz, st);
                        }
                        const lcx<N> x = m[0][k2], y = m[1][k2], z = m[2][k2];
                        m[0][k2] = {lfma(kxz, z.re, lfma(kxy, y.re, lmul(kxx, x.re))), lfma(kxz, z.im, lfma(kxy, y.im, lmul(kxx, x.im)))};
                        m[1][k2] = {lfma(kyz, z.re, lfma(kyy, y.re, lmul(kxy, x.re))), lfma(kyz, z.im, lfma(kyy, y.im, lmul(kxy, x.im)))};
                        m[2][k2] = {lfma(kzz, z.re, lfma(kyz, y.re, lmul(kxz, x.re))), lfma(kzz, z.im, lfma(kyz, y.im, lmul(kxz, x.im)))};
                    }
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        lfft<-1, G, N>(m[c]);
#pragma unroll
                        for (int u = 0; u < G; ++u) sm[(c * G + u) * US + it] = m[c][u];
                    }
                }
            } else {
#pragma unroll 1
                for (int i2 = threadIdx.x; i2 < 2 * Q * TP; i2 += NT) {
                    const bool zc = i2 >= Q * TP;
                    const int it = zc ? i2 - Q * TP : i2;
                    const int k1 = it / TP, pp = it % TP;
                    if (zc) {
                        lcx<N> m[G];
#pragma unroll
                        for (int u = 0; u < G; ++u) m[u] = sm[(2 * G + u) * US + it];
                        lfft<1, G, N>(m);
#pragma unroll
                        for (int k2 = 0; k2 < G; ++k2) {
                            const int kz = k1 + Q * k2;
                            const N kzz = sk[(2 * KZ + (lane_fold<L, Q>(k1, k2) ? L - kz : kz)) * TP + pp];
                            m[k2] = {lmul(kzz, m[k2].re), lmul(kzz, m[k2].im)};
                        }
                        lfft<-1, G, N>(m);
#pragma unroll
                        for (int u = 0; u < G; ++u) sm[(2 * G + u) * US + it] = m[u];
                    } else {
                        lcx<N> m[2][G];
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
#pragma unroll
                            for (int u = 0; u < G; ++u) m[c][u] = sm[(c * G + u) * US + it];
                            lfft<1, G, N>(m[c]);
                        }
#pragma unroll
                        for (int k2 = 0; k2 < G; ++k2) {
                            const bool fold = lane_fold<L, Q>(k1, k2);
                            const int kz = k1 + Q * k2;
                            const N* K = sk + (fold ? L - kz : kz) * TP + pp;
                            const N kxx = K[0], kyy = K[KZ * TP];
                            N kxy = K[3 * KZ * TP];
                            if (!(2 * Q * k2 + 2 * (Q - 1) <= L)) kxy = lmul(kxy, lane<N>::all(fold ? -1.0 : 1.0));
                            const lcx<N> x = m[0][k2], y = m[1][k2];
                            m[0][k2] = {lfma(kxy, y.re, lmul(kxx, x.re)), lfma(kxy, y.im, lmul(kxx, x.im))};
                            m[1][k2] = {lfma(kyy, y.re, lmul(kxy, x.re)), lfma(kyy, y.im, lmul(kxy, x.im))};
                        }
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            lfft<-1, G, N>(m[c]);
#pragma unroll
                            for (int u = 0; u < G; ++u) sm[(c * G + u) * US + it] = m[c][u];
                        }
                    }
                }
            }
            __syncthreads();
            if (ST && s == SIDES - 1) {
                if (w + (int)gridDim.x < ntile) lane_tile<N, NC, KZ, TP, NT, D3>(sk, a, (w + gridDim.x) * (TP * W));
                lane_commit();
            }

#pragma unroll
            for (int cc = 0; cc < 3 / CS; ++cc) {
                const int c = c0 + cc;
                lcx<N> v[Q];
#pragma unroll
                for (int k1 = 0; k1 < Q; ++k1) {
                    lcx<N> r = sm[(c * G + t) * US + k1 * TP + pr];
                    if (G > 1 && k1 > 0) r = ST ? lctws<-1>(r, stw[t * k1]) : lctwr<-1>(r, ltw_load<N>(a.tw, t * k1));
                    v[k1] = r;
                }
                lfft<-1, Q, N>(v);
                if (valid) {
                    cplx<T>* g = a.base + off + c * a.comp_stride;
#pragma unroll
                    for (int q = 0; q < QIN; ++q) {
                        const int n = q * G + t;
                        if (D3 && c == 1) v[q] = {lmul(v[q].re, flip), lmul(v[q].im, flip)};
                        if (n < a.n_out) lmem<N>::store(g + n * a.line_stride, v[q]);
                    }
                }
            }
            if (!ST) return;
        }
    }
    lane_wait<0>();
}

// ---------------------------------------------------------------------------
// Middle pass of one film: a few hundred columns, so the time is the latency
// of one CTA.  Three groups of G threads per lane, one component each in
// every phase; the spectra meet in shared memory: phase 2 stores the G-point
// DFT in place, then every item forms its own row of K^ M^ from the other
// component's values before the inverse.
// ---------------------------------------------------------------------------
template <typename N, int L, int G, int Q, int TP>
constexpr size_t lane_film_smem() {
    return (size_t)3 * G * lane_us<N, Q, TP>() * 2 * sizeof(N) + (size_t)4 * (L / 2 + 1) * TP * sizeof(N);
}

template <typename N, int L, int G, int Q, int TP>
__global__ void __launch_bounds__(3 * G * TP) lane_film_kernel(LaneArgs<typename lane<N>::real> a) {
    using T = typename lane<N>::real;
    static_assert(L == G * Q, "line split");
    constexpr int W = lane<N>::width, NT = 3 * G * TP, KZ = L / 2 + 1;
    constexpr int QIN = ((L + 1) / 2 + G - 1) / G;
    constexpr int US = lane_us<N, Q, TP>();
    constexpr int NI = (Q + G - 1) / G;                           // phase-2 items per thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lcx<N>* sm = reinterpret_cast<lcx<N>*>(smem_raw);
    N* sk = reinterpret_cast<N*>(sm + 3 * G * US);
    const int pblk = blockIdx.x * (TP * W);
    lane_tile<N, 4, KZ, TP, NT, false>(sk, a, pblk);              // (the tensor is older than any launch)
    lane_commit();
    dep_wait();
    const int pr = threadIdx.x % TP, t = (threadIdx.x / TP) % G, c = threadIdx.x / (G * TP);
    const int p = pblk + pr * W;
    const int o = p / a.Wk, kx = p - o * a.Wk;
    const bool valid = p < a.n_cols && kx < a.Kx;
    cplx<T>* g = a.base + (valid ? (long long)o * a.o_stride + kx : 0) + c * a.comp_stride;
    {
        lcx<N> v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int n = q * G + t;
            v[q] = (q < QIN && valid && n < a.n_in) ? lmem<N>::load(g + n * a.line_stride) : lzero<N>();
        }
        lfft<1, Q, N, QIN>(v);
#pragma unroll
        for (int k1 = 0; k1 < Q; ++k1) {
            lcx<N> r = v[k1];
            if (G > 1 && k1 > 0) r = lctwr<1>(r, ltw_load<N>(a.tw, t * k1));
            sm[(c * G + t) * US + k1 * TP + pr] = r;
        }
    }
    lane_wait<0>();
    __syncthreads();
    lcx<N> m[NI][G];
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int k1 = t + i * G, it = k1 * TP + pr;
        if (Q % G == 0 || k1 < Q) {
#pragma unroll
            for (int u = 0; u < G; ++u) m[i][u] = sm[(c * G + u) * US + it];
            lfft<1, G, N>(m[i]);
            if (c < 2) {
#pragma unroll
                for (int u = 0; u < G; ++u) sm[(c * G + u) * US + it] = m[i][u];
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int k1 = t + i * G, it = k1 * TP + pr;
        if (Q % G == 0 || k1 < Q) {
#pragma unroll
            for (int k2 = 0; k2 < G; ++k2) {
                const bool fold = lane_fold<L, Q>(k1, k2);
                const int kz = k1 + Q * k2;
                const N* K = sk + (fold ? L - kz : kz) * TP + pr;
                const N kd = K[c * KZ * TP];
                lcx<N> h = {lmul(kd, m[i][k2].re), lmul(kd, m[i][k2].im)};
                if (c < 2) {
                    N kxy = K[3 * KZ * TP];
                    if (!(2 * Q * k2 + 2 * (Q - 1) <= L)) kxy = lmul(kxy, lane<N>::all(fold ? -1.0 : 1.0));
                    const lcx<N> y = sm[((1 - c) * G + k2) * US + it];
                    h = {lfma(kxy, y.re, h.re), lfma(kxy, y.im, h.im)};
                }
                m[i][k2] = h;
            }
            lfft<-1, G, N>(m[i]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int k1 = t + i * G, it = k1 * TP + pr;
        if (Q % G == 0 || k1 < Q) {
#pragma unroll
            for (int u = 0; u < G; ++u) sm[(c * G + u) * US + it] = m[i][u];
        }
    }
    __syncthreads();
    lcx<N> v[Q];
#pragma unroll
    for (int k1 = 0; k1 < Q; ++k1) {
        lcx<N> r = sm[(c * G + t) * US + k1 * TP + pr];
        if (G > 1 && k1 > 0) r = lctwr<-1>(r, ltw_load<N>(a.tw, t * k1));
        v[k1] = r;
    }
    lfft<-1, Q, N>(v);
    if (valid) {
#pragma unroll
        for (int q = 0; q < QIN; ++q) {
            const int n = q * G + t;
            if (n < a.n_out) lmem<N>::store(g + n * a.line_stride, v[q]);
        }
    }
}

// ---------------------------------------------------------------------------
// Y passes of 3-D grids (forward: ny inputs -> Py outputs; inverse: Py
// inputs -> ny outputs), G threads per lane and one shared-memory exchange.
// Columns are the flattened (component, z, kx) list with its pad columns.
//  forward  thread t: Q-point FFTs of x[q G + t] (zero past n_in), twiddle
//           W_L^(t k1), exchange; item k1: G-point DFT -> X[k1 + Q k2].
//  inverse  item k1: inverse G-point DFT of H[k1 + Q k2], twiddle, exchange;
//           thread t: inverse Q-point FFT -> y[q G + t].
// In place: a column belongs to one CTA, which has read it when it writes.
// ---------------------------------------------------------------------------
template <typename N, int L, int G, int Q, int TP>
constexpr size_t lane_col_smem() { return (size_t)G * lane_us<N, Q, TP>() * 2 * sizeof(N); }

template <typename N, int L, int G, int Q, int TP, int DIR, int MINB>
__global__ void __launch_bounds__(G * TP, MINB) lane_col_kernel(LaneArgs<typename lane<N>::real> a) {
    using T = typename lane<N>::real;
    static_assert(L == G * Q, "line split");
    constexpr int W = lane<N>::width, QIN = lane_qin<L>(G), US = lane_us<N, Q, TP>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lcx<N>* sm = reinterpret_cast<lcx<N>*>(smem_raw);
    const int pr = threadIdx.x % TP, t = threadIdx.x / TP;
    const int p = blockIdx.x * (TP * W) + pr * W;
    const int o = p / a.Wk, kx = p - o * a.Wk;
    const bool valid = p < a.n_cols && kx < a.Kx;
    cplx<T>* g = a.base + (valid ? (long long)o * a.o_stride + kx : 0);
    const long long ls = a.line_stride;
    dep_wait();
    if constexpr (DIR > 0) {
        lcx<N> v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int n = q * G + t;
            v[q] = q < QIN && valid && n < a.n_in ? lmem<N>::load(g + n * ls) : lzero<N>();
        }
        lfft<1, Q, N, QIN>(v);
#pragma unroll
        for (int k1 = 0; k1 < Q; ++k1) {
            lcx<N> r = v[k1];
            if (G > 1 && k1 > 0) r = lctwr<1>(r, ltw_load<N>(a.tw, t * k1));
            sm[t * US + k1 * TP + pr] = r;
        }
        __syncthreads();
#pragma unroll 1
        for (int k1 = t; k1 < Q; k1 += G) {
            lcx<N> m[G];
#pragma unroll
            for (int u = 0; u < G; ++u) m[u] = sm[u * US + k1 * TP + pr];
            lfft<1, G, N>(m);
            if (valid) {
#pragma unroll
                for (int k2 = 0; k2 < G; ++k2) lmem<N>::store(g + (k1 + Q * k2) * ls, m[k2]);
            }
        }
    } else {
#pragma unroll 1
        for (int k1 = t; k1 < Q; k1 += G) {
            lcx<N> m[G];
#pragma unroll
            for (int k2 = 0; k2 < G; ++k2) m[k2] = valid ? lmem<N>::load(g + (k1 + Q * k2) * ls) : lzero<N>();
            lfft<-1, G, N>(m);
#pragma unroll
            for (int u = 0; u < G; ++u) {
                lcx<N> r = m[u];
                if (G > 1 && u > 0) r = lctwr<-1>(r, ltw_load<N>(a.tw, u * k1));
                sm[u * US + k1 * TP + pr] = r;
            }
        }
        __syncthreads();
        lcx<N> v[Q];
#pragma unroll
        for (int k1 = 0; k1 < Q; ++k1) v[k1] = sm[t * US + k1 * TP + pr];
        lfft<-1, Q, N>(v);
        if (valid) {
#pragma unroll
            for (int q = 0; q < QIN; ++q) {
                const int n = q * G + t;
                if (n < a.n_out) lmem<N>::store(g + n * ls, v[q]);
            }
        }
    }
}

}  // namespace mm
