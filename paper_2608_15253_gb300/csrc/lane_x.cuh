// X passes of the demag convolution on register FFTs (fft_lane.cuh): real
// rows <-> half spectra through a complex transform of half the padded
// length, M = G * Q, with one shared-memory exchange per row.
//
// G threads share a row.  Forward: thread t transforms the Q strided pairs
// z[q G + t] = x[2n] + i x[2n+1], twiddles them and stores them; then each
// thread takes "slots" of two items (k1, Q - k1), G points each: their
// spectra hold Z[k] and Z[M - k] for the same k, so the split
//   X[k] = E + W^k O,  X[M-k] = conj(E - W^k O),
//   E = (Z[k] + conj Z[M-k]) / 2,  O = -i (Z[k] - conj Z[M-k]) / 2
// happens in registers, one twiddle per pair.  Slot 0 holds the items 0 and
// Q/2, which pair with themselves.  Inverse: the same backwards.  Rows of a
// power-of-two G stay within a warp and need no CTA barrier.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "ctx.h"
#include "fft_lane.cuh"

namespace mm {

template <typename T>
struct XLaneArgs {
    const T* in;                // forward, stage 0: rows of [component][z][y][x]
    T* out;                     // inverse: rows
    cplx<T>* spec;              // [component][z][spec_rows][Wk]
    int rows, rows_per_plane, spec_rows_per_plane, nx, Wk;
    long long cells;            // cells per component: row r starts at cell (r nx) mod cells
    const cplx<T>* tw;          // exp(-2 pi i q / (2 M))
    T ms;                       // uniform Ms, or per region:
    const uint8_t* region;
    const Region<T>* lut;
    // stage > 0: the rows are the RK45 stage state m0 + sum_j (dt a_sj) k_j,
    // formed here and kept in ms_out
    const DevState* st;
    const T* k[7];              // slopes; slots 0 and 6 swap roles with st->k_first
    const T* m0;
    T* ms_out;
    int stage;
};

template <int M, int G, int Q>
struct XSplit {
    static_assert(M == G * Q, "row split");
    static constexpr int NS = Q % 2 ? (Q + 1) / 2 : (Q > 1 ? Q / 2 : 1);   // slots per row
    static constexpr int NSL = (NS + G - 1) / G;                            // per thread
    static constexpr int NB = Q % 2 ? 0 : (G + 1) / 2;                      // pairs of item Q/2 in slot 0
    static constexpr int NE = NB + G / 2 + 1;                               // all pairs of slot 0 (at most G + 1)
    static constexpr int QIN = ((M + 1) / 2 + G - 1) / G;                   // strided inputs that can be nonzero
    static constexpr int US = Q | 1;                                        // odd: threads write to different banks
    static constexpr int LINE = G * US;                                     // complex values per row
    static constexpr bool WARP = (32 % G) == 0;                             // a row never crosses a warp
};
template <bool WARP> __device__ __forceinline__ void xsync() {
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
}
template <typename T> __device__ __forceinline__ const T* stage_row(const DevState* st, int s);
template <> __device__ __forceinline__ const float* stage_row<float>(const DevState* st, int s) { return st->cf32[s]; }
template <> __device__ __forceinline__ const double* stage_row<double>(const DevState* st, int s) { return st->cf64[s]; }

// The RK45 stage state m0 + sum_{j < stage} (dt a_sj) k_j of the thread's pairs
// of an even row.  Two slopes at a time: enough loads on their way at once, and
// one body for every stage (a body per stage cost more in instruction fetches
// than it gave: a 256x256 film's forward pass spent half its time on them).
template <typename T, int G, int QIN>
__device__ __forceinline__ void x_stage_pairs(const XLaneArgs<T>& a, long long g0, int t, int nin, cplx<T> (&x)[QIN]) {
    const T* cf = stage_row<T>(a.st, a.stage);
    const int kf = a.st->k_first;
    const long long o = g0 / 2;                                   // in pairs: even rows
    auto slot = [&](int s) { return reinterpret_cast<const cplx<T>*>(s == 0 ? (kf ? a.k[6] : a.k[0]) : a.k[s]) + o; };
#pragma unroll
    for (int q = 0; q < QIN; ++q)
        x[q] = q * G + t < nin ? reinterpret_cast<const cplx<T>*>(a.m0)[o + q * G + t] : mkc<T>(0, 0);
#pragma unroll 1
    for (int s = 0; s < a.stage; s += 2) {
        const bool two = s + 1 < a.stage && !(s == 0 && a.stage == 6);   // a_7,2 = 0
        const T c0 = cf[s], c1 = two ? cf[s + 1] : (T)0;
        const cplx<T>*k0 = slot(s), *k1 = two ? slot(s + 1) : k0;
        cplx<T> d0[QIN], d1[QIN];
#pragma unroll
        for (int q = 0; q < QIN; ++q) d0[q] = q * G + t < nin ? k0[q * G + t] : mkc<T>(0, 0);
#pragma unroll
        for (int q = 0; q < QIN; ++q) d1[q] = two && q * G + t < nin ? k1[q * G + t] : mkc<T>(0, 0);
#pragma unroll
        for (int q = 0; q < QIN; ++q) {
            x[q].x = x[q].x + c0 * d0[q].x;
            x[q].y = x[q].y + c0 * d0[q].y;
            x[q].x = x[q].x + c1 * d1[q].x;
            x[q].y = x[q].y + c1 * d1[q].y;
        }
    }
}

template <typename T> __device__ __forceinline__ lcx<T> xsel(bool c, lcx<T> a, lcx<T> b) { return {c ? a.re : b.re, c ? a.im : b.im}; }

// X[k] and X[M-k] from Z[k], Z[M-k]; w = W^k as (cos, -sin)
template <typename T>
__device__ __forceinline__ void x_split(lcx<T> z, lcx<T> zm, cplx<T> w, cplx<T>& xk, cplx<T>& xm) {
    const T h = (T)0.5;
    const T er = h * (z.re + zm.re), ei = h * (z.im - zm.im);
    const T orr = h * (z.im + zm.im), oi = h * (zm.re - z.re);              // -i (z - conj zm) / 2
    const T pr = w.x * orr - w.y * oi, pi = w.x * oi + w.y * orr;
    xk = mkc<T>(er + pr, ei + pi);
    xm = mkc<T>(er - pr, pi - ei);
}
// Z'[k] and Z'[M-k] from X[k], X[M-k] (unnormalised)
template <typename T>
__device__ __forceinline__ void x_merge(cplx<T> xk, cplx<T> xm, cplx<T> w, lcx<T>& z, lcx<T>& zm) {
    const T er = xk.x + xm.x, ei = xk.y - xm.y, dr = xk.x - xm.x, di = xk.y + xm.y;
    const T orr = dr * w.x + di * w.y, oi = di * w.x - dr * w.y;            // d conj(w)
    z = {er - oi, ei + orr};
    zm = {er + oi, orr - ei};
}

// Half spectrum X[0..M] of one row to the pairs of its real values:
// store(n, (x[2n], x[2n+1])) for n = q G + t, q < QIN.  sm: the row's LINE
// values; taken() runs when they are in registers.  INPLACE: X lies where sm
// does (the rows of a warp; no store to a row that is not valid).
template <typename T, int M, int G, int Q, bool INPLACE = false, typename Taken, typename Store>
__device__ __forceinline__ void lane_c2r_row(const cplx<T>* X, const cplx<T>* __restrict__ tw, lcx<T>* sm,
                                             int t, bool valid, Taken taken, Store store) {
    using S = XSplit<M, G, Q>;
    static_assert(!INPLACE || S::WARP, "in place: rows within warps");
    lcx<T> zks[INPLACE ? S::NSL : 1][G + 1], zms[INPLACE ? S::NSL : 1][G + 1];
    auto gather = [&](int i, lcx<T>* zk, lcx<T>* zm) {
        const int j = t + i * G;
#pragma unroll
        for (int e = 0; e < (i == 0 ? (S::NE > G ? S::NE : G) : G); ++e) {
            int k = j + Q * e;
            if (i == 0 && j == 0) k = e < S::NB ? Q / 2 + Q * e : Q * (e - S::NB);
            if (i == 0 && e >= G && j != 0) k = 0;
            if (i == 0 && j == 0 && e >= S::NE) k = 0;
            cplx<T> xk = mkc<T>(0, 0), xm = mkc<T>(0, 0);
            if (valid) { xk = X[k]; xm = X[M - k]; }
            x_merge<T>(xk, xm, __ldg(tw + k), zk[e], zm[e]);
        }
    };
    if constexpr (INPLACE) {
#pragma unroll
        for (int i = 0; i < S::NSL; ++i)
            if (t + i * G < S::NS) gather(i, zks[i], zms[i]);
        __syncwarp();                                             // every value of the spectrum is in registers
    }
#pragma unroll
    for (int i = 0; i < S::NSL; ++i) {
        const int j = t + i * G;
        if (S::NS % G != 0 && j >= S::NS) continue;
        lcx<T>* zk = zks[INPLACE ? i : 0];
        lcx<T>* zm = zms[INPLACE ? i : 0];
        if (!INPLACE) gather(i, zk, zm);
        if (INPLACE && !valid) continue;
        lcx<T> a[G], b[G];
#pragma unroll
        for (int x = 0; x < G; ++x) {
            a[x] = zk[x];
            b[x] = zm[G - 1 - x];
            if (i == 0 && j == 0) {
                a[x] = x <= G / 2 ? zk[S::NB + x] : zm[S::NB + G - x];
                if (S::NB > 0) b[x] = x < S::NB ? zk[x] : zm[G - 1 - x];
            }
        }
        lfft<-1, G, T>(a);
        lfft<-1, G, T>(b);
        const int k1 = j, k1b = i == 0 && j == 0 ? Q / 2 : Q - j;
#pragma unroll
        for (int u = 0; u < G; ++u) {
            sm[u * S::US + k1] = u > 0 ? lctwr<-1>(a[u], ltw_load<T>(tw, 2 * u * k1)) : a[u];
            if (Q > 1 && !(Q % 2 && i == 0 && j == 0))
                sm[u * S::US + k1b] = u > 0 ? lctwr<-1>(b[u], ltw_load<T>(tw, 2 * u * k1b)) : b[u];
        }
    }
    xsync<S::WARP>();
    lcx<T> v[Q];
#pragma unroll
    for (int k1 = 0; k1 < Q; ++k1) v[k1] = sm[t * S::US + k1];
    taken();
    lfft<-1, Q, T>(v);
#pragma unroll
    for (int q = 0; q < S::QIN; ++q) store(q * G + t, mkc<T>(v[q].re, v[q].im));
}

// What the rows of a forward pass are: a state with one Ms, the RK45 stage
// state with one Ms (both of even length), or anything (odd rows, many
// materials).
enum XInput { X_PLAIN = 0, X_STAGE = 1, X_ANY = 2 };

template <typename T, int M, int G, int Q, int ROWS, int IN>
__global__ void __launch_bounds__(G* ROWS) lane_r2c_kernel(XLaneArgs<T> a) {
    using S = XSplit<M, G, Q>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dep_wait();
    if (IN != X_PLAIN && a.stage > 0 && !a.st->active) return;
    const int t = threadIdx.x % G, rl = threadIdx.x / G;
    lcx<T>* sm = reinterpret_cast<lcx<T>*>(smem_raw) + rl * S::LINE;
    const int row = blockIdx.x * (blockDim.x / G) + rl;
    if (row >= a.rows) return;                                    // (its row's threads only: barriers do not wait for them)
    const int nin = (a.nx + 1) / 2;
    const long long g0 = (long long)row * a.nx;
    lcx<T> v[Q];
    // ---- packed pairs of the row times Ms of their cells
    if constexpr (IN != X_ANY) {
        cplx<T> x[S::QIN];
        if constexpr (IN == X_STAGE) {
            x_stage_pairs<T, G, S::QIN>(a, g0, t, nin, x);
#pragma unroll
            for (int q = 0; q < S::QIN; ++q)
                if (q * G + t < nin) reinterpret_cast<cplx<T>*>(a.ms_out + g0)[q * G + t] = x[q];
        } else {
#pragma unroll
            for (int q = 0; q < S::QIN; ++q)
                x[q] = q * G + t < nin ? reinterpret_cast<const cplx<T>*>(a.in + g0)[q * G + t] : mkc<T>(0, 0);
        }
#pragma unroll
        for (int q = 0; q < S::QIN; ++q) v[q] = {x[q].x * a.ms, x[q].y * a.ms};
    } else {
        // single values where the row is odd (no alignment; the last pair is half empty)
        T x[2 * S::QIN];
        const bool even = a.nx % 2 == 0;
        auto fill = [&](const T* src, T c, bool first) {          // x (+)= c src
            if (even) {
                const cplx<T>* p = reinterpret_cast<const cplx<T>*>(src + g0);
#pragma unroll
                for (int q = 0; q < S::QIN; ++q) {
                    const cplx<T> d = q * G + t < nin ? p[q * G + t] : mkc<T>(0, 0);
                    x[2 * q] = first ? d.x : x[2 * q] + c * d.x;
                    x[2 * q + 1] = first ? d.y : x[2 * q + 1] + c * d.y;
                }
            } else {
#pragma unroll
                for (int q = 0; q < 2 * S::QIN; ++q) {
                    const int n = 2 * ((q / 2) * G + t) + q % 2;
                    const T d = n < a.nx ? src[g0 + n] : (T)0;
                    x[q] = first ? d : x[q] + c * d;
                }
            }
        };
        fill(a.stage > 0 ? a.m0 : a.in, (T)1, true);
        if (a.stage > 0) {
            const T* cf = stage_row<T>(a.st, a.stage);
            const int kf = a.st->k_first;
#pragma unroll 1
            for (int s = 0; s < a.stage; ++s)
                if (!(s == 1 && a.stage == 6)) fill(s == 0 ? (kf ? a.k[6] : a.k[0]) : a.k[s], cf[s], false);   // a_7,2 = 0
#pragma unroll
            for (int q = 0; q < 2 * S::QIN; ++q) {
                const int n = 2 * ((q / 2) * G + t) + q % 2;
                if (n < a.nx) a.ms_out[g0 + n] = x[q];
            }
        }
        if (a.region) {
            const uint8_t* rg = a.region + g0 % a.cells;
#pragma unroll
            for (int q = 0; q < 2 * S::QIN; ++q) {
                const int n = 2 * ((q / 2) * G + t) + q % 2;
                if (n < a.nx) x[q] *= __ldg(&a.lut[rg[n]].Ms);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 2 * S::QIN; ++q) x[q] *= a.ms;
        }
#pragma unroll
        for (int q = 0; q < S::QIN; ++q) v[q] = {x[2 * q], x[2 * q + 1]};
    }
#pragma unroll
    for (int q = S::QIN; q < Q; ++q) v[q] = lzero<T>();
    lfft<1, Q, T, (S::QIN < Q ? S::QIN : Q)>(v);
#pragma unroll
    for (int k1 = 0; k1 < Q; ++k1)
        sm[t * S::US + k1] = k1 > 0 && G > 1 ? lctwr<1>(v[k1], ltw_load<T>(a.tw, 2 * t * k1)) : v[k1];
    xsync<S::WARP>();

    cplx<T>* out = a.spec + ((long long)(row / a.rows_per_plane) * a.spec_rows_per_plane + row % a.rows_per_plane) * a.Wk;
#pragma unroll
    for (int i = 0; i < S::NSL; ++i) {
        const int j = t + i * G;
        if (S::NS % G != 0 && j >= S::NS) continue;
        const bool s0 = i == 0 && j == 0;                         // slot 0: items 0 and Q/2
        const int k1b = s0 ? Q / 2 : Q - j;
        lcx<T> z[G], y[G];
#pragma unroll
        for (int u = 0; u < G; ++u) {
            z[u] = sm[u * S::US + j];
            y[u] = sm[u * S::US + k1b];                           // (odd Q, slot 0: unused)
        }
        lfft<1, G, T>(z);
        lfft<1, G, T>(y);
#pragma unroll
        for (int e = 0; e < (i == 0 ? (S::NE > G ? S::NE : G) : G); ++e) {
            constexpr int nb = S::NB;
            const int x = e - nb;                                 // slot 0, pair of item 0
            lcx<T> p = z[e < G ? e : 0], m = y[e < G ? G - 1 - e : 0];
            int k = j + Q * e;
            if (i == 0) {
                if (e < nb) {
                    p = xsel(s0, y[e < G ? e : 0], p);
                    k = s0 ? Q / 2 + Q * e : k;
                } else {
                    p = xsel(s0, z[x >= 0 && x < G ? x : 0], p);
                    m = xsel(s0, z[x >= 0 && x < G ? (G - x) % G : 0], m);
                    k = s0 ? Q * x : k;
                }
            }
            const bool on = e < G ? (e < S::NE || !s0) : s0;      // mostly known at compile time
            cplx<T> xk, xm;
            x_split<T>(p, m, __ldg(a.tw + (on ? k : 0)), xk, xm);
            if (on) {
                out[k] = xk;
                out[M - k] = xm;
            }
        }
    }
}

template <typename T, int M, int G, int Q, int ROWS>
__global__ void __launch_bounds__(G* ROWS) lane_c2r_kernel(XLaneArgs<T> a) {
    using S = XSplit<M, G, Q>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dep_wait();
    const int t = threadIdx.x % G, rl = threadIdx.x / G;
    lcx<T>* sm = reinterpret_cast<lcx<T>*>(smem_raw) + rl * S::LINE;
    const int row = blockIdx.x * (blockDim.x / G) + rl;
    if (row >= a.rows) return;                                    // (its row's threads only)
    const cplx<T>* X = a.spec + ((long long)(row / a.rows_per_plane) * a.spec_rows_per_plane + row % a.rows_per_plane) * a.Wk;
    T* out = a.out + (long long)row * a.nx;
    const int nx = a.nx;
    lane_c2r_row<T, M, G, Q>(X, a.tw, sm, t, true, [] {}, [&](int n, cplx<T> v) {
        if (nx % 2 == 0) {
            if (2 * n < nx) reinterpret_cast<cplx<T>*>(out)[n] = v;
        } else {
            if (2 * n < nx) out[2 * n] = v.x;
            if (2 * n + 1 < nx) out[2 * n + 1] = v.y;
        }
    });
}

// ---------------------------------------------------------------------------
// A row per warp in radix-4 Stockham passes: for FP64 grids of a few hundred
// rows.  An FP64 instruction of a warp holds its scheduler for 64 clocks (two
// fused multiply-adds per clock and SM), so what counts there is the number
// of instructions per warp with every warp on a scheduler of its own: 130 per
// row of M = 128 on 32 lanes against 400 for four rows on the G = 8 split.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int fine_radix(int M, int p) {
    int n = M;
    for (int q = 0;; ++q) {
        const int r = n % 4 == 0 ? 4 : n % 2 == 0 ? 2 : n % 3 == 0 ? 3 : 1;
        if (q == p) return r;
        n /= r;
    }
}
__host__ __device__ constexpr int fine_npass(int M) {
    int n = M, p = 0;
    while (n > 1) { n /= fine_radix(M, p); ++p; }
    return p;
}
__host__ __device__ constexpr int fine_ns(int M, int p) {
    int ns = 1;
    for (int q = 0; q < p; ++q) ns *= fine_radix(M, q);
    return ns;
}
__host__ __device__ constexpr int fine_at(int i) { return i + (i >> 3); }
__host__ __device__ constexpr int fine_line(int M) { return fine_at(M) + 1; }

template <typename T, int DIR, int M, int P, int TS = 2, typename Load, typename Store>
__device__ __forceinline__ void fine_pass(const cplx<T>* __restrict__ tw, Load load, Store store) {
    constexpr int R = fine_radix(M, P), NS = fine_ns(M, P), NB = M / R, SPAN = M / (NS * R), NBL = (NB + 31) / 32;
    const int lane_id = threadIdx.x & 31;
    lcx<T> v[NBL][R];
#pragma unroll
    for (int i = 0; i < NBL; ++i) {
        const int j = lane_id + 32 * i;
        if (NB % 32 == 0 || j < NB) {
#pragma unroll
            for (int t = 0; t < R; ++t) v[i][t] = load(j + t * NB);
        }
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NBL; ++i) {
        const int j = lane_id + 32 * i;
        if (NB % 32 != 0 && j >= NB) continue;
        const int k = j % NS;
        if constexpr (NS > 1) {
#pragma unroll
            for (int t = 1; t < R; ++t) v[i][t] = lctwr<DIR>(v[i][t], ltw_load<T>(tw, TS * t * k * SPAN));
        }
        bool zu[R];
#pragma unroll
        for (int t = 0; t < R; ++t) zu[t] = DIR > 0 && P == 0 && R == 4 && t >= 2;   // the zero-padded half of a row
        ldft<DIR, R, T>(v[i], zu);
        const int dst = (j / NS) * NS * R + k;
#pragma unroll
        for (int t = 0; t < R; ++t) store(dst + t * NS, v[i][t]);
    }
    __syncwarp();
}
// passes P .. PE - 1, shared memory to shared memory
template <typename T, int DIR, int M, int P, int PE, int TS = 2>
__device__ __forceinline__ void fine_passes(lcx<T>* sm, const cplx<T>* __restrict__ tw) {
    if constexpr (P < PE) {
        fine_pass<T, DIR, M, P, TS>(tw, [&](int i) { return sm[fine_at(i)]; }, [&](int i, lcx<T> v) { sm[fine_at(i)] = v; });
        fine_passes<T, DIR, M, P + 1, PE, TS>(sm, tw);
    }
}

template <typename T, int M>
__global__ void __launch_bounds__(128) fine_r2c_kernel(XLaneArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dep_wait();
    if (a.stage > 0 && !a.st->active) return;
    lcx<T>* sm = reinterpret_cast<lcx<T>*>(smem_raw) + (threadIdx.x >> 5) * fine_line(M);
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= a.rows) return;                                    // whole warp
    const long long g0 = (long long)row * a.nx;
    const int kf = a.stage > 0 ? a.st->k_first : 0;
    const T* cf = a.stage > 0 ? stage_row<T>(a.st, a.stage) : nullptr;
    const uint8_t* rg = a.region ? a.region + g0 % a.cells : nullptr;
    auto value = [&](int n) -> T {                                // Ms x[n], the stage state formed and kept
        if (n >= a.nx) return (T)0;
        const long long e = g0 + n;
        T x;
        if (a.stage > 0) {
            T k[6];
#pragma unroll
            for (int s = 0; s < 6; ++s)
                k[s] = s < a.stage && !(s == 1 && a.stage == 6) ? (s == 0 ? (kf ? a.k[6] : a.k[0]) : a.k[s])[e] : (T)0;
            x = a.m0[e];
#pragma unroll
            for (int s = 0; s < 6; ++s)
                if (s < a.stage && !(s == 1 && a.stage == 6)) x += cf[s] * k[s];
            a.ms_out[e] = x;
        } else {
            x = a.in[e];
        }
        return rg ? x * __ldg(&a.lut[rg[n]].Ms) : x * a.ms;
    };
    constexpr int NP = fine_npass(M);
    fine_pass<T, 1, M, 0>(a.tw, [&](int i) -> lcx<T> { return {value(2 * i), value(2 * i + 1)}; },
                          [&](int i, lcx<T> v) { sm[fine_at(i)] = v; });
    fine_passes<T, 1, M, 1, NP>(sm, a.tw);
    cplx<T>* out = a.spec + ((long long)(row / a.rows_per_plane) * a.spec_rows_per_plane + row % a.rows_per_plane) * a.Wk;
    for (int k = threadIdx.x & 31; k <= M / 2; k += 32) {
        cplx<T> xk, xm;
        x_split<T>(sm[fine_at(k)], sm[fine_at(k == 0 ? 0 : M - k)], __ldg(a.tw + k), xk, xm);
        out[k] = xk;
        out[M - k] = xm;
    }
}

// Half spectrum of one row to store(n, (x[2n], x[2n+1])), by one warp; sm: the
// row's fine_line values.
template <typename T, int M, typename Store>
__device__ __forceinline__ void fine_c2r_row(const cplx<T>* X, const cplx<T>* __restrict__ tw, lcx<T>* sm, Store store) {
    for (int k = threadIdx.x & 31; k <= M / 2; k += 32) {
        lcx<T> z, zm;
        x_merge<T>(X[k], X[M - k], __ldg(tw + k), z, zm);
        sm[fine_at(k)] = z;
        if (k > 0 && 2 * k != M) sm[fine_at(M - k)] = zm;
    }
    __syncwarp();
    constexpr int NP = fine_npass(M);
    fine_passes<T, -1, M, 0, NP - 1>(sm, tw);
    fine_pass<T, -1, M, NP - 1>(tw, [&](int i) { return sm[fine_at(i)]; }, store);
}

template <typename T, int M>
__global__ void __launch_bounds__(128) fine_c2r_kernel(XLaneArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    dep_wait();
    lcx<T>* sm = reinterpret_cast<lcx<T>*>(smem_raw) + (threadIdx.x >> 5) * fine_line(M);
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= a.rows) return;                                    // whole warp
    const cplx<T>* X = a.spec + ((long long)(row / a.rows_per_plane) * a.spec_rows_per_plane + row % a.rows_per_plane) * a.Wk;
    T* out = a.out + (long long)row * a.nx;
    fine_c2r_row<T, M>(X, a.tw, sm, [&](int n, lcx<T> v) {
        if (2 * n < a.nx) out[2 * n] = v.re;
        if (2 * n + 1 < a.nx) out[2 * n + 1] = v.im;
    });
}

// Middle pass of one FP64 film, a column per CTA and a component per warp, in
// the same passes: 180 FP64 instructions per warp at L = 64 against 400 on the
// 8 x 8 split of conv_lane.cuh.
template <typename T>
struct FineFilmArgs {
    cplx<T>* base;              // [component][y][Wk]
    long long comp_stride;
    int Wk, ny;
    const T* khat;              // [4][L/2+1][Wk]
    long long kc;
    const cplx<T>* tw;          // exp(-2 pi i q / L)
};

template <typename T, int L>
__global__ void __launch_bounds__(96) fine_film_kernel(FineFilmArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int NP = fine_npass(L), PER = (L + 31) / 32;
    const int c = threadIdx.x >> 5, lane_id = threadIdx.x & 31, kx = blockIdx.x;
    lcx<T>* line = reinterpret_cast<lcx<T>*>(smem_raw) + c * fine_line(L);
    lcx<T>* other = reinterpret_cast<lcx<T>*>(smem_raw) + (1 - c) * fine_line(L);   // c < 2
    // this thread's tensor values: diagonal and, for x and y, the coupling
    T kd[PER], ko[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int k = lane_id + 32 * i, kf = k <= L / 2 ? k : L - k;
        kd[i] = ko[i] = (T)0;
        if (k < L) {
            kd[i] = __ldg(a.khat + c * a.kc + (long long)kf * a.Wk + kx);
            if (c < 2) ko[i] = __ldg(a.khat + 3 * a.kc + (long long)kf * a.Wk + kx) * (k <= L / 2 ? (T)1 : (T)-1);
        }
    }
    dep_wait();                                                   // (the tensor is older than any launch)
    cplx<T>* g = a.base + c * a.comp_stride + kx;
    fine_pass<T, 1, L, 0, 1>(a.tw, [&](int n) -> lcx<T> {
        if (n >= a.ny) return lzero<T>();
        const cplx<T> x = g[(long long)n * a.Wk];
        return {x.x, x.y};
    }, [&](int i, lcx<T> v) { line[fine_at(i)] = v; });
    fine_passes<T, 1, L, 1, NP, 1>(line, a.tw);
    __syncthreads();
    lcx<T> h[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int k = lane_id + 32 * i;
        h[i] = lzero<T>();
        if (k < L) {
            const lcx<T> m = line[fine_at(k)];
            h[i] = {kd[i] * m.re, kd[i] * m.im};
            if (c < 2) {
                const lcx<T> o = other[fine_at(k)];
                h[i] = {fma(ko[i], o.re, h[i].re), fma(ko[i], o.im, h[i].im)};
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < PER; ++i)
        if (lane_id + 32 * i < L) line[fine_at(lane_id + 32 * i)] = h[i];
    __syncwarp();
    fine_passes<T, -1, L, 0, NP - 1, 1>(line, a.tw);
    fine_pass<T, -1, L, NP - 1, 1>(a.tw, [&](int i) { return line[fine_at(i)]; }, [&](int n, lcx<T> v) {
        if (n < a.ny) g[(long long)n * a.Wk] = mkc<T>(v.re, v.im);
    });
}

}  // namespace mm
