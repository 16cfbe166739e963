// Register FFTs over "lanes": the real type N of a complex value is float2
// (two neighbouring columns side by side, every operation one packed
// two-lane instruction), float or double.  Real and imaginary parts are
// separate N values, so a quarter turn is a renaming and an addition, a
// twiddle or the tensor product costs one packed instruction where the
// (re, im) layout needs one per part.  Twiddles with a compile-time exponent
// are literals; every index is a compile-time constant after unrolling.
#pragma once

#include "common.cuh"
#include "fft_ct.cuh"

namespace mm {

// cos and sin of 2 pi q / L for 0 <= q < L: the angle is reduced to the first
// octant in integers, then summed as a Taylor series in double.
struct LaneTrig { double c, s; };
constexpr LaneTrig lane_trig(int q, int L) {
    // eighths of a turn: e = floor(8 q / L), remainder r / (8 L) turns of ...
    int e = 8 * q / L;
    int r = 8 * q - e * L;                    // 0 <= r < L: angle = (e + r / L) * pi / 4
    const bool odd = e & 1;
    if (odd) r = L - r;                       // reflect: angle within the octant from its nearer axis
    const double x = kPi / 4.0 * (double)r / (double)L;
    double s = 0.0, c = 0.0, t = 1.0;
    for (int n = 0; n < 24; ++n) {            // t = x^n / n!
        const double sg = (n / 2) % 2 ? -1.0 : 1.0;
        if (n % 2) s += sg * t;
        else c += sg * t;
        t = t * x / (n + 1);
    }
    // odd octants: angle = (e + 1) pi / 4 - x, even: e pi / 4 + x
    const int quarter = (odd ? e + 1 : e) / 2 % 4;
    const double sx = odd ? -s : s;
    if (quarter == 0) return {c, sx};
    if (quarter == 1) return {-sx, c};
    if (quarter == 2) return {-c, -sx};
    return {sx, -c};
}
template <int L>
struct LaneTable {
    double c[L], s[L];
    constexpr LaneTable() : c(), s() {
        for (int q = 0; q < L; ++q) {
            const LaneTrig v = lane_trig(q, L);
            c[q] = v.c;
            s[q] = v.s;
        }
    }
};
template <int L> __device__ constexpr LaneTable<L> lane_table{};

// ---- lane arithmetic ------------------------------------------------------
__device__ __forceinline__ float2 ladd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 lsub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 lmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 lfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float ladd(float a, float b) { return a + b; }
__device__ __forceinline__ float lsub(float a, float b) { return a - b; }
__device__ __forceinline__ float lmul(float a, float b) { return a * b; }
__device__ __forceinline__ float lfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double ladd(double a, double b) { return a + b; }
__device__ __forceinline__ double lsub(double a, double b) { return a - b; }
__device__ __forceinline__ double lmul(double a, double b) { return a * b; }
__device__ __forceinline__ double lfma(double a, double b, double c) { return fma(a, b, c); }

template <typename N> struct lane;
template <> struct lane<float2> {
    using real = float;
    static constexpr int width = 2;
    static __device__ __forceinline__ float2 all(double v) { return make_float2((float)v, (float)v); }
};
template <> struct lane<float> {
    using real = float;
    static constexpr int width = 1;
    static __device__ __forceinline__ float all(double v) { return (float)v; }
};
template <> struct lane<double> {
    using real = double;
    static constexpr int width = 1;
    static __device__ __forceinline__ double all(double v) { return v; }
};

template <typename N> struct alignas(2 * sizeof(N)) lcx { N re, im; };

template <typename N> __device__ __forceinline__ lcx<N> lzero() { return {lane<N>::all(0.0), lane<N>::all(0.0)}; }
template <typename N> __device__ __forceinline__ lcx<N> lcadd(lcx<N> a, lcx<N> b) { return {ladd(a.re, b.re), ladd(a.im, b.im)}; }
template <typename N> __device__ __forceinline__ lcx<N> lcsub(lcx<N> a, lcx<N> b) { return {lsub(a.re, b.re), lsub(a.im, b.im)}; }
// z: b is known to be zero (compile time, after unrolling)
template <typename N> __device__ __forceinline__ lcx<N> lcadd(lcx<N> a, lcx<N> b, bool z) { return z ? a : lcadd(a, b); }
template <typename N> __device__ __forceinline__ lcx<N> lcsub(lcx<N> a, lcx<N> b, bool z) { return z ? a : lcsub(a, b); }
// a + (-i)^DIR t, a - (-i)^DIR t
template <int DIR, typename N> __device__ __forceinline__ lcx<N> lcadd_rot(lcx<N> a, lcx<N> t) {
    return DIR > 0 ? lcx<N>{ladd(a.re, t.im), lsub(a.im, t.re)} : lcx<N>{lsub(a.re, t.im), ladd(a.im, t.re)};
}
// v * (c - i s) (DIR > 0: the forward twiddle of cos c, sin s) or v * (c + i s)
template <int DIR, typename N> __device__ __forceinline__ lcx<N> lctw(lcx<N> v, N c, N s, N ms) {
    // ms = -s
    if (DIR > 0) return {lfma(v.im, s, lmul(v.re, c)), lfma(v.re, ms, lmul(v.im, c))};
    return {lfma(v.im, ms, lmul(v.re, c)), lfma(v.re, s, lmul(v.im, c))};
}
// v * W_L^q (DIR > 0) or its conjugate; q a compile-time constant after unrolling
template <int DIR, int L, typename N> __device__ __forceinline__ lcx<N> lctwq(lcx<N> v, int q) {
    if (q == 0) return v;
    const double c = lane_table<L>.c[q], s = lane_table<L>.s[q];
    return lctw<DIR, N>(v, lane<N>::all(c), lane<N>::all(s), lane<N>::all(-s));
}

// ---- butterflies ----------------------------------------------------------
template <int DIR, typename N>
__device__ __forceinline__ void ldft4(lcx<N>& a, lcx<N>& b, lcx<N>& c, lcx<N>& d, bool zc, bool zd) {
    const lcx<N> a0 = lcadd(a, c, zc), a1 = lcsub(a, c, zc), a2 = lcadd(b, d, zd), t = lcsub(b, d, zd);
    a = lcadd(a0, a2);
    c = lcsub(a0, a2);
    b = lcadd_rot<DIR>(a1, t);
    d = lcadd_rot<-DIR>(a1, t);
}

// R-point DFT in place; zu[t]: input t is known zero (only a trailing run)
template <int DIR, int R, typename N>
__device__ __forceinline__ void ldft(lcx<N>* v, const bool* zu) {
    if constexpr (R == 2) {
        const lcx<N> a = v[0], b = v[1];
        v[0] = lcadd(a, b, zu[1]);
        v[1] = lcsub(a, b, zu[1]);
    } else if constexpr (R == 3) {
        const N h = lane<N>::all(-0.5), s3 = lane<N>::all(0.86602540378443864676), m3 = lane<N>::all(-0.86602540378443864676);
        const lcx<N> t1 = lcadd(v[1], v[2], zu[2]), t3 = lcsub(v[1], v[2], zu[2]);
        const lcx<N> t2 = {lfma(t1.re, h, v[0].re), lfma(t1.im, h, v[0].im)};
        v[0] = lcadd(v[0], t1);
        // t2 +- (-i)^DIR s3 t3
        const N p = DIR > 0 ? s3 : m3, q = DIR > 0 ? m3 : s3;
        v[1] = {lfma(t3.im, p, t2.re), lfma(t3.re, q, t2.im)};
        v[2] = {lfma(t3.im, q, t2.re), lfma(t3.re, p, t2.im)};
    } else if constexpr (R == 4) {
        ldft4<DIR>(v[0], v[1], v[2], v[3], zu[2], zu[3]);
    } else {
        static_assert(R == 8, "radix 2, 3, 4 or 8");
        const N h = lane<N>::all(0.70710678118654752440);
        lcx<N> b0 = lcadd(v[0], v[4], zu[4]), c0 = lcsub(v[0], v[4], zu[4]);
        lcx<N> b1 = lcadd(v[1], v[5], zu[5]), c1 = lcsub(v[1], v[5], zu[5]);
        lcx<N> b2 = lcadd(v[2], v[6], zu[6]), t2 = lcsub(v[2], v[6], zu[6]);
        lcx<N> b3 = lcadd(v[3], v[7], zu[7]), c3 = lcsub(v[3], v[7], zu[7]);
        // c1 *= W8, c3 *= W8^3 up to the factor h; the sign of W8^3 is taken into the sums below
        c1 = DIR > 0 ? lcx<N>{ladd(c1.re, c1.im), lsub(c1.im, c1.re)} : lcx<N>{lsub(c1.re, c1.im), ladd(c1.im, c1.re)};
        c3 = DIR > 0 ? lcx<N>{lsub(c3.im, c3.re), ladd(c3.re, c3.im)} : lcx<N>{ladd(c3.re, c3.im), lsub(c3.im, c3.re)};
        // now W8 v1 = h c1; W8^3 v3 = h (c3.re, -c3.im) forward, -h c3 inverse
        const lcx<N> w3 = c3;
        lcx<N> a2, t;
        if (DIR > 0) {
            a2 = {ladd(c1.re, w3.re), lsub(c1.im, w3.im)};
            t = {lsub(c1.re, w3.re), ladd(c1.im, w3.im)};
        } else {
            a2 = lcsub(c1, w3);
            t = lcadd(c1, w3);
        }
        ldft4<DIR>(b0, b1, b2, b3, false, false);
        const lcx<N> a0 = lcadd_rot<DIR>(c0, t2), a1 = lcadd_rot<-DIR>(c0, t2);
        const N mh = lane<N>::all(-0.70710678118654752440);
        v[0] = b0; v[2] = b1; v[4] = b2; v[6] = b3;
        v[1] = {lfma(a2.re, h, a0.re), lfma(a2.im, h, a0.im)};
        v[5] = {lfma(a2.re, mh, a0.re), lfma(a2.im, mh, a0.im)};
        // a1 +- (-i)^DIR h t
        const N p = DIR > 0 ? h : mh, q = DIR > 0 ? mh : h;
        v[3] = {lfma(t.im, p, a1.re), lfma(t.re, q, a1.im)};
        v[7] = {lfma(t.im, q, a1.re), lfma(t.re, p, a1.im)};
    }
}

// In-register DFT of length M, natural order in and out, mixed radix 8/4/2/3
// Stockham passes.  Inputs at index >= NZ are known zeros (the zero-padded
// part of a line): their additions fold away.
template <int DIR, int M, typename N, int NZ = M, int P = 0>
__device__ __forceinline__ void lfft(lcx<N> (&v)[M]) {
    if constexpr (P < ct_npass(M)) {
        constexpr int R = ct_radix(M, P), NS = ct_ns(M, P), NB = M / R, SPAN = M / (NS * R);
        lcx<N> w[M];
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            lcx<N> u[R];
            bool zu[R];
#pragma unroll
            for (int t = 0; t < R; ++t) {
                u[t] = v[j + t * NB];
                zu[t] = P == 0 && j + t * NB >= NZ;
            }
            const int k = j % NS;
            if constexpr (NS > 1) {
#pragma unroll
                for (int t = 1; t < R; ++t) u[t] = lctwq<DIR, M, N>(u[t], t * k * SPAN);
            }
            ldft<DIR, R, N>(u, zu);
            const int dst = (j / NS) * NS * R + k;
#pragma unroll
            for (int t = 0; t < R; ++t) w[dst + t * NS] = u[t];
        }
#pragma unroll
        for (int i = 0; i < M; ++i) v[i] = w[i];
        lfft<DIR, M, N, M, P + 1>(v);
    }
}

// ---- global memory --------------------------------------------------------
// One value of N's columns from / to the interleaved (re, im) spectrum.
__device__ __forceinline__ lcx<float2> lload(const float2* p) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    return {make_float2(v.x, v.z), make_float2(v.y, v.w)};
}
__device__ __forceinline__ void lstore(float2* p, lcx<float2> v) {
    *reinterpret_cast<float4*>(p) = make_float4(v.re.x, v.im.x, v.re.y, v.im.y);
}
template <typename N> struct lmem {     // float2: two columns
    static __device__ __forceinline__ lcx<N> load(const float2* p) { return lload(p); }
    static __device__ __forceinline__ void store(float2* p, lcx<N> v) { lstore(p, v); }
};
template <> struct lmem<float> {
    static __device__ __forceinline__ lcx<float> load(const float2* p) { const float2 v = *p; return {v.x, v.y}; }
    static __device__ __forceinline__ void store(float2* p, lcx<float> v) { *p = make_float2(v.re, v.im); }
};
template <> struct lmem<double> {
    static __device__ __forceinline__ lcx<double> load(const double2* p) { const double2 v = *p; return {v.x, v.y}; }
    static __device__ __forceinline__ void store(double2* p, lcx<double> v) { *p = make_double2(v.re, v.im); }
};

// Twiddle table entry for a runtime exponent: (c, s, -s) of exp(-2 pi i q / L)
// with every value repeated over the lanes.  Two 16-byte loads for float2.
template <typename N> struct ltw { N c, s, ms; };
template <typename N> __device__ __forceinline__ ltw<N> ltw_load(const cplx<typename lane<N>::real>* __restrict__ tw, int q);
template <> __device__ __forceinline__ ltw<float2> ltw_load<float2>(const float2* __restrict__ tw, int q) {
    const float2 w = __ldg(tw + q);          // (c, -s)
    return {make_float2(w.x, w.x), make_float2(-w.y, -w.y), make_float2(w.y, w.y)};
}
template <> __device__ __forceinline__ ltw<float> ltw_load<float>(const float2* __restrict__ tw, int q) {
    const float2 w = __ldg(tw + q);
    return {w.x, -w.y, w.y};
}
template <> __device__ __forceinline__ ltw<double> ltw_load<double>(const double2* __restrict__ tw, int q) {
    const double2 w = __ldg(tw + q);
    return {w.x, -w.y, w.y};
}
template <int DIR, typename N> __device__ __forceinline__ lcx<N> lctwr(lcx<N> v, const ltw<N>& w) {
    return lctw<DIR, N>(v, w.c, w.s, w.ms);
}

}  // namespace mm
