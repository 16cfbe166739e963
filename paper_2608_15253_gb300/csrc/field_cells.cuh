// Bodies of the field kernels: one cell of any grid, and V cells of a row of
// one material, with the demag field read from memory or handed in.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"
#include "ctx.h"
#include "field_dev.cuh"

namespace mm {

// Output of one present cell for the launch's mode: H, the slope k (to
// `out` or to the FSAL slot of stage kstage), the Heun / Depondt-Mertens
// predictor (m*, with k or Omega to out2) or corrector (renormalised); the
// step is the attempt's dt_eff (the fixed dt for the fixed-step schemes).
template <typename T>
__device__ __forceinline__ void cell_store(const FieldArgs<T>& a, long long i, const v3<T>& m, const v3<T>& H,
                                           const v3<T>& k) {
    const long long N = a.N;
    if (a.mode == MODE_H) {
        st3(a.out, N, i, H);
    } else if (a.mode == MODE_K) {
        T* o = a.out;
        if (!o) {
            const int kf = a.st->k_first;
            o = a.kptr[a.kstage == 0 ? kf : 6 - kf];
        }
        st3(o, N, i, k);
    } else if (a.mode == MODE_HEUN1) {
        const T dt = (T)a.st->dt_eff;
        st3(a.out2, N, i, k);
        st3(a.out, N, i, m + dt * k);
    } else if (a.mode == MODE_HEUN2) {  // m_new = normalise(m0 + dt/2 (k1 + k2))
        const T dt = (T)a.st->dt_eff;
        const v3<T> m0 = ld3(a.m0, N, i);
        const v3<T> k1 = ld3(a.k1, N, i);
        v3<T> mn = m0 + ((T)0.5 * dt) * (k1 + k);
        const T inv = (T)1 / sqrt(dot(mn, mn));
        st3(a.out, N, i, inv * mn);
    } else if (a.mode == MODE_DM1) {   // Omega_1 and m* = R(Omega_1 dt) m
        const T dt = (T)a.st->dt_eff;
        st3(a.out2, N, i, k);
        st3(a.out, N, i, rodrigues<T>(m, k, dt));
    } else {  // MODE_DM2: m_new = R((Omega_1 + Omega_2) dt / 2) m0
        const T dt = (T)a.st->dt_eff;
        const v3<T> m0 = ld3(a.m0, N, i);
        const v3<T> w1 = ld3(a.k1, N, i);
        const v3<T> mn = rodrigues<T>(m0, (T)0.5 * (w1 + k), dt);
        const T inv = (T)1 / sqrt(dot(mn, mn));
        st3(a.out, N, i, inv * mn);
    }
}

// UNIF: one material (coefficients passed by value in the launch
// parameters, no region map or coefficient-table loads).
template <typename T, bool UNIF, bool EXT>
__device__ __forceinline__ void field_cell(const FieldArgs<T>& a, int x, int y, int z) {
    const long long N = a.N;
    const long long i = ((long long)z * a.ny + y) * a.nx + x;
    const int ri = UNIF ? 0 : (a.region ? a.region[i] : 0);
    const Region<T>& R = UNIF ? a.R0 : a.lut[ri];
    const v3<T> m = ld3(a.m, N, i);
    if (R.present == (T)0) {
        const v3<T> zero = mk3<T>(0, 0, 0);
        T* o = a.out;
        if (!o) {
            const int kf = a.st->k_first;
            o = a.kptr[a.kstage == 0 ? kf : 6 - kf];
        }
        if (a.mode == MODE_HEUN1 || a.mode == MODE_DM1) { st3(o, N, i, zero); st3(a.out2, N, i, zero); }
        else st3(o, N, i, zero);
        return;
    }
    const long long step = a.step_override >= 0 ? a.step_override : (a.st ? a.st->step : 0);
    v3<T> H, k;
    cell_field<T, UNIF, EXT>(a, x, y, z, i, ri, R, m, nullptr, step, H, k, a.mode != MODE_H, a.mode >= MODE_DM1);
    cell_store<T>(a, i, m, H, k);
}

// One material, FP32, nx a multiple of V (2 or 4): each thread owns V
// consecutive cells of a row.  The state, its y/z neighbours, the demag
// field and the outputs move as 8- or 16-byte vectors; the x neighbours of
// the inner cells come from the thread's own registers, only the two
// row-end neighbours are scalar loads.
template <int V> struct fvec;
template <> struct fvec<2> { using t = float2; };
template <> struct fvec<4> { using t = float4; };

template <int V>
__device__ __forceinline__ typename fvec<V>::t ldv(const float* p) {
    return __ldg(reinterpret_cast<const typename fvec<V>::t*>(p));
}
template <int V>
__device__ __forceinline__ void stv(float* p, const typename fvec<V>::t& v) {
    *reinterpret_cast<typename fvec<V>::t*>(p) = v;
}
__device__ __forceinline__ float fget(const float2& v, int q) { return q == 0 ? v.x : v.y; }
__device__ __forceinline__ float fget(const float4& v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }
__device__ __forceinline__ void fset(float2& v, int q, float x) { if (q == 0) v.x = x; else v.y = x; }
__device__ __forceinline__ void fset(float4& v, int q, float x) {
    if (q == 0) v.x = x; else if (q == 1) v.y = x; else if (q == 2) v.z = x; else v.w = x;
}

// The V cells x0 .. x0 + V - 1 of row (z, y).  HD_SMEM: the demag field of
// the cells comes from shared memory (hds[c * hd_stride + q], the fused
// inverse-X-pass kernel below), else from a.Hd in global memory.  QUIET:
// slopes only (MODE_K), no thermal field, no spin torque -- the variant for
// deterministic runs without current, with far fewer registers.
template <int V, bool EXT, bool HD_SMEM, bool QUIET = false>
__device__ __forceinline__ void field_vec_cells(const FieldArgs<float>& a, int x0, int y, int z, const float* hds,
                                                int hd_stride) {
    using VT = typename fvec<V>::t;
    const long long N = a.N;
    const long long i0 = ((long long)z * a.ny + y) * a.nx + x0;
    const Region<float>& R = a.R0;
    const long long step = a.step_override >= 0 ? a.step_override : (a.st ? a.st->step : 0);
    VT mc[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) mc[c] = ldv<V>(a.m + c * N + i0);
    const unsigned nbt = MM_TERM_EXCHANGE | MM_TERM_DMI | (EXT ? MM_TERM_SURFACE : 0u);
    const bool need_nb = (a.terms & nbt) || (!QUIET && a.tq == MM_TORQUE_ZL);
    // neighbour rows (y+, y-, z+, z-) as vectors, row-end x neighbours as scalars
    VT nr[4][3];
    bool rin[4] = {false, false, false, false};
    float xl[3] = {0, 0, 0}, xr[3] = {0, 0, 0};
    bool lin = false, rinx = false;
    if (need_nb) {
        const long long sy = a.nx, sz = (long long)a.nx * a.ny;
        const int ny = a.ny, nz = a.nz;
        const int qs[4] = {y + 1, y - 1, z + 1, z - 1};
        const int dm[4] = {ny, ny, nz, nz};
        const int pr[4] = {a.py, a.py, a.pz, a.pz};
        const int ps[4] = {y, y, z, z};
        const long long st[4] = {sy, sy, sz, sz};
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            int q = qs[s];
            bool inside = q >= 0 && q < dm[s];
            if (!inside && pr[s]) { q = (q + dm[s]) % dm[s]; inside = true; }
            rin[s] = inside;
            if (inside) {
                const long long j = i0 + (long long)(q - ps[s]) * st[s];
#pragma unroll
                for (int c = 0; c < 3; ++c) nr[s][c] = ldv<V>(a.m + c * N + j);
            }
        }
        int ql = x0 - 1, qr = x0 + V;
        lin = ql >= 0;
        rinx = qr < a.nx;
        if (!lin && a.px) { ql += a.nx; lin = true; }
        if (!rinx && a.px) { qr -= a.nx; rinx = true; }
        const long long row = i0 - x0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (lin) xl[c] = __ldg(a.m + c * N + row + ql);
            if (rinx) xr[c] = __ldg(a.m + c * N + row + qr);
        }
    }
    VT hd[3];
    const bool dem = (a.terms & MM_TERM_DEMAG) && (HD_SMEM || a.Hd);
    if (dem) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            hd[c] = HD_SMEM ? *reinterpret_cast<const VT*>(hds + c * hd_stride) : ldv<V>(a.Hd + c * N + i0);
    }
    VT o1[3], o2[3];
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const v3<float> m = mk3<float>(fget(mc[0], q), fget(mc[1], q), fget(mc[2], q));
        v3<float> nbv[6];
        bool nbp[6];
        float cnb[6];
        if (need_nb) {
            // x+ / x-
            const bool pp = q < V - 1 || rinx, pm = q > 0 || lin;
            nbp[0] = pp;
            nbp[1] = pm;
            nbv[0] = q < V - 1 ? mk3<float>(fget(mc[0], q + 1), fget(mc[1], q + 1), fget(mc[2], q + 1))
                               : (rinx ? mk3<float>(xr[0], xr[1], xr[2]) : ghost_value<float, EXT>(m, 0, 1, a.hx, R.ratio, R.ratio_b));
            nbv[1] = q > 0 ? mk3<float>(fget(mc[0], q - 1), fget(mc[1], q - 1), fget(mc[2], q - 1))
                           : (lin ? mk3<float>(xl[0], xl[1], xl[2]) : ghost_value<float, EXT>(m, 0, -1, a.hx, R.ratio, R.ratio_b));
            cnb[0] = pp ? a.c_uniform : R.cg;
            cnb[1] = pm ? a.c_uniform : R.cg;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int slot = 2 + s, d = 1 + s / 2, sg = (s & 1) ? -1 : 1;
                nbp[slot] = rin[s];
                nbv[slot] = rin[s] ? mk3<float>(fget(nr[s][0], q), fget(nr[s][1], q), fget(nr[s][2], q))
                                   : ghost_value<float, EXT>(m, d, sg, d == 1 ? a.hy : a.hz, R.ratio, R.ratio_b);
                cnb[slot] = rin[s] ? a.c_uniform : R.cg;
            }
        }
        const v3<float> hq = dem ? mk3<float>(fget(hd[0], q), fget(hd[1], q), fget(hd[2], q)) : mk3<float>(0, 0, 0);
        v3<float> H, k;
        cell_field_nb<float, EXT, QUIET>(a, i0 + q, R, m, nbv, nbp, cnb, dem, hq, step, H, k,
                                         QUIET || a.mode != MODE_H, !QUIET && a.mode >= MODE_DM1);
        v3<float> r1 = H, r2 = k;
        if (QUIET || a.mode == MODE_K) r1 = k;
        else if (QUIET) {
        } else if (a.mode == MODE_HEUN1) {
            const float dt = (float)a.st->dt_eff;
            r1 = m + dt * k;
            r2 = k;
        } else if (a.mode == MODE_HEUN2) {
            const float dt = (float)a.st->dt_eff;
            const long long i = i0 + q;
            const v3<float> m0 = ld3(a.m0, N, i);
            const v3<float> k1 = ld3(a.k1, N, i);
            v3<float> mn = m0 + (0.5f * dt) * (k1 + k);
            r1 = (1.0f / sqrtf(dot(mn, mn))) * mn;
        } else if (a.mode == MODE_DM1) {
            r1 = rodrigues<float>(m, k, (float)a.st->dt_eff);
            r2 = k;
        } else if (a.mode == MODE_DM2) {
            const long long i = i0 + q;
            const v3<float> m0 = ld3(a.m0, N, i);
            const v3<float> w1 = ld3(a.k1, N, i);
            const v3<float> mn = rodrigues<float>(m0, 0.5f * (w1 + k), (float)a.st->dt_eff);
            r1 = (1.0f / sqrtf(dot(mn, mn))) * mn;
        }
        fset(o1[0], q, r1.x); fset(o1[1], q, r1.y); fset(o1[2], q, r1.z);
        fset(o2[0], q, r2.x); fset(o2[1], q, r2.y); fset(o2[2], q, r2.z);
    }
    float* o = a.out;
    if (!o) {
        const int kf = a.st->k_first;
        o = a.kptr[a.kstage == 0 ? kf : 6 - kf];
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) stv<V>(o + c * N + i0, o1[c]);
    if (!QUIET && (a.mode == MODE_HEUN1 || a.mode == MODE_DM1)) {
#pragma unroll
        for (int c = 0; c < 3; ++c) stv<V>(a.out2 + c * N + i0, o2[c]);
    }
}

}  // namespace mm
