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
    return *reinterpret_cast<const typename fvec<V>::t*>(p);
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

// What V cells x0 .. x0 + V - 1 of row (z, y) need of the state: themselves and
// their neighbours.  Read on its own, so that the fused kernel's idle threads can
// do it ahead of the barrier that brings the demag field: plain loads are not
// moved across it.
template <int V>
struct VecIn {
    using VT = typename fvec<V>::t;
    VT m[3], nr[4][3];              // the cells; the neighbour rows y+, y-, z+, z-
    float xl[3], xr[3];             // the two row-end x neighbours
    bool rin[4], lin, rinx;
};

template <int V, bool EXT, bool QUIET>
__device__ __forceinline__ void field_vec_load(const FieldArgs<float>& a, int x0, int y, int z, VecIn<V>& in) {
    const long long N = a.N;
    const long long i0 = ((long long)z * a.ny + y) * a.nx + x0;
#pragma unroll
    for (int c = 0; c < 3; ++c) in.m[c] = ldv<V>(a.m + c * N + i0);
    const unsigned nbt = MM_TERM_EXCHANGE | MM_TERM_DMI | (EXT ? MM_TERM_SURFACE : 0u);
    in.lin = in.rinx = false;
#pragma unroll
    for (int s = 0; s < 4; ++s) in.rin[s] = false;
    if ((a.terms & nbt) || (!QUIET && a.tq == MM_TORQUE_ZL)) {
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
            in.rin[s] = inside;
            if (inside) {
                const long long j = i0 + (long long)(q - ps[s]) * st[s];
#pragma unroll
                for (int c = 0; c < 3; ++c) in.nr[s][c] = ldv<V>(a.m + c * N + j);
            }
        }
        int ql = x0 - 1, qr = x0 + V;
        in.lin = ql >= 0;
        in.rinx = qr < a.nx;
        if (!in.lin && a.px) { ql += a.nx; in.lin = true; }
        if (!in.rinx && a.px) { qr -= a.nx; in.rinx = true; }
        const long long row = i0 - x0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (in.lin) in.xl[c] = a.m[c * N + row + ql];
            if (in.rinx) in.xr[c] = a.m[c * N + row + qr];
        }
    }
}

// The output of these cells.  HD_SMEM: their demag field comes from shared
// memory (hds[c * hd_stride + q], the fused inverse-X-pass kernel), else from
// a.Hd in global memory.  QUIET: slopes only (MODE_K), no thermal field, no spin
// torque -- the variant for deterministic runs without current, with far fewer
// registers.  What a mode reads and writes beside the slope is done for all cells
// together: a cell at a time, a corrector's loads wait for the store of the other
// cell's thermal field, and a small grid for its instructions.  512x512x32 Heun
// without demag 291 -> 272 us a step, at 300 K 386 -> 336; with demag 1755 -> 1692;
// 256x256 films 36.3 -> 36.7 (the price of plain loads there, 37.8 without this).
template <int V, bool EXT, bool HD_SMEM, bool QUIET>
__device__ __forceinline__ void field_vec_finish(const FieldArgs<float>& a, int x0, int y, int z, const VecIn<V>& in,
                                                 const float* hds, int hd_stride) {
    using VT = typename fvec<V>::t;
    const long long N = a.N;
    const long long i0 = ((long long)z * a.ny + y) * a.nx + x0;
    const Region<float>& R = a.R0;
    const unsigned nbt = MM_TERM_EXCHANGE | MM_TERM_DMI | (EXT ? MM_TERM_SURFACE : 0u);
    const bool need_nb = (a.terms & nbt) || (!QUIET && a.tq == MM_TORQUE_ZL);
    VT th[3];
    if (!QUIET && (a.terms & MM_TERM_THERMAL) && a.th_scale != 0.f) {
        if (a.noise && (a.mode == MODE_HEUN2 || a.mode == MODE_DM2)) {
#pragma unroll
            for (int c = 0; c < 3; ++c) th[c] = ldv<V>(a.noise + c * N + i0);
        } else {
            const long long step = a.step_override >= 0 ? a.step_override : (a.st ? a.st->step : 0);
#pragma unroll
            for (int q = 0; q < V; ++q) {
                const v3<float> t = thermal_h<float>(a, i0 + q, a.R0, step);
                fset(th[0], q, t.x); fset(th[1], q, t.y); fset(th[2], q, t.z);
            }
            if (a.noise) {
#pragma unroll
                for (int c = 0; c < 3; ++c) stv<V>(a.noise + c * N + i0, th[c]);
            }
        }
    }
    VT hd[3];
    const bool dem = (a.terms & MM_TERM_DEMAG) && (HD_SMEM || a.Hd);
    if (dem) {
#pragma unroll
        for (int c = 0; c < 3; ++c)
            hd[c] = HD_SMEM ? *reinterpret_cast<const VT*>(hds + c * hd_stride) : ldv<V>(a.Hd + c * N + i0);
    }
    auto get = [](const VT* v, int q) { return mk3<float>(fget(v[0], q), fget(v[1], q), fget(v[2], q)); };
    VT o1[3], o2[3];
    auto put = [&](int q, const v3<float>& r) { fset(o1[0], q, r.x); fset(o1[1], q, r.y); fset(o1[2], q, r.z); };
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const v3<float> m = get(in.m, q);
        v3<float> nbv[6];
        bool nbp[6];
        float cnb[6];
        if (need_nb) {
            // x+ / x-
            const bool pp = q < V - 1 || in.rinx, pm = q > 0 || in.lin;
            nbp[0] = pp;
            nbp[1] = pm;
            nbv[0] = q < V - 1 ? get(in.m, q < V - 1 ? q + 1 : q)
                               : (in.rinx ? mk3<float>(in.xr[0], in.xr[1], in.xr[2]) : ghost_value<float, EXT>(m, 0, 1, a.hx, R.ratio, R.ratio_b));
            nbv[1] = q > 0 ? get(in.m, q > 0 ? q - 1 : q)
                           : (in.lin ? mk3<float>(in.xl[0], in.xl[1], in.xl[2]) : ghost_value<float, EXT>(m, 0, -1, a.hx, R.ratio, R.ratio_b));
            cnb[0] = pp ? a.c_uniform : R.cg;
            cnb[1] = pm ? a.c_uniform : R.cg;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const int slot = 2 + s, d = 1 + s / 2, sg = (s & 1) ? -1 : 1;
                nbp[slot] = in.rin[s];
                nbv[slot] = in.rin[s] ? get(in.nr[s], q)
                                      : ghost_value<float, EXT>(m, d, sg, d == 1 ? a.hy : a.hz, R.ratio, R.ratio_b);
                cnb[slot] = in.rin[s] ? a.c_uniform : R.cg;
            }
        }
        const v3<float> hq = dem ? get(hd, q) : mk3<float>(0, 0, 0), thq = get(th, q);
        v3<float> H, k;
        cell_field_nb<float, EXT, QUIET>(a, i0 + q, R, m, nbv, nbp, cnb, dem, hq, 0, H, k, QUIET || HD_SMEM || a.mode != MODE_H,
                                         !QUIET && a.mode >= MODE_DM1, &thq);
        put(q, QUIET ? k : H);
        if (!QUIET) { fset(o2[0], q, k.x); fset(o2[1], q, k.y); fset(o2[2], q, k.z); }
    }
    // the stage's output of all cells, the mode looked up once
    if (QUIET) {
    } else if (a.mode == MODE_K) {
#pragma unroll
        for (int c = 0; c < 3; ++c) o1[c] = o2[c];
    } else if (HD_SMEM || a.mode != MODE_H) {
        const float dt = (float)a.st->dt_eff;
        if (a.mode == MODE_HEUN1) {
#pragma unroll
            for (int q = 0; q < V; ++q) put(q, get(in.m, q) + dt * get(o2, q));
        } else if (a.mode == MODE_DM1) {
#pragma unroll
            for (int q = 0; q < V; ++q) put(q, rodrigues<float>(get(in.m, q), get(o2, q), dt));
        } else {
            VT b0[3], b1[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                b0[c] = ldv<V>(a.m0 + c * N + i0);
                b1[c] = ldv<V>(a.k1 + c * N + i0);
            }
#pragma unroll
            for (int q = 0; q < V; ++q) {
                const v3<float> m0 = get(b0, q), kk = get(b1, q) + get(o2, q);
                const v3<float> mn = a.mode == MODE_HEUN2 ? m0 + (0.5f * dt) * kk : rodrigues<float>(m0, 0.5f * kk, dt);
                put(q, (1.0f / sqrtf(dot(mn, mn))) * mn);
            }
        }
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
