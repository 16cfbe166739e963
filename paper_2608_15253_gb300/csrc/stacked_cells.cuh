#pragma once

#include <cuda_runtime.h>

#include "batch_dev.cuh"

namespace mm {

// The field kernel of stacked ensembles without bulk DMI and the further local terms: what every cell
// shares comes with the launch, the absent z neighbours (whose ghosts equal the
// cell) are left out, the slope is Omega x m for Heun too, and the step's
// thermal field is drawn in the predictor and read in the corrector (12 bytes a
// cell against 230 instructions; drawn again where the buffer could not be
// had).  Rows of a multiple of four cells go four cells to a thread, every row
// as one 16-byte access, which keeps more of the 60 to 72 bytes a cell on
// their way.
template <int V> struct rowv { float v[V]; };
template <int V>
__device__ __forceinline__ rowv<V> row_ld(const float* p) {
    rowv<V> r;
    if constexpr (V == 4) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(p));
        r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
    } else {
        r.v[0] = __ldg(p);
    }
    return r;
}
template <int V>
__device__ __forceinline__ rowv<V> row_get(const float* p) {   // shared memory
    rowv<V> r;
    if constexpr (V == 4) {
        const float4 t = *reinterpret_cast<const float4*>(p);
        r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
    } else {
        r.v[0] = *p;
    }
    return r;
}
template <int V>
__device__ __forceinline__ void row_st(float* p, const rowv<V>& r) {
    if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
    else *p = r.v[0];
}

// Cells x .. x + V - 1 of row y of film q; HD_SMEM: their demag field lies at
// hds, components nx apart (else a.hd).
template <int V, int STAGE, bool DM, bool HD_SMEM>
__device__ __forceinline__ void stacked_lean_cells(const StackArgs& a, int q, int x, int y, const float* hds) {
    const int nx = a.nx, ny = a.ny, N = nx * ny, i = y * nx + x;
    const RepDev& rp = a.rep[a.members[q]];
    if (!rp.active) return;              // an idle retire/refill slot keeps its state
    const FieldArgs<float>& fa = a.fa;
    const Region<float>& R = fa.R0;
    const long long off = rp.off, film = (long long)q * 3 * N;
    const float* U = (STAGE == 1 ? a.m0 : a.ms) + off + i;
    rowv<V> M[3], YP[3], YM[3], HD[3], TH[3], O1[3], O2[3];
    float xl[3], xr[3];
    const bool inl = x > 0, inr = x + V < nx, inu = y + 1 < ny, ind = y > 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        M[c] = row_ld<V>(U + c * N);
        YP[c] = row_ld<V>(U + c * N + (inu ? nx : 0));
        YM[c] = row_ld<V>(U + c * N - (ind ? nx : 0));
        xl[c] = __ldg(U + c * N - (inl ? 1 : 0));
        xr[c] = __ldg(U + c * N + (inr ? V : 0));
    }
    if (HD_SMEM || a.hd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) HD[c] = HD_SMEM ? row_get<V>(hds + c * nx) : row_ld<V>(a.hd + film + c * N + i);
    }
    const bool hot = (fa.terms & MM_TERM_THERMAL) && rp.th_scale != 0.f;
    if (hot) {
        if (STAGE == 2 && a.noise) {
#pragma unroll
            for (int c = 0; c < 3; ++c) TH[c] = row_ld<V>(a.noise + film + c * N + i);
        } else {
            const long long step = a.st->step - rp.step0;
            const float sg = R.sigma0 * rp.th_scale;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const U4 w = philox(U4{(uint32_t)(i + v), (uint32_t)step, (uint32_t)((unsigned long long)step >> 32), 0u},
                                    rp.key0, rp.key1);
                float n[3];
                box_muller<float>(w, n);
#pragma unroll
                for (int c = 0; c < 3; ++c) TH[c].v[v] = sg * n[c];
            }
            if (a.noise) {
#pragma unroll
                for (int c = 0; c < 3; ++c) row_st<V>(a.noise + film + c * N + i, TH[c]);
            }
        }
    }
    rowv<V> M0[3], K1[3];
    if (STAGE == 2) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            M0[c] = row_ld<V>(a.m0 + off + c * N + i);
            K1[c] = row_ld<V>(a.k1 + off + c * N + i);
        }
    }
    const float dt = (float)a.st->dt;
    const float cx = fa.ix2 * fa.c_uniform, cy = fa.iy2 * fa.c_uniform;
    const float gx = 0.5f * R.dmi / fa.hx, gy = 0.5f * R.dmi / fa.hy;
    const v3<float> p = mk3<float>(fa.p[0], fa.p[1], fa.p[2]), u = mk3<float>(R.ux, R.uy, R.uz);
    const float base = rp.tq_base * R.inv_Ms;
    auto vec = [](const rowv<V>* r, int v) { return mk3<float>(r[0].v[v], r[1].v[v], r[2].v[v]); };
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const v3<float> m = vec(M, v);
        v3<float> H = mk3<float>(0.f, 0.f, 0.f);
        if (fa.terms & (MM_TERM_EXCHANGE | MM_TERM_DMI)) {
            v3<float> xp = v < V - 1 ? vec(M, v < V - 1 ? v + 1 : v) : mk3<float>(xr[0], xr[1], xr[2]);
            v3<float> xm = v > 0 ? vec(M, v > 0 ? v - 1 : v) : mk3<float>(xl[0], xl[1], xl[2]);
            v3<float> yp = vec(YP, v), ym = vec(YM, v);
            if (v == V - 1 && !inr) xp = ghost_value<float, false>(m, 0, 1, fa.hx, R.ratio, 0.f);
            if (v == 0 && !inl) xm = ghost_value<float, false>(m, 0, -1, fa.hx, R.ratio, 0.f);
            if (!inu) yp = ghost_value<float, false>(m, 1, 1, fa.hy, R.ratio, 0.f);
            if (!ind) ym = ghost_value<float, false>(m, 1, -1, fa.hy, R.ratio, 0.f);
            if (fa.terms & MM_TERM_EXCHANGE) H = cx * ((xp - m) + (xm - m)) + cy * ((yp - m) + (ym - m));
            if (fa.terms & MM_TERM_DMI) {
                const v3<float> dx = gx * (xp - xm), dy = gy * (yp - ym);
                H = H + mk3<float>(dx.z, dy.z, -dx.x - dy.y);
            }
        }
        if (fa.terms & MM_TERM_ANISOTROPY) H = H + (R.ku * dot(m, u)) * u;
        if (fa.terms & MM_TERM_ZEEMAN) H = H + mk3<float>(fa.hext[0], fa.hext[1], fa.hext[2]);
        if (HD_SMEM || a.hd) H = H + vec(HD, v);
        if (hot) H = H + vec(TH, v);
        v3<float> w = R.gm * (H + R.alpha * cross(m, H));
        if (fa.tq == MM_TORQUE_SOT || fa.tq == MM_TORQUE_STT) {
            float hdl, hfl;
            if (fa.tq == MM_TORQUE_SOT) {
                hdl = fa.theta_half * base;
                hfl = fa.fl_ratio * hdl;
            } else {
                hdl = fa.P * fa.L2 / ((fa.L2 + 1.f) + (fa.L2 - 1.f) * dot(m, p)) * base;
                hfl = fa.eps_p * base;
            }
            w = w + (R.gm * (hdl + R.alpha * hfl)) * cross(m, p) + (R.gm * (hfl - R.alpha * hdl)) * p;
        }
        const v3<float> k = DM ? w : cross(w, m);
        v3<float> r;
        if (STAGE == 1) {
            r = DM ? rodrigues<float>(m, k, dt) : m + dt * k;
            O2[0].v[v] = k.x; O2[1].v[v] = k.y; O2[2].v[v] = k.z;
        } else {
            const v3<float> m0 = vec(M0, v), kp = vec(K1, v);
            const v3<float> mn = DM ? rodrigues<float>(m0, 0.5f * (kp + k), dt) : m0 + (0.5f * dt) * (kp + k);
            r = rsqrtf(dot(mn, mn)) * mn;
        }
        O1[0].v[v] = r.x; O1[1].v[v] = r.y; O1[2].v[v] = r.z;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        row_st<V>((STAGE == 1 ? a.ms : a.m0) + off + c * N + i, O1[c]);
        if (STAGE == 1) row_st<V>(a.k1 + off + c * N + i, O2[c]);
    }
}

}  // namespace mm
