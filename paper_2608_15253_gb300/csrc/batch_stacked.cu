// Replica batching by size class (the "stacked" launch shape): the replicas
// of one grid size are stored back to back, so a stage runs, per class, the
// 2-D demag passes over all of its films at once (demag_apply_stacked2d) and
// then this kernel: field, torque and the Heun or Depondt-Mertens stage
// update of every cell of the class, one thread per cell, each replica with
// its own Philox key, temperature and current.  A few well-filled launches
// per class replace one CTA per replica.  With retire/refill on, idle slots
// are skipped and a per-slot stop test follows the corrector.
#include <cuda_runtime.h>

#include "batch_dev.cuh"

namespace mm {

__global__ void __launch_bounds__(256) stacked_field_kernel(StackArgs a) {
    if (!a.st->active) return;
    const int x = blockIdx.x * 32 + (threadIdx.x & 31);
    const int y = blockIdx.y * 8 + (threadIdx.x >> 5);
    const int q = blockIdx.z;
    const int nx = a.nx, ny = a.ny;
    if (x >= nx || y >= ny) return;
    const RepDev& rp = a.rep[a.members[q]];
    if (!rp.active) return;              // an idle retire/refill slot keeps its state
    const long long N = (long long)nx * ny;
    const long long i = (long long)y * nx + x;
    FieldArgs<float> fa = a.fa;
    fa.N = N;
    fa.nx = nx;
    fa.ny = ny;
    fa.nz = 1;
    fa.key0 = rp.key0;
    fa.key1 = rp.key1;
    fa.th_scale = rp.th_scale;
    fa.tq_base = rp.tq_base;
    const Region<float>& R = fa.lut[0];
    const float* mE = (a.stage == 1 ? a.m0 : a.ms) + rp.off;
    const v3<float> m = ld3(mE, N, i);
    v3<float> nbv[6];
    bool nbp[6];
    float cnb[6];
    const float c_pair = __ldg(fa.cpair);
    const int pos[2] = {x, y}, dim[2] = {nx, ny};
    const long long stride[2] = {1, nx};
    const float hh[2] = {fa.hx, fa.hy};
#pragma unroll
    for (int d = 0; d < 2; ++d) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int sg = s == 0 ? 1 : -1;
            const int qd = pos[d] + sg;
            const int slot = 2 * d + s;
            const bool in = qd >= 0 && qd < dim[d];
            nbp[slot] = in;
            if (in) {
                nbv[slot] = ld3(mE, N, i + sg * stride[d]);
                cnb[slot] = c_pair;
            } else {
                nbv[slot] = ghost_value<float, true>(m, d, sg, hh[d], R.ratio, R.ratio_b);
                cnb[slot] = R.cg;
            }
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        nbp[4 + s] = false;
        nbv[4 + s] = ghost_value<float, true>(m, 2, s == 0 ? 1 : -1, fa.hz, R.ratio, R.ratio_b);
        cnb[4 + s] = R.cg;
    }
    const bool dem = a.hd != nullptr;
    const v3<float> hd = dem ? ld3(a.hd + (long long)q * 3 * N, N, i) : mk3<float>(0.f, 0.f, 0.f);
    const long long step = a.st->step - rp.step0;
    v3<float> H, k;
    cell_field_nb<float, true>(fa, i, R, m, nbv, nbp, cnb, dem, hd, step, H, k, true, a.dm != 0);
    const float dt = (float)a.st->dt;
    if (a.stage == 1) {
        st3(a.k1 + rp.off, N, i, k);
        st3(a.ms + rp.off, N, i, a.dm ? rodrigues<float>(m, k, dt) : m + dt * k);
    } else {
        const v3<float> m0 = ld3(a.m0 + rp.off, N, i);
        const v3<float> kp = ld3(a.k1 + rp.off, N, i);
        const v3<float> mn = a.dm ? rodrigues<float>(m0, 0.5f * (kp + k), dt) : m0 + (0.5f * dt) * (kp + k);
        st3(a.m0 + rp.off, N, i, rsqrtf(dot(mn, mn)) * mn);
    }
}

// The same without bulk DMI and the further local terms: what every cell
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
__device__ __forceinline__ void row_st(float* p, const rowv<V>& r) {
    if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
    else *p = r.v[0];
}

template <int V, int STAGE, bool DM>
__global__ void __launch_bounds__(256) stacked_lean_kernel(StackArgs a) {
    if (!a.st->active) return;
    const int nx = a.nx, ny = a.ny, N = nx * ny, q = blockIdx.z;
    const int i = V * (blockIdx.x * 256 + threadIdx.x);
    if (i >= N) return;
    const int y = i / nx, x = i - y * nx;
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
    if (a.hd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) HD[c] = row_ld<V>(a.hd + film + c * N + i);
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
        if (a.hd) H = H + vec(HD, v);
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

template <int V>
static void stacked_lean_launch(const StackArgs& a, int Rc, cudaStream_t s) {
    const dim3 grid((a.nx * a.ny / V + 255) / 256, 1, Rc);
    if (a.dm) {
        if (a.stage == 1) stacked_lean_kernel<V, 1, true><<<grid, 256, 0, s>>>(a);
        else stacked_lean_kernel<V, 2, true><<<grid, 256, 0, s>>>(a);
    } else {
        if (a.stage == 1) stacked_lean_kernel<V, 1, false><<<grid, 256, 0, s>>>(a);
        else stacked_lean_kernel<V, 2, false><<<grid, 256, 0, s>>>(a);
    }
}

// Retire/refill on the stacked shape (Results, "Replica batching"): after
// the corrector of every class, one CTA per slot forms the mean of m . axis
// over its replica, runs the stop test and, when a new trial takes the
// slot, writes its initial state.
__global__ void __launch_bounds__(256) stacked_trials_kernel(BatchArgs a) {
    if (!a.st->active) return;
    const int idx = blockIdx.x;
    const RepDev rp = a.rep[idx];
    if (!rp.active) return;                           // uniform over the CTA
    const long long N = (long long)rp.nx * rp.ny;
    const float* m = a.m0 + rp.off;
    const float ax = a.tr.axis[0], ay = a.tr.axis[1], az = a.tr.axis[2];
    float part = 0.f;
    for (long long i = threadIdx.x; i < N; i += 256) part += m[i] * ax + m[N + i] * ay + m[2 * N + i] * az;
    slot_retire_refill<256>(a, rp, idx, part, N, a.st->step);
}

void stacked_trials_launch(const BatchArgs& a, int R, cudaStream_t s) {
    stacked_trials_kernel<<<R, 256, 0, s>>>(a);
}

void stacked_field_launch(const StackArgs& a, int Rc, cudaStream_t s) {
    dim3 grid((a.nx + 31) / 32, (a.ny + 7) / 8, Rc);
    if (a.ext) stacked_field_kernel<<<grid, 256, 0, s>>>(a);
    else if (a.nx % 4 == 0) stacked_lean_launch<4>(a, Rc, s);   // (every film and class then starts on 16 bytes)
    else stacked_lean_launch<1>(a, Rc, s);
}

}  // namespace mm
