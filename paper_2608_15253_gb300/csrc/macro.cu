// Replica-batched blocks of fused steps for replicas without demag (Results,
// "Replica batching": the single-cell ensemble with local fields, spin
// torque and thermal noise, the thermally assisted switching sweep, and
// the small exchange-coupled films of the batching table).  A one-cell
// replica's step is local: one thread per slot holds the moment in
// registers for a block of steps and runs the predictor, the corrector and,
// with retire/refill on, the stop test and the start of the next trial,
// without leaving the thread.  A small film is one CTA with its state in
// shared memory (tile_kernel).
#include <cuda_runtime.h>

#include "batch_dev.cuh"

namespace mm {

__global__ void __launch_bounds__(32) macro_kernel(MacroArgs a) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= a.R) return;
    RepDev rp = a.rep[r];
    if (!rp.active) return;
    FieldArgs<float> fa = a.fa;
    fa.N = 1;
    fa.nx = fa.ny = fa.nz = 1;
    fa.m = a.m + rp.off;            // never read: every neighbour is absent
    fa.key0 = rp.key0;
    fa.key1 = rp.key1;
    fa.th_scale = rp.th_scale;
    fa.tq_base = rp.tq_base;
    const Region<float>& R = fa.lut[0];
    // the step's thermal draw is the same in both evaluations: drawn once
    // per step and added through the precomputed-field slot
    const bool hot = (fa.terms & MM_TERM_THERMAL) != 0;
    fa.terms = (fa.terms & ~MM_TERM_THERMAL) | MM_TERM_DEMAG;
    const float dt = (float)a.st->dt;
    const long long step0 = a.st->step;
    const bool dm = a.dm != 0;
    const v3<float> ax = mk3<float>(a.tr.axis[0], a.tr.axis[1], a.tr.axis[2]);
    float* mp = a.m + rp.off;
    v3<float> m = mk3<float>(mp[0], mp[1], mp[2]);
    const v3<float> zero = mk3<float>(0.f, 0.f, 0.f);
    // the draws do not depend on the state: the next step's is computed one
    // step ahead, so its Philox rounds overlap this step's dependent chain
    v3<float> hnext = hot && fa.th_scale != 0.f ? thermal_h<float>(fa, 0, R, step0 - rp.step0) : zero;
    for (int s = 0; s < a.nsteps; ++s) {
        const long long step = step0 + s;
        const long long ctr = step - rp.step0;    // the trial's own step: its noise counter
        v3<float> H, w1, w2;
        const v3<float> hth = hnext;
        if (hot && fa.th_scale != 0.f) hnext = thermal_h<float>(fa, 0, R, ctr + 1);
        cell_field<float, false, true>(fa, 0, 0, 0, 0, 0, R, m, &hth, ctr, H, w1, true, dm);
        const v3<float> ms = dm ? rodrigues<float>(m, w1, dt) : m + dt * w1;
        cell_field<float, false, true>(fa, 0, 0, 0, 0, 0, R, ms, &hth, ctr, H, w2, true, dm);
        const v3<float> mn = dm ? rodrigues<float>(m, 0.5f * (w1 + w2), dt) : m + (0.5f * dt) * (w1 + w2);
        m = rsqrtf(dot(mn, mn)) * mn;
        if (a.trials) {
            if (trial_check(a.tr, rp, a.rep + r, dot(m, ax), step + 1 - rp.step0, step + 1)) {
                m = mk3<float>(__ldg(a.tr.m_init), __ldg(a.tr.m_init + 1), __ldg(a.tr.m_init + 2));
                fa.key0 = rp.key0;
                fa.key1 = rp.key1;
                fa.th_scale = rp.th_scale;
                fa.tq_base = rp.tq_base;
                hnext = hot && fa.th_scale != 0.f ? thermal_h<float>(fa, 0, R, 0) : zero;
            }
            if (!rp.active) break;
        }
    }
    mp[0] = m.x;
    mp[1] = m.y;
    mp[2] = m.z;
}

// The same without bulk DMI and the further local terms,
// written out for one cell: every neighbour is absent, so the ghosts cancel in
// the exchange term and leave D/(2A) times the DMI coefficient (m_x, m_y, 2
// m_z) in the interfacial one, and what does not depend on m is formed once.
// The slope is Omega x m for Heun too.  Bound by the chain of dependent
// operations of a step.  1024 replicas, 1024 Depondt-Mertens steps at 300 K
// under spin-orbit torque, one GB300: 0.35 ms; 0.78 with each thread drawing
// its own thermal field (in the shadow of the chain, but in order with it),
// 2.62 with the general field function and angle functions as well.
struct MacroCell {
    v3<float> h0, u, p;         // applied field, anisotropy axis, polarisation
    float ku, dmi, alpha, gm;
    float cdl, cfl;             // gamma' mu0 times the damping- and field-like parts (SOT)
    float base, P, L2, eps_p;   // STT
    int tq;
};

__device__ __forceinline__ void macro_current(MacroCell& c, const FieldArgs<float>& fa, const Region<float>& R, float tq_base) {
    c.base = tq_base * R.inv_Ms;
    const float hdl = fa.theta_half * c.base, hfl = fa.fl_ratio * hdl;
    c.cdl = R.gm * (hdl + R.alpha * hfl);
    c.cfl = R.gm * (hfl - R.alpha * hdl);
}

__device__ __forceinline__ v3<float> macro_omega(const MacroCell& c, const v3<float>& m, const v3<float>& th) {
    v3<float> H = c.h0 + th;
    H = H + (c.ku * dot(m, c.u)) * c.u;
    H = H + c.dmi * mk3<float>(m.x, m.y, 2.f * m.z);
    v3<float> w = c.gm * (H + c.alpha * cross(m, H));
    if (c.tq == MM_TORQUE_SOT) {
        w = w + c.cdl * cross(m, c.p) + c.cfl * c.p;
    } else if (c.tq == MM_TORQUE_STT) {
        const float eps = c.P * c.L2 / ((c.L2 + 1.f) + (c.L2 - 1.f) * dot(m, c.p));
        const float hdl = eps * c.base, hfl = c.eps_p * c.base;
        w = w + (c.gm * (hdl + c.alpha * hfl)) * cross(m, c.p) + (c.gm * (hfl - c.alpha * hdl)) * c.p;
    }
    return w;
}

__device__ __forceinline__ MacroCell macro_cell(const FieldArgs<float>& fa, const Region<float>& R, float tq_base) {
    const unsigned terms = fa.terms;
    MacroCell c;
    c.h0 = (terms & MM_TERM_ZEEMAN) ? mk3<float>(fa.hext[0], fa.hext[1], fa.hext[2]) : mk3<float>(0.f, 0.f, 0.f);
    c.u = mk3<float>(R.ux, R.uy, R.uz);
    c.p = mk3<float>(fa.p[0], fa.p[1], fa.p[2]);
    c.ku = (terms & MM_TERM_ANISOTROPY) ? R.ku : 0.f;
    c.dmi = (terms & MM_TERM_DMI) ? R.dmi * R.ratio : 0.f;
    c.alpha = R.alpha;
    c.gm = R.gm;
    c.P = fa.P;
    c.L2 = fa.L2;
    c.eps_p = fa.eps_p;
    c.tq = fa.tq;
    macro_current(c, fa, R, tq_base);
    return c;
}

__device__ __forceinline__ v3<float> macro_step(const MacroCell& c, const v3<float>& m, const v3<float>& th, float dt, bool dm) {
    const v3<float> w1 = macro_omega(c, m, th);
    v3<float> mn;
    if (dm) {
        const v3<float> w2 = macro_omega(c, rodrigues<float>(m, w1, dt), th);
        mn = rodrigues<float>(m, 0.5f * (w1 + w2), dt);
    } else {
        const v3<float> k1 = cross(w1, m);
        const v3<float> ms = m + dt * k1;
        const v3<float> k2 = cross(macro_omega(c, ms, th), ms);
        mn = m + (0.5f * dt) * (k1 + k2);
    }
    return rsqrtf(dot(mn, mn)) * mn;
}

// Retire/refill: a slot's noise stream changes when its trial does, so the
// thread draws for itself, one step ahead.
__global__ void __launch_bounds__(32) macro_trials_kernel(MacroArgs a) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= a.R) return;
    RepDev rp = a.rep[r];
    if (!rp.active) return;
    FieldArgs<float> fa = a.fa;
    fa.key0 = rp.key0;
    fa.key1 = rp.key1;
    fa.th_scale = rp.th_scale;
    const Region<float>& R = fa.lut[0];
    MacroCell c = macro_cell(fa, R, rp.tq_base);
    const v3<float> zero = mk3<float>(0.f, 0.f, 0.f);
    const float dt = (float)a.st->dt;
    const long long step0 = a.st->step;
    const bool dm = a.dm != 0, hot = (fa.terms & MM_TERM_THERMAL) != 0;
    const v3<float> ax = mk3<float>(a.tr.axis[0], a.tr.axis[1], a.tr.axis[2]);
    float* mp = a.m + rp.off;
    v3<float> m = mk3<float>(mp[0], mp[1], mp[2]);
    v3<float> hnext = hot && fa.th_scale != 0.f ? thermal_h<float>(fa, 0, R, step0 - rp.step0) : zero;
    for (int s = 0; s < a.nsteps; ++s) {
        const long long step = step0 + s;
        const v3<float> hth = hnext;
        if (hot && fa.th_scale != 0.f) hnext = thermal_h<float>(fa, 0, R, step - rp.step0 + 1);
        m = macro_step(c, m, hth, dt, dm);
        if (trial_check(a.tr, rp, a.rep + r, dot(m, ax), step + 1 - rp.step0, step + 1)) {
            m = mk3<float>(__ldg(a.tr.m_init), __ldg(a.tr.m_init + 1), __ldg(a.tr.m_init + 2));
            fa.key0 = rp.key0;
            fa.key1 = rp.key1;
            fa.th_scale = rp.th_scale;
            macro_current(c, fa, R, rp.tq_base);
            hnext = hot && fa.th_scale != 0.f ? thermal_h<float>(fa, 0, R, 0) : zero;
        }
        if (!rp.active) break;
    }
    mp[0] = m.x;
    mp[1] = m.y;
    mp[2] = m.z;
}

// Without trials the draws are known for every step: warp 0 of a CTA steps 32
// replicas, its other warps draw the thermal fields of the next kDraws steps
// into the other half of a buffer, a barrier per kDraws steps between them.
constexpr int kDraws = 12, kDrawWarps = 3;

__global__ void __launch_bounds__(32 * (1 + kDrawWarps)) macro_lean_kernel(MacroArgs a) {
    __shared__ float s_h[2][kDraws][3][32];
    const int lane_id = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int r = blockIdx.x * 32 + lane_id;
    const RepDev rp = a.rep[r < a.R ? r : 0];
    const bool on = r < a.R && rp.active;
    FieldArgs<float> fa = a.fa;
    fa.key0 = rp.key0;
    fa.key1 = rp.key1;
    fa.th_scale = rp.th_scale;
    const Region<float>& R = fa.lut[0];
    const long long ctr0 = a.st->step - rp.step0;
    const bool hot = (fa.terms & MM_TERM_THERMAL) != 0 && fa.th_scale != 0.f;
    auto draw = [&](int blk) {                                    // steps blk kDraws ... of the buffer's half
        for (int s = warp - 1; s < kDraws; s += kDrawWarps) {
            const v3<float> h = hot ? thermal_h<float>(fa, 0, R, ctr0 + (long long)blk * kDraws + s) : mk3<float>(0.f, 0.f, 0.f);
            float* d = &s_h[blk & 1][s][0][lane_id];
            d[0] = h.x;
            d[32] = h.y;
            d[64] = h.z;
        }
    };
    const int nblk = (a.nsteps + kDraws - 1) / kDraws;
    if (warp > 0) {
        draw(0);
        for (int b = 0; b < nblk; ++b) {
            __syncthreads();
            if (b + 1 < nblk) draw(b + 1);
        }
        return;
    }
    const MacroCell c = macro_cell(fa, R, rp.tq_base);
    const float dt = (float)a.st->dt;
    const bool dm = a.dm != 0;
    float* mp = a.m + rp.off;
    v3<float> m = mk3<float>(mp[0], mp[1], mp[2]);
    for (int b = 0; b < nblk; ++b) {
        __syncthreads();
        const int n = min(kDraws, a.nsteps - b * kDraws);
        for (int s = 0; s < n; ++s) {
            const float* d = &s_h[b & 1][s][0][lane_id];
            m = macro_step(c, m, mk3<float>(d[0], d[32], d[64]), dt, dm);
        }
    }
    if (on) {
        mp[0] = m.x;
        mp[1] = m.y;
        mp[2] = m.z;
    }
}

// One film replica (nz = 1, no demag, at most 1024 cells) per CTA, one cell
// per thread: the state lives in shared memory buffer A, the predictor in
// buffer B, each thread's own m and Omega_1 (or slope k1) in registers.  Per
// step: predictor from A's neighbours -> B, barrier, corrector from B's
// neighbours -> A, (retire/refill: block reduction and the stop test),
// barrier.  Neighbours come from shared memory, ghosts where the film ends.
template <bool EXT>
__global__ void __launch_bounds__(kTileMaxCells) tile_kernel(MacroArgs a) {
    extern __shared__ float tsm[];
    __shared__ float s_red[kTileMaxCells / 32];
    __shared__ int s_new;
    RepDev rp = a.rep[blockIdx.x];
    if (!rp.active) return;   // uniform across the CTA
    const int nx = rp.nx, ny = rp.ny, N = nx * ny;
    float* A = tsm;
    float* B = tsm + 3 * a.nmax;
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
    const float c_pair = __ldg(fa.cpair);
    const int i = threadIdx.x;
    const bool own = i < N;
    const int x = own ? i % nx : 0, y = own ? i / nx : 0;
    const float dt = (float)a.st->dt;
    const long long step0 = a.st->step;
    const bool dm = a.dm != 0;
    const v3<float> ax = mk3<float>(a.tr.axis[0], a.tr.axis[1], a.tr.axis[2]);
    float* mg = a.m + rp.off;
    v3<float> m = own ? mk3<float>(mg[i], mg[N + i], mg[2 * N + i]) : mk3<float>(0.f, 0.f, 0.f);
    if (own) { A[i] = m.x; A[N + i] = m.y; A[2 * N + i] = m.z; }
    __syncthreads();
    // neighbour values of cell i from buffer S (ghosts outside the film)
    auto gather = [&](const float* S, const v3<float>& mc, v3<float>* nbv, bool* nbp, float* cnb) {
        const int pos[2] = {x, y}, dim[2] = {nx, ny}, stride[2] = {1, nx};
        const float hh[2] = {fa.hx, fa.hy};
#pragma unroll
        for (int d = 0; d < 2; ++d) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int sg = s == 0 ? 1 : -1;
                const int q = pos[d] + sg;
                const int slot = 2 * d + s;
                const bool in = q >= 0 && q < dim[d];
                nbp[slot] = in;
                if (in) {
                    const int j = i + sg * stride[d];
                    nbv[slot] = mk3<float>(S[j], S[N + j], S[2 * N + j]);
                    cnb[slot] = c_pair;
                } else {
                    nbv[slot] = ghost_value<float, EXT>(mc, d, sg, hh[d], R.ratio, R.ratio_b);
                    cnb[slot] = R.cg;
                }
            }
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            nbp[4 + s] = false;
            nbv[4 + s] = ghost_value<float, EXT>(mc, 2, s == 0 ? 1 : -1, fa.hz, R.ratio, R.ratio_b);
            cnb[4 + s] = R.cg;
        }
    };
    const v3<float> zero = mk3<float>(0.f, 0.f, 0.f);
    for (int s = 0; s < a.nsteps; ++s) {
        const long long step = step0 + s;
        const long long ctr = step - rp.step0;
        v3<float> w1 = zero, H;
        if (own) {
            v3<float> nbv[6];
            bool nbp[6];
            float cnb[6];
            gather(A, m, nbv, nbp, cnb);
            cell_field_nb<float, EXT>(fa, i, R, m, nbv, nbp, cnb, false, zero, ctr, H, w1, true, dm);
            const v3<float> ms = dm ? rodrigues<float>(m, w1, dt) : m + dt * w1;
            B[i] = ms.x; B[N + i] = ms.y; B[2 * N + i] = ms.z;
        }
        __syncthreads();
        float proj = 0.f;
        if (own) {
            const v3<float> ms = mk3<float>(B[i], B[N + i], B[2 * N + i]);
            v3<float> nbv[6];
            bool nbp[6];
            float cnb[6];
            gather(B, ms, nbv, nbp, cnb);
            v3<float> w2;
            cell_field_nb<float, EXT>(fa, i, R, ms, nbv, nbp, cnb, false, zero, ctr, H, w2, true, dm);
            const v3<float> mn = dm ? rodrigues<float>(m, 0.5f * (w1 + w2), dt) : m + (0.5f * dt) * (w1 + w2);
            m = rsqrtf(dot(mn, mn)) * mn;
            A[i] = m.x; A[N + i] = m.y; A[2 * N + i] = m.z;
            proj = dot(m, ax);
        }
        if (a.trials) {
            for (int o = 16; o > 0; o >>= 1) proj += __shfl_xor_sync(0xffffffffu, proj, o);
            if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = proj;
            __syncthreads();
            if (threadIdx.x == 0) {
                float tot = 0.f;
                for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += s_red[w];
                s_new = trial_check(a.tr, rp, a.rep + blockIdx.x, tot / (float)N, step + 1 - rp.step0, step + 1);
                s_red[0] = rp.active ? 1.f : 0.f;
            }
            __syncthreads();
            const int refill = s_new;
            const bool alive = s_red[0] != 0.f;
            if (refill) {
                rp = a.rep[blockIdx.x];   // the new trial's key, scales and start step
                fa.key0 = rp.key0;
                fa.key1 = rp.key1;
                fa.th_scale = rp.th_scale;
                fa.tq_base = rp.tq_base;
                if (own) {
                    m = mk3<float>(__ldg(a.tr.m_init + i), __ldg(a.tr.m_init + N + i), __ldg(a.tr.m_init + 2 * N + i));
                    A[i] = m.x; A[N + i] = m.y; A[2 * N + i] = m.z;
                }
            }
            __syncthreads();
            if (!alive) break;
        } else {
            __syncthreads();
        }
    }
    if (own) { mg[i] = m.x; mg[N + i] = m.y; mg[2 * N + i] = m.z; }
}

cudaError_t tile_kernel_attributes() {
    cudaError_t e = cudaFuncSetAttribute(tile_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(6 * kTileMaxCells * sizeof(float)));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(tile_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(6 * kTileMaxCells * sizeof(float)));
}

void tile_kernel_launch(const MacroArgs& a, cudaStream_t s) {
    const int nt = (a.nmax + 31) / 32 * 32;
    if (a.ext) tile_kernel<true><<<a.R, nt, 6 * a.nmax * sizeof(float), s>>>(a);
    else tile_kernel<false><<<a.R, nt, 6 * a.nmax * sizeof(float), s>>>(a);
}

// fixed-step bookkeeping of a block of n steps, to the time t where it is given
__global__ void macro_advance_kernel(DevState* st, int n, bool given, double t) {
    if (given) st->t = t;
    else st->t += n * st->dt;
    st->step += n;
    st->accepted += n;
    st->attempts += n;
}

void macro_kernel_launch(const MacroArgs& a, cudaStream_t s) {
    const int nt = 32;
    if (a.ext) macro_kernel<<<(a.R + nt - 1) / nt, nt, 0, s>>>(a);
    else if (a.trials) macro_trials_kernel<<<(a.R + nt - 1) / nt, nt, 0, s>>>(a);
    else macro_lean_kernel<<<(a.R + nt - 1) / nt, nt * (1 + kDrawWarps), 0, s>>>(a);
}

void macro_advance_launch(DevState* st, int nsteps, const double* t, cudaStream_t s) {
    macro_advance_kernel<<<1, 1, 0, s>>>(st, nsteps, t != nullptr, t ? *t : 0.0);
}

}  // namespace mm
