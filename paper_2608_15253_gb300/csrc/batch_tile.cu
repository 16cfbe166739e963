// Ensembles of small films with demag (Results, "Replica batching"; the
// 16x16 row of the batching table): one CTA per film runs a block of Heun or
// Depondt-Mertens steps without leaving the SM.  The state, the predictor and
// the spectrum stay in shared memory; per evaluation
//   X   rows of Ms m -> half spectra in place (lane_x.cuh's split),
//   Y   columns: forward FFT, H^ = K^ M^, inverse (conv_lane.cuh's split),
//   X   half spectra -> the demag field's rows in place,
//   F   field, torque and stage update of the thread's cells,
// with a CTA barrier between.  The step's thermal draw is made once and kept
// in registers for both evaluations.  The stacked shape spends five launches of
// 5 to 10 us on each evaluation of 256 films of 16x16, at a fifth of the chip's
// warps; here an evaluation is six barriers: 64 Depondt-Mertens steps of those
// films 4.7 -> 0.68 ms on one GB300 (10.6 us a step, bound by the chain of
// phases in a CTA; 288 threads, which would take every phase in one round,
// spill: 0.81 ms).
//
// Taken for every ensemble of one such size, whatever their number: against the
// class passes of this library, us a Depondt-Mertens step at 300 K,
//   films          64            256           1024          8192
//   8x8        5.9 / 110     6.1 / 205    10.5 / 594     57 / 4132
//   12x12     11.6 / 117    12.4 / 256    28.8 / 827    189 / 6027
//   16x16      8.3 / 57     10.8 / 67     36.4 / 89     261 / 338
//   24x24     13.5 / 58     25.3 / 72     87.0 / 131    673 / 721
//   32x32     15.4 / 59     29.3 / 80      102 / 162    779 / 973
// (two to eight of the smaller films share an SM, one of 24x24 or 32x32).
#include <cuda_runtime.h>

#include <algorithm>

#include "batch_dev.cuh"
#include "conv_lane.cuh"
#include "lane_x.cuh"

namespace mm {

// Row pitch of the spectrum (complex): a row's exchange line fits in its place.
template <int M, int G, int Q>
__host__ __device__ constexpr int tile_pitch() {
    return XSplit<M, G, Q>::LINE > M + 1 ? XSplit<M, G, Q>::LINE : M + 1;
}
template <int M, int G1, int Q1, int L, int G2, int Q2>
constexpr size_t tile_demag_smem() {
    constexpr size_t ny = (L + 1) / 2;
    return 3 * ny * tile_pitch<M, G1, Q1>() * sizeof(float2) + (size_t)3 * L * (M + 1) * sizeof(float2) +
           2 * 3 * ny * M * sizeof(float);
}

struct TileDemagArgs {
    MacroArgs a;
    const ClsDev* cls;      // the one size class
};

template <int M, int G1, int Q1, int L, int G2, int Q2, int NT, int MINB, bool EXT>
__global__ void __launch_bounds__(NT, MINB) tile_demag_kernel(TileDemagArgs ta) {
    using XS = XSplit<M, G1, Q1>;
    static_assert(XS::WARP && L == G2 * Q2, "rows within warps");
    constexpr int NY = (L + 1) / 2, KP = tile_pitch<M, G1, Q1>(), KX = M + 1, KZ = L / 2 + 1;
    constexpr int QIN = lane_qin<L>(G2);
    constexpr int CPT = (M * NY + NT - 1) / NT;                   // cells per thread
    extern __shared__ __align__(16) unsigned char smem_raw[];
    lcx<float>* S = reinterpret_cast<lcx<float>*>(smem_raw);      // [3][ny][KP]
    lcx<float>* E = S + 3 * NY * KP;                              // [3][G2][Q2][KX]
    float* A = reinterpret_cast<float*>(E + 3 * L * KX);
    __shared__ float s_red[NT / 32];
    __shared__ int s_new;
    const MacroArgs& a = ta.a;
    RepDev rp = a.rep[blockIdx.x];
    if (!rp.active) return;                                       // uniform across the CTA
    const ClsDev& cd = *ta.cls;
    const int nx = rp.nx, ny = rp.ny, N = nx * ny, Wk = cd.Wk;
    float* B = A + 3 * N;
    FieldArgs<float> fa = a.fa;
    fa.N = N;
    fa.nx = nx;
    fa.ny = ny;
    fa.nz = 1;
    fa.key0 = rp.key0;
    fa.key1 = rp.key1;
    fa.th_scale = rp.th_scale;
    fa.tq_base = rp.tq_base;
    const bool hot = (fa.terms & MM_TERM_THERMAL) != 0;
    fa.terms = (fa.terms & ~MM_TERM_THERMAL) | MM_TERM_DEMAG;     // the draw rides with the demag field
    const Region<float>& R = fa.lut[0];
    const float c_pair = __ldg(fa.cpair), Ms = R.Ms;
    const int tid = threadIdx.x;
    const float dt = (float)a.st->dt;
    const long long step0 = a.st->step;
    const bool dm = a.dm != 0;
    const v3<float> ax = mk3<float>(a.tr.axis[0], a.tr.axis[1], a.tr.axis[2]);
    const v3<float> zero = mk3<float>(0.f, 0.f, 0.f);
    float* mg = a.m + rp.off;
    for (int e = tid; e < 3 * N; e += NT) A[e] = mg[e];
    __syncthreads();

    // demag field of state U into the rows of S: component c, row y at hrow(c, y)[x]
    auto hrow = [&](int c, int y) { return reinterpret_cast<float*>(S + (c * ny + y) * KP); };
    auto demag = [&](const float* U) {
        // rows forward
#pragma unroll 1
        for (int task = tid; task < (3 * ny * G1 + 31) / 32 * 32; task += NT) {
            const int row = task / G1, t = task % G1;
            const bool on = row < 3 * ny;
            lcx<float>* line = S + (on ? row : 0) * KP;
            const float* u = U + (on ? row : 0) * nx;
            lcx<float> v[Q1];
#pragma unroll
            for (int q = 0; q < Q1; ++q) {
                const int n = 2 * (q * G1 + t);
                v[q] = lzero<float>();
                if (q < XS::QIN && on) {
                    if (n < nx) v[q].re = Ms * u[n];
                    if (n + 1 < nx) v[q].im = Ms * u[n + 1];
                }
            }
            lfft<1, Q1, float, (XS::QIN < Q1 ? XS::QIN : Q1)>(v);
            if (on) {
#pragma unroll
                for (int k1 = 0; k1 < Q1; ++k1)
                    line[t * XS::US + k1] = k1 > 0 && G1 > 1 ? lctwr<1>(v[k1], ltw_load<float>(cd.twx, 2 * t * k1)) : v[k1];
            }
            __syncwarp();
            lcx<float> z[XS::NSL][G1], y[XS::NSL][G1];
#pragma unroll
            for (int i = 0; i < XS::NSL; ++i) {
                const int j = t + i * G1;
                if (j < XS::NS) {
                    const int k1b = j == 0 ? Q1 / 2 : Q1 - j;
#pragma unroll
                    for (int u2 = 0; u2 < G1; ++u2) {
                        z[i][u2] = line[u2 * XS::US + j];
                        y[i][u2] = line[u2 * XS::US + k1b];
                    }
                }
            }
            __syncwarp();                                         // the line becomes the spectrum
#pragma unroll
            for (int i = 0; i < XS::NSL; ++i) {
                const int j = t + i * G1;
                if (j >= XS::NS || !on) continue;
                lfft<1, G1, float>(z[i]);
                lfft<1, G1, float>(y[i]);
#pragma unroll
                for (int e = 0; e < (i == 0 ? (XS::NE > G1 ? XS::NE : G1) : G1); ++e) {
                    int k = j + Q1 * e;
                    lcx<float> p = z[i][e < G1 ? e : 0], m = y[i][e < G1 ? G1 - 1 - e : 0];
                    bool use = e < G1;
                    if (i == 0 && j == 0) {
                        if (e < XS::NB) {
                            k = Q1 / 2 + Q1 * e;
                            p = y[i][e < G1 ? e : 0];
                        } else {
                            constexpr int nb = XS::NB;
                            const int x = e - nb;
                            k = Q1 * x;
                            p = z[i][x < G1 ? x : 0];
                            m = z[i][x < G1 ? (G1 - x) % G1 : 0];
                        }
                        use = e < XS::NE;
                    }
                    if (use) {
                        float2 xk, xm;
                        x_split<float>(p, m, __ldg(cd.twx + k), xk, xm);
                        line[k] = {xk.x, xk.y};
                        line[M - k] = {xm.x, xm.y};
                    }
                }
            }
        }
        __syncthreads();
        // columns forward: thread (component, t, column)
#pragma unroll 1
        for (int task = tid; task < 3 * G2 * KX; task += NT) {
            const int col = task % KX, ct = task / KX, t = ct % G2, c = ct / G2;
            lcx<float> v[Q2];
#pragma unroll
            for (int q = 0; q < Q2; ++q) {
                const int n = q * G2 + t;
                v[q] = q < QIN && n < ny ? S[(c * ny + n) * KP + col] : lzero<float>();
            }
            lfft<1, Q2, float, QIN>(v);
#pragma unroll
            for (int k1 = 0; k1 < Q2; ++k1)
                E[(ct * Q2 + k1) * KX + col] = k1 > 0 ? lctwr<1>(v[k1], ltw_load<float>(cd.twy, t * k1)) : v[k1];
        }
        __syncthreads();
        // across the line parts, tensor, and back: items (z | x and y, k1, column)
        const float* K = cd.khat;
        const long long kcs = (long long)cd.Ky * Wk;
#pragma unroll 1
        for (int task = tid; task < 2 * Q2 * KX; task += NT) {
            const bool zc = task >= Q2 * KX;
            const int it = zc ? task - Q2 * KX : task, k1 = it / KX, col = it % KX;
            if (zc) {
                lcx<float> m[G2];
#pragma unroll
                for (int u = 0; u < G2; ++u) m[u] = E[((2 * G2 + u) * Q2) * KX + it];
                lfft<1, G2, float>(m);
#pragma unroll
                for (int k2 = 0; k2 < G2; ++k2) {
                    const int kz = k1 + Q2 * k2;
                    const float k = __ldg(K + 2 * kcs + (long long)(lane_fold<L, Q2>(k1, k2) ? L - kz : kz) * Wk + col);
                    m[k2] = {k * m[k2].re, k * m[k2].im};
                }
                lfft<-1, G2, float>(m);
#pragma unroll
                for (int u = 0; u < G2; ++u) E[((2 * G2 + u) * Q2) * KX + it] = m[u];
            } else {
                lcx<float> m[2][G2];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
#pragma unroll
                    for (int u = 0; u < G2; ++u) m[c][u] = E[((c * G2 + u) * Q2) * KX + it];
                    lfft<1, G2, float>(m[c]);
                }
#pragma unroll
                for (int k2 = 0; k2 < G2; ++k2) {
                    const bool fold = lane_fold<L, Q2>(k1, k2);
                    const int kz = k1 + Q2 * k2;
                    const float* Kp = K + (long long)(fold ? L - kz : kz) * Wk + col;
                    const float kxx = __ldg(Kp), kyy = __ldg(Kp + kcs), kxy = (fold ? -1.f : 1.f) * __ldg(Kp + 3 * kcs);
                    const lcx<float> x = m[0][k2], y = m[1][k2];
                    m[0][k2] = {kxx * x.re + kxy * y.re, kxx * x.im + kxy * y.im};
                    m[1][k2] = {kxy * x.re + kyy * y.re, kxy * x.im + kyy * y.im};
                }
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    lfft<-1, G2, float>(m[c]);
#pragma unroll
                    for (int u = 0; u < G2; ++u) E[((c * G2 + u) * Q2) * KX + it] = m[c][u];
                }
            }
        }
        __syncthreads();
#pragma unroll 1
        for (int task = tid; task < 3 * G2 * KX; task += NT) {
            const int col = task % KX, ct = task / KX, t = ct % G2, c = ct / G2;
            lcx<float> v[Q2];
#pragma unroll
            for (int k1 = 0; k1 < Q2; ++k1) {
                const lcx<float> r = E[(ct * Q2 + k1) * KX + col];
                v[k1] = k1 > 0 ? lctwr<-1>(r, ltw_load<float>(cd.twy, t * k1)) : r;
            }
            lfft<-1, Q2, float>(v);
#pragma unroll
            for (int q = 0; q < QIN; ++q) {
                const int n = q * G2 + t;
                if (n < ny) S[(c * ny + n) * KP + col] = v[q];
            }
        }
        __syncthreads();
        // rows back, in place
#pragma unroll 1
        for (int task = tid; task < (3 * ny * G1 + 31) / 32 * 32; task += NT) {
            const int row = task / G1, t = task % G1;
            const bool on = row < 3 * ny;
            lcx<float>* line = S + (on ? row : 0) * KP;
            lane_c2r_row<float, M, G1, Q1, true>(reinterpret_cast<const float2*>(line), cd.twx, line, t, on,
                                                 [] { __syncwarp(); }, [&](int n, float2 v) {
                if (on && 2 * n < nx) reinterpret_cast<float2*>(line)[n] = v;
            });
        }
        __syncthreads();
    };

    auto gather = [&](const float* U, int i, int x, int y, const v3<float>& mc, v3<float>* nbv, bool* nbp, float* cnb) {
        const int pos[2] = {x, y}, dim[2] = {nx, ny}, stride[2] = {1, nx};
        const float hh[2] = {fa.hx, fa.hy};
#pragma unroll
        for (int d = 0; d < 2; ++d) {
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const int sg = s == 0 ? 1 : -1;
                const int q = pos[d] + sg, slot = 2 * d + s;
                const bool in = q >= 0 && q < dim[d];
                nbp[slot] = in;
                if (in) {
                    const int j = i + sg * stride[d];
                    nbv[slot] = mk3<float>(U[j], U[N + j], U[2 * N + j]);
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
    // slope or rotation vector of cell i of state U, the draw th added to the demag field
    auto slope = [&](const float* U, int i, const v3<float>& th, v3<float>& m) {
        const int y = i / nx, x = i - y * nx;
        m = mk3<float>(U[i], U[N + i], U[2 * N + i]);
        v3<float> nbv[6], H, k;
        bool nbp[6];
        float cnb[6];
        gather(U, i, x, y, m, nbv, nbp, cnb);
        const v3<float> hd = mk3<float>(hrow(0, y)[x], hrow(1, y)[x], hrow(2, y)[x]) + th;
        cell_field_nb<float, EXT>(fa, i, R, m, nbv, nbp, cnb, true, hd, 0, H, k, true, dm);
        return k;
    };

    for (int s = 0; s < a.nsteps; ++s) {
        const long long step = step0 + s;
        v3<float> th[CPT], w1[CPT], m0[CPT];
        demag(A);
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const int i = tid + q * NT;
            if (i < N) {
                th[q] = hot && fa.th_scale != 0.f ? thermal_h<float>(fa, i, R, step - rp.step0) : zero;
                w1[q] = slope(A, i, th[q], m0[q]);
                const v3<float> ms = dm ? rodrigues<float>(m0[q], w1[q], dt) : m0[q] + dt * w1[q];
                B[i] = ms.x; B[N + i] = ms.y; B[2 * N + i] = ms.z;
            }
        }
        __syncthreads();
        demag(B);
        float proj = 0.f;
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const int i = tid + q * NT;
            if (i < N) {
                v3<float> ms;
                const v3<float> w2 = slope(B, i, th[q], ms);
                const v3<float> mn = dm ? rodrigues<float>(m0[q], 0.5f * (w1[q] + w2), dt) : m0[q] + (0.5f * dt) * (w1[q] + w2);
                const v3<float> mu = rsqrtf(dot(mn, mn)) * mn;
                A[i] = mu.x; A[N + i] = mu.y; A[2 * N + i] = mu.z;
                proj += dot(mu, ax);
            }
        }
        if (a.trials) {
            for (int o = 16; o > 0; o >>= 1) proj += __shfl_xor_sync(0xffffffffu, proj, o);
            if ((tid & 31) == 0) s_red[tid >> 5] = proj;
            __syncthreads();
            if (tid == 0) {
                float tot = 0.f;
                for (int w = 0; w < NT / 32; ++w) tot += s_red[w];
                s_new = trial_check(a.tr, rp, a.rep + blockIdx.x, tot / (float)N, step + 1 - rp.step0, step + 1);
                s_red[0] = rp.active ? 1.f : 0.f;
            }
            __syncthreads();
            const int refill = s_new;
            const bool alive = s_red[0] != 0.f;
            if (refill) {
                rp = a.rep[blockIdx.x];                           // the new trial's key, scales and start step
                fa.key0 = rp.key0;
                fa.key1 = rp.key1;
                fa.th_scale = rp.th_scale;
                fa.tq_base = rp.tq_base;
                for (int e = tid; e < 3 * N; e += NT) A[e] = __ldg(a.tr.m_init + e);
            }
            __syncthreads();
            if (!alive) break;
        } else {
            __syncthreads();
        }
    }
    for (int e = tid; e < 3 * N; e += NT) mg[e] = A[e];
}

// (half length M = G1 Q1 of the rows, length L = G2 Q2 of the columns, threads,
// CTAs per SM that the registers leave room for)
#define MM_TILE_DEMAG(X) \
    X(8, 2, 4, 16, 4, 4, 64, 8) X(12, 4, 3, 24, 4, 6, 128, 4) X(16, 4, 4, 32, 4, 8, 256, 2) X(24, 4, 6, 48, 6, 8, 512, 1) \
    X(32, 4, 8, 64, 8, 8, 512, 1)

using TileDemagKern = void (*)(TileDemagArgs);
struct TileDemagShape {
    TileDemagKern kern[2];
    int threads;
    size_t smem;
};
static TileDemagShape tile_demag_shape(int M, int L) {
    switch (M * 10000 + L) {
#define MM_CASE(m, g1, q1, l, g2, q2, nt, mb) \
    case m * 10000 + l: return {{tile_demag_kernel<m, g1, q1, l, g2, q2, nt, mb, false>, tile_demag_kernel<m, g1, q1, l, g2, q2, nt, mb, true>}, \
                                nt, tile_demag_smem<m, g1, q1, l, g2, q2>()};
        MM_TILE_DEMAG(MM_CASE)
#undef MM_CASE
        default: return {{nullptr, nullptr}, 0, 0};
    }
}

bool tile_demag_supported(int Lh, int Py) { return tile_demag_shape(Lh, Py).threads != 0; }

cudaError_t tile_demag_attributes(int Lh, int Py) {
    const TileDemagShape s = tile_demag_shape(Lh, Py);
    for (TileDemagKern k : s.kern) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s.smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

void tile_demag_launch(const MacroArgs& a, const ClsDev* cls, int Lh, int Py, cudaStream_t stream) {
    const TileDemagShape s = tile_demag_shape(Lh, Py);
    s.kern[a.ext ? 1 : 0]<<<a.R, s.threads, s.smem, stream>>>(TileDemagArgs{a, cls});
}

}  // namespace mm
