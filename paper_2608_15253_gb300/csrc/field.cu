// Fused effective field + LLG torque + stage update (Methods, "Physics and
// discretization", Eq. 1; the spin torques enter every integrator stage).
//
// One thread per cell.  The six-point exchange Laplacian, interfacial DMI
// (central differences; at an absent neighbour in the plane the ghost value
// m_i - h (D/2A)(z x n) x m_i, the sign that makes the discrete field the
// gradient of the discrete energy), uniaxial anisotropy, Zeeman, the demag
// field read from the FFT path, and the Philox4x32-10 thermal field are
// summed in registers; the torque and the requested stage update follow
// without writing H.
#include <cuda_runtime.h>

#include <algorithm>

#include "common.cuh"
#include "ctx.h"
#include "field_x.cuh"
#include "launch.h"

namespace mm {

template <typename T, bool UNIF, bool EXT>
__global__ void __launch_bounds__(256) field_kernel(FieldArgs<T> a) {
    dep_wait();
    if (a.gate && !a.st->active) return;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x < a.nx && y < a.ny) field_cell<T, UNIF, EXT>(a, x, y, blockIdx.z);
}

template <int V, bool EXT, bool QUIET = false>
__global__ void __launch_bounds__(256) field_vec_kernel(FieldArgs<float> a) {
    dep_wait();
    if (a.gate && !a.st->active) return;
    const int x0 = V * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x0 < a.nx && y < a.ny) {
        VecIn<V> in;
        field_vec_load<V, EXT, QUIET>(a, x0, y, blockIdx.z, in);
        field_vec_finish<V, EXT, false, QUIET>(a, x0, y, blockIdx.z, in, nullptr, 0);
    }
}

constexpr int kFieldV = 4;   // cells per thread of the one-material FP32 kernel (4 measured faster than 2)

template <typename T>
static FieldArgs<T> field_args(mm_ctx* c, int mode, unsigned terms, const T* m, const T* Hd, T* out, T* out2,
                               const T* m0, const T* k1, long long step_override, int gate, int kstage) {
    FieldArgs<T> a{};
    a.gate = gate;
    a.kstage = kstage;
    a.kptr = (T* const*)c->d_kslot;
    const mm_grid& g = c->grid;
    a.m = m; a.m0 = m0; a.k1 = k1; a.out = out; a.out2 = out2;
    a.Hd = Hd;
    a.Bc = (const T*)c->d_bcell;
    for (int d = 0; d < 3; ++d) a.hext[d] = (T)c->Hext[d];
    a.region = c->uniform ? nullptr : (const uint8_t*)c->d_region;
    a.lut = (const Region<T>*)c->d_lut;
    a.cpair = (const T*)c->d_cpair;
    a.nreg = c->nreg;
    a.nx = g.nx; a.ny = g.ny; a.nz = g.nz;
    a.N = c->N;
    a.hx = (T)g.dx; a.hy = (T)g.dy; a.hz = (T)g.dz;
    a.ix2 = (T)(1.0 / (g.dx * g.dx)); a.iy2 = (T)(1.0 / (g.dy * g.dy)); a.iz2 = (T)(1.0 / (g.dz * g.dz));
    a.px = g.pbc[0] != 0; a.py = g.pbc[1] != 0; a.pz = g.pbc[2] != 0;
    a.terms = terms;
    a.mode = mode;
    a.key0 = (uint32_t)(c->seed & 0xFFFFFFFFull);
    a.key1 = (uint32_t)(c->seed >> 32);
    const double V = g.dx * g.dy * g.dz;
    a.th_scale = c->Tr > 0 ? (T)std::sqrt(c->Tr / (V * c->cfg.dt)) : (T)0;
    // the predictor's draw serves the corrector (one draw per step by the scheme)
    a.noise = mode == MODE_HEUN1 || mode == MODE_HEUN2 || mode == MODE_DM1 || mode == MODE_DM2 ? (T*)c->d_hbuf : nullptr;
    a.st = c->d_state;
    a.step_override = step_override;
    a.cubic_w1 = c->cubic_energy ? (T)0.5 : (T)1;
    a.cubic_w2 = c->cubic_energy ? (T)(1.0 / 3.0) : (T)1;
    for (int k = 0; k < 6; ++k) a.strain[k] = (T)c->strain[k];
    a.strain_cell = (const T*)c->d_strain;
    a.rk1 = c->rkky_k1;
    a.rk2 = c->rkky_k2;
    a.rkky_c = (T)(c->rkky_J / g.dz);
    const mm_torque& q = c->tq;
    a.tq = q.kind;
    if (q.kind == MM_TORQUE_SOT || q.kind == MM_TORQUE_STT) {
        const double tF = q.t_F > 0 ? q.t_F : g.nz * g.dz;
        a.tq_base = (T)(kHbar * c->J / (kQe * kMu0 * tF));
        double pn = std::sqrt(q.p[0] * q.p[0] + q.p[1] * q.p[1] + q.p[2] * q.p[2]);
        if (pn == 0) pn = 1;
        for (int d = 0; d < 3; ++d) a.p[d] = (T)(q.p[d] / pn);
        a.theta_half = (T)(0.5 * q.theta_SH);
        a.fl_ratio = (T)q.fl_ratio;
        a.P = (T)q.P;
        a.L2 = (T)(q.Lambda * q.Lambda);
        a.eps_p = (T)q.eps_prime;
    } else if (q.kind == MM_TORQUE_ZL) {
        double u = c->J * q.P * kMuB / kQe;
        if (q.match_mumax) u /= (1.0 + q.xi * q.xi);
        a.zl_u = (T)u;
        a.xi = (T)q.xi;
        double dn = std::sqrt(q.dir[0] * q.dir[0] + q.dir[1] * q.dir[1] + q.dir[2] * q.dir[2]);
        if (dn == 0) dn = 1;
        for (int d = 0; d < 3; ++d) a.dir[d] = (T)(q.dir[d] / dn);
    }
    if constexpr (sizeof(T) == 4) { a.R0 = c->r0f; a.c_uniform = c->c00f; }
    else { a.R0 = c->r0d; a.c_uniform = c->c00d; }
    return a;
}

// The QUIET kernels apply: slopes only, no thermal field, no spin torque,
// none of the further local terms.
static bool field_quiet(const mm_ctx* c, int mode, unsigned terms) {
    return mode == MODE_K && !c->ext_terms && c->tq.kind == MM_TORQUE_NONE && (!(terms & MM_TERM_THERMAL) || !(c->Tr > 0));
}

static double field_bytes(const mm_ctx* c, int mode, unsigned terms, bool hd) {
    const double es = (double)c->esz;
    double bytes = 3 * es * 2 * c->N;          // read m, write out
    if (hd && (terms & MM_TERM_DEMAG)) bytes += 3 * es * c->N;
    if (mode == MODE_HEUN1 || mode == MODE_DM1) bytes += 3 * es * c->N;
    if (mode == MODE_HEUN2 || mode == MODE_DM2) bytes += 6 * es * c->N;
    return bytes;
}

static const char* const kFieldNames[6] = {"field_H", "field_k", "field_heun1", "field_heun2", "field_dm1",
                                           "field_dm2"};

template <typename T>
static void field_launch_t(mm_ctx* c, int mode, unsigned terms, const T* m, const T* Hd, T* out, T* out2,
                           const T* m0, const T* k1, long long step_override, int gate, int kstage) {
    FieldArgs<T> a = field_args<T>(c, mode, terms, m, Hd, out, out2, m0, k1, step_override, gate, kstage);
    const mm_grid& g = c->grid;
    // rows of 32 cells per warp, eight warps to a CTA; on small grids fewer, so
    // that every scheduler gets a warp (FP64, 128x32: 15.4 -> 10.7 us; 16 CTAs of
    // eight warps left the other SMs' FP64 pipes idle)
    const bool vec = sizeof(T) == 4 && c->uniform && !a.region && g.nx % kFieldV == 0 && a.R0.present != (T)0;
    const int gx = vec ? (g.nx / kFieldV + 31) / 32 : (g.nx + 31) / 32;
    int by = 8;
    while (by > 1 && (long long)gx * ((g.ny + by - 1) / by) * g.nz < 4 * sm_count()) by /= 2;
    dim3 blk(32, by);
    dim3 grd(gx, (g.ny + by - 1) / by, g.nz);
    LaunchScope ls(c, kFieldNames[mode], field_bytes(c, mode, terms, Hd != nullptr));
    if (c->uniform && !a.region) {
        if constexpr (sizeof(T) == 4) {
            if (vec) {
                if (c->ext_terms) launch_dep(field_vec_kernel<kFieldV, true>, grd, blk, 0, c, a);
                else if (field_quiet(c, mode, terms))
                    launch_dep(field_vec_kernel<kFieldV, false, true>, grd, blk, 0, c, a);
                else launch_dep(field_vec_kernel<kFieldV, false>, grd, blk, 0, c, a);
                return;
            }
        }
        if (c->ext_terms) launch_dep(field_kernel<T, true, true>, grd, blk, 0, c, a);
        else launch_dep(field_kernel<T, true, false>, grd, blk, 0, c, a);
    } else {
        if (c->ext_terms) launch_dep(field_kernel<T, false, true>, grd, blk, 0, c, a);
        else launch_dep(field_kernel<T, false, false>, grd, blk, 0, c, a);
    }
}

void field_launch(mm_ctx* c, int mode, unsigned terms, const void* m, const void* Hd, void* out, void* out2,
                  const void* m0, const void* k1, long long step_override, int gate, int kstage) {
    if (c->prec == 32)
        field_launch_t<float>(c, mode, terms, (const float*)m, (const float*)Hd, (float*)out, (float*)out2,
                              (const float*)m0, (const float*)k1, step_override, gate, kstage);
    else
        field_launch_t<double>(c, mode, terms, (const double*)m, (const double*)Hd, (double*)out, (double*)out2,
                               (const double*)m0, (const double*)k1, step_override, gate, kstage);
}

// Inverse X pass + field kernel in one launch (FP32, one material, even nx,
// any length of the X passes' register kernels).  One GB300, against the two
// kernels: 512x512x64 256 us (198 + 201), 250x250x40 56 us (35 + 55),
// 256x256x16 26.3 us, a 200x50 film 8.7 us (8.1 + 9.4).  Region maps and odd rows
// take the two kernels: a cell at a time in this one, 150x150x24 with a region
// map took 44 us against 11.3 + 21.
//
// FP64: slopes alone, and grids of no more rows than SMs (field_fine_d.cu: a row
// or less per CTA; with more rows the FP64 pipes are busy either way).
bool field_c2r_fusable(const mm_ctx* c, int mode, unsigned terms) {
    const mm_grid& g = c->grid;
    if (!c->dm.on || !c->uniform || c->d_region || g.nx > c->dm.Lh) return false;
    if (c->prec == 64)
        return c->r0d.present != 0.0 && field_quiet(c, mode, terms) && (long long)g.ny * g.nz <= sm_count() &&
               fine_field(c->dm.Lh).kern;
    return c->r0f.present != 0.f && g.nx % 2 == 0 && field_x_full(c->dm.Lh).group > 0;
}

// opts the kernels of the plan's length into their shared memory and loads
// them, outside any stream capture
cudaError_t field_c2r_setup(const mm_ctx* c) {
    cudaError_t e = cudaSuccess;
    const int M = c->dm.Lh;
    if (c->prec == 64) {
        const FineField f = fine_field(M);
        return f.kern ? cudaFuncSetAttribute(f.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fine_field_smem(f, M, 1)) : e;
    }
    for (const FieldX& f : {field_x_quiet(M), field_x_full(M), field_x_ext(M)}) {
        if (f.group == 0) continue;
        const size_t smem = field_x_smem(f.group, f.line, M, std::max(1, 96 / (3 * f.group)));
        for (const auto kern : f.kern)
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    }
    return e;
}

static void fine_field_launch(mm_ctx* c, int mode, unsigned terms, const double* m, double* out, long long step_override,
                              int gate, int kstage) {
    const FieldArgs<double> a = field_args<double>(c, mode, terms, m, nullptr, out, nullptr, nullptr, nullptr,
                                                   step_override, gate, kstage);
    const DemagPlan& d = c->dm;
    const int nx = c->grid.nx, rows = c->grid.ny * c->grid.nz;
    const FineField f = fine_field(d.Lh);
    const int parts = std::max(1, std::min(sm_count() / rows, (nx + 31) / 32)), warps = std::min(4, ((nx + parts - 1) / parts + 31) / 32);
    const FineSpec sp{(const double2*)d.spec, (const double2*)d.tw_x, d.PyA, d.Wk, parts};
    LaunchScope ls(c, "c2r_field", field_bytes(c, mode, terms, false) + 3.0 * rows * (d.Kx * sizeof(double2)));
    launch_dep(f.kern, rows * parts, 96 + 32 * warps, fine_field_smem(f, nx, parts), c, a, sp);
}

void field_c2r_launch(mm_ctx* c, int mode, unsigned terms, const void* m, void* out, void* out2, const void* m0,
                      const void* k1, long long step_override, int gate, int kstage) {
    if (c->prec == 64) {
        fine_field_launch(c, mode, terms, (const double*)m, (double*)out, step_override, gate, kstage);
        return;
    }
    FieldArgs<float> a = field_args<float>(c, mode, terms, (const float*)m, nullptr, (float*)out, (float*)out2,
                                           (const float*)m0, (const float*)k1, step_override, gate, kstage);
    const DemagPlan& d = c->dm;
    const int nx = c->grid.nx;
    const long long rows = (long long)c->grid.ny * c->grid.nz;
    const bool quiet = !c->ext_terms && field_quiet(c, mode, terms);
    const FieldX f = c->ext_terms ? field_x_ext(d.Lh) : quiet ? field_x_quiet(d.Lh) : field_x_full(d.Lh);
    const int four = quiet && nx % 4 == 0;
    const int rpc = c2r_rows(f.group, rows);
    const long long grid = (rows + rpc - 1) / rpc;
    const C2RSpec sp{(const float2*)d.spec, (const float2*)d.tw_x, d.PyA, d.Wk, rpc};
    // grids that fill the chip with CTAs of 96 threads: five of them per SM; on
    // smaller ones more threads share the cells (a 512x512 film: 12.0 us against 14.2)
    const int cells = (rpc * nx / (four ? 4 : 2) + 31) / 32 * 32, most = grid >= 5LL * sm_count() ? 96 : kC2RThreads;
    LaunchScope ls(c, "c2r_field", field_bytes(c, mode, terms, false) + 3.0 * rows * (d.Kx * sizeof(float2)));
    launch_dep(f.kern[four], (unsigned)grid, std::max(field_x_fft(f.group, rpc), std::min(most, cells)),
               field_x_smem(f.group, f.line, nx, rpc), c, a, sp);
}

// Raw Philox words and the thermal field of every cell at a given step.
template <typename T>
__global__ void thermal_raw_kernel(long long N, uint32_t k0, uint32_t k1, long long step, const uint8_t* region,
                                   const Region<T>* lut, T th_scale, uint32_t* raw, T* h) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= N) return;
    const U4 r = philox(U4{(uint32_t)i, (uint32_t)step, (uint32_t)((unsigned long long)step >> 32), 0u}, k0, k1);
    if (raw) {
        raw[4 * i] = r.x; raw[4 * i + 1] = r.y; raw[4 * i + 2] = r.z; raw[4 * i + 3] = r.w;
    }
    if (h) {
        T n[3];
        box_muller<T>(r, n);
        const Region<T>& R = lut[region ? region[i] : 0];
        const T sg = R.present != (T)0 ? R.sigma0 * th_scale : (T)0;
        h[i] = sg * n[0]; h[N + i] = sg * n[1]; h[2 * N + i] = sg * n[2];
    }
}

void thermal_raw_launch(mm_ctx* c, long long step, uint32_t* d_raw, void* d_h) {
    const double V = c->grid.dx * c->grid.dy * c->grid.dz;
    const double sc = c->Tr > 0 ? std::sqrt(c->Tr / (V * c->cfg.dt)) : 0.0;
    const unsigned blocks = (unsigned)((c->N + 255) / 256);
    const uint8_t* reg = c->uniform ? nullptr : (const uint8_t*)c->d_region;
    LaunchScope ls(c, "thermal_raw", 0.0);
    if (c->prec == 32)
        thermal_raw_kernel<float><<<blocks, 256, 0, c->stream>>>(c->N, (uint32_t)c->seed, (uint32_t)(c->seed >> 32),
                                                                 step, reg, (const Region<float>*)c->d_lut, (float)sc,
                                                                 d_raw, (float*)d_h);
    else
        thermal_raw_kernel<double><<<blocks, 256, 0, c->stream>>>(c->N, (uint32_t)c->seed, (uint32_t)(c->seed >> 32),
                                                                  step, reg, (const Region<double>*)c->d_lut, sc,
                                                                  d_raw, (double*)d_h);
}

}  // namespace mm
