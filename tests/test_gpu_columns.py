"""GPU parity of the demag passes at every line length that has a kernel of
its own, and at both ends of the range of sizes that is padded to it: the
middle pass of a film, of many films and of a 3-D grid, the Y passes and the
X passes (with the RK45 stage state formed inside).
The demag field is compared with the FP64 oracle's transforms; the bars are
those of the field tests (an FP32 transform of these lengths rounds to a few
1e-7 of the largest field, FP64 to a few 1e-16)."""
import numpy as np
import pytest

import workloads as W
from gpu_util import TERMS, make_ctx, need_gpu, oracle_problem, rel_err

pytestmark = pytest.mark.gpu

LENGTHS = sorted(2 ** a * 3 ** b for a in range(11) for b in range(7) if 2 <= 2 ** a * 3 ** b <= 1024)
MAT = W.Material(Ms=8.0e5, A=1.3e-11, alpha=0.02)


def _sizes(L):
    """The smallest and the largest n that are padded to L (2n - 1 points)."""
    below = max([v for v in LENGTHS if v < L], default=0)
    return sorted({below // 2 + 1, (L + 1) // 2} - {1})


def _check(grid, prec):
    mm = need_gpu()
    from oracle.demag import demag_spectrum, h_demag
    ctx = make_ctx(mm, grid, MAT, precision=prec, demag=True)
    try:
        mm.mm_set_m(ctx, 0, W.m_random_sphere(grid, seed=grid.n))
        m = mm.mm_get_m(ctx, 0, (3,) + grid.shape)
        p = oracle_problem(grid, MAT)
        ref = h_demag(m, p, demag_spectrum(p.shape, p.d))
        H = mm.mm_get_heff(ctx, 0, m.shape, TERMS["demag"])
        assert rel_err(H, ref) < (1e-11 if prec == 64 else 5e-6)
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("L", [v for v in LENGTHS if v >= 12])
def test_film_middle_pass(L, prec):
    for ny in _sizes(L):
        _check(W.Grid(5 if ny % 2 else 10, ny, 1, 2e-9, 2e-9, 1e-9), prec)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("L", [v for v in LENGTHS if v >= 27])
def test_y_passes(L, prec):
    for ny in _sizes(L):
        _check(W.Grid(3, ny, 2, 2e-9, 2e-9, 2e-9), prec)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("L", [v for v in LENGTHS if 9 <= v <= 144])
def test_z_middle_pass(L, prec):
    for nz in _sizes(L):
        _check(W.Grid(9, 6, nz, 3e-9, 3e-9, 3e-9), prec)


@pytest.mark.parametrize("n", [16, 18, 27, 33, 54, 72, 81, 108])
def test_many_films_match_one(n):
    """Enough films for the kernel of ensembles: the first and the last
    replica, two Heun steps, against the FP64 oracle."""
    mm = need_gpu()
    from oracle.llg import Solver
    R = 2 * 160 * 32 // (n + 1) + 1
    cell = (2e-9, 2e-9, 1e-9)
    M = mm.Material(MAT.Ms, MAT.A, MAT.alpha)
    cfg = mm.make_config(precision=32, integrator=mm.MM_HEUN, demag=mm.MM_DEMAG_EXACT, dt=1e-13)
    ctx = mm.mm_create_batch([mm.make_grid(n, n, 1, *cell)] * R, M.s, cfg)
    try:
        mm.mm_batch_set_shape(ctx, 0)
        g = W.Grid(n, n, 1, *cell)
        m0 = {r: W.m_perp(g, seed=r, tilt=0.3) for r in (0, R - 1)}
        for r, m in m0.items():
            mm.mm_set_m(ctx, r, m)
        mm.mm_step(ctx, 2)
        p = oracle_problem(g, MAT)
        for r, m in m0.items():
            o = Solver(p, m, terms=("exchange", "zeeman", "demag"), dt=1e-13)
            for _ in range(2):
                o.heun_step()
            assert np.abs(mm.mm_get_m(ctx, r, m.shape) - o.m).max() <= 1e-5
    finally:
        mm.mm_destroy(ctx)


X_LENGTHS = [v for v in LENGTHS if v % 2 == 0 and v >= 24]


@pytest.mark.parametrize("cells", [False, True])
@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("L", X_LENGTHS)
def test_x_passes(L, prec, cells):
    """Rows padded to L, the smallest and the largest, even and odd; with many
    materials the source Ms comes from the region map."""
    mm = need_gpu()
    from oracle.demag import demag_spectrum, h_demag
    below = max([v for v in LENGTHS if v % 2 == 0 and v < L])
    for nx in sorted({below // 2 + 1, L // 2 - 1, L // 2} - {1}):
        grid = W.Grid(nx, 3, 1, 2e-9, 2e-9, 1e-9)
        mat = W.with_cells(MAT, W.random_material_cells(grid, nx)) if cells else MAT
        ctx = make_ctx(mm, grid, mat, precision=prec, demag=True)
        try:
            mm.mm_set_m(ctx, 0, W.m_random_sphere(grid, seed=nx))
            m = mm.mm_get_m(ctx, 0, (3,) + grid.shape)
            p = oracle_problem(grid, mat)
            ref = np.where(p.present, h_demag(m, p, demag_spectrum(p.shape, p.d)), 0.0)
            H = mm.mm_get_heff(ctx, 0, m.shape, TERMS["demag"])
            assert rel_err(H, ref) < (1e-11 if prec == 64 else 5e-6)
        finally:
            mm.mm_destroy(ctx)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("shape", [(33, 4, 1), (50, 3, 2), (21, 5, 2), (128, 6, 1), (171, 2, 1), (64, 40, 14)])
def test_stage_state_formed_in_the_x_pass(shape, prec):
    """Ten RK45 steps replayed from the oracle: rows of odd and even length,
    one FP64 grid of more rows than take the row-per-warp kernel."""
    mm = need_gpu()
    from oracle.llg import Solver
    grid = W.Grid(*shape, 2e-9, 2e-9, 2e-9)
    m0 = W.m_random_sphere(grid, seed=7)
    o = Solver(oracle_problem(grid, MAT), m0, dt=1e-14, rtol=1e-6)
    dts = [o.rk45_step() for _ in range(10)]
    ctx = make_ctx(mm, grid, MAT, precision=prec, dt=1e-14, rtol=1e-6)
    try:
        mm.mm_set_m(ctx, 0, m0)
        mm.mm_step_dt(ctx, dts)
        assert np.abs(mm.mm_get_m(ctx, 0, m0.shape) - o.m).max() <= (1e-11 if prec == 64 else 1e-5)
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("kind", ["slopes", "current", "cubic"])
@pytest.mark.parametrize("L", X_LENGTHS)
def test_x_pass_inside_the_field_kernel(L, kind):
    """FP32 rows padded to L, of the smallest and the largest even length (four
    cells a thread where four divide it): two RK4 steps, two Heun steps with a
    current and a temperature, two RK4 steps with the further local terms,
    against the FP64 oracle."""
    mm = need_gpu()
    from oracle.llg import Solver, Torque, replica_seed
    below = max([v for v in LENGTHS if v % 2 == 0 and v < L])
    lo = below // 2 + 1
    for nx in sorted({lo + lo % 2, L // 2 - L // 2 % 2}):
        grid = W.Grid(nx, 5, 2, 2e-9, 2e-9, 2e-9)
        mat = W.Material(Ms=8.0e5, A=1.3e-11, alpha=0.02, Kc1=4.5e4 if kind == "cubic" else 0.0)
        terms = ("exchange", "zeeman", "demag") + (("cubic",) if kind == "cubic" else ())
        m0 = W.m_perp(grid, seed=nx, tilt=0.3)
        T, tq = (300.0, Torque(kind="sot", J=2e11, p=(0, 1, 0), theta_SH=0.1, fl_ratio=0.3)) if kind == "current" else (0.0, Torque())
        o = Solver(oracle_problem(grid, mat), m0, terms=terms, dt=1e-14, T=T, seed=replica_seed(5, 0), torque=tq)
        ctx = make_ctx(mm, grid, mat, precision=32, dt=1e-14, T=T, seed=5, integrator="heun" if T else "rk4")
        try:
            if T:
                mm.mm_set_torque(ctx, mm.make_torque(mm.MM_TORQUE_SOT, p=(0, 1, 0), theta_SH=0.1, fl_ratio=0.3), 2e11)
            mm.mm_set_m(ctx, 0, m0)
            mm.mm_step(ctx, 2)
            for _ in range(2):
                o.heun_step() if T else o.rk4_step()
            assert np.abs(mm.mm_get_m(ctx, 0, m0.shape) - o.m).max() <= 1e-5, nx
        finally:
            mm.mm_destroy(ctx)


@pytest.mark.parametrize("L", X_LENGTHS)
def test_x_pass_inside_the_fp64_slopes(L):
    """FP64 rows padded to L, even and odd, few enough that CTAs share a row: two
    RK4 steps and two RK45 steps of the oracle's sizes."""
    mm = need_gpu()
    from oracle.llg import Solver
    below = max([v for v in LENGTHS if v % 2 == 0 and v < L])
    for nx in sorted({below // 2 + 1, L // 2 - 1, L // 2} - {1}):
        grid = W.Grid(nx, 5, 2, 2e-9, 2e-9, 2e-9)
        m0 = W.m_perp(grid, seed=nx, tilt=0.3)
        for integrator in ("rk4", "rk45"):
            o = Solver(oracle_problem(grid, MAT), m0, terms=("exchange", "zeeman", "demag"), dt=1e-14, rtol=1e-6)
            dts = [(o.rk4_step(), 1e-14)[1] if integrator == "rk4" else o.rk45_step() for _ in range(2)]
            ctx = make_ctx(mm, grid, MAT, precision=64, dt=1e-14, rtol=1e-6, integrator=integrator)
            try:
                mm.mm_set_m(ctx, 0, m0)
                mm.mm_step(ctx, 2) if integrator == "rk4" else mm.mm_step_dt(ctx, dts)
                assert np.abs(mm.mm_get_m(ctx, 0, m0.shape) - o.m).max() <= 1e-11, (nx, integrator)
            finally:
                mm.mm_destroy(ctx)


@pytest.mark.parametrize("integrator", ["heun", "dm"])
@pytest.mark.parametrize("n", [(8, 8), (7, 8), (12, 12), (16, 16), (15, 16), (16, 15), (24, 24), (32, 32), (31, 32)])
def test_small_film_ensembles_match_oracle(n, integrator):
    """Films of one small size in the stacked shape (a block of steps per
    launch): the whole range of the sizes it takes, a temperature and a current
    per replica, 12 steps against the FP64 oracle."""
    mm = need_gpu()
    from oracle.llg import Solver, Torque
    nx, ny = n
    R, cell = 5, (2e-9, 2e-9, 1e-9)
    mat = W.Material(Ms=1.1e6, A=2e-11, alpha=0.05, Ku1=9e5, D=1e-3)
    M = mm.Material(mat.Ms, mat.A, mat.alpha, mat.Ku1, mat.u, mat.D)
    cfg = mm.make_config(precision=32, integrator=mm.MM_HEUN if integrator == "heun" else mm.MM_DM,
                         demag=mm.MM_DEMAG_EXACT, dt=1e-14)
    seeds = np.arange(1, R + 1, dtype=np.uint64) * np.uint64(7919)
    T, J = np.linspace(0.0, 400.0, R), np.linspace(1e11, 3e11, R)
    ctx = mm.mm_create_batch([mm.make_grid(nx, ny, 1, *cell)] * R, M.s, cfg, seeds)
    try:
        mm.mm_batch_set_shape(ctx, 0)
        mm.mm_set_temperature(ctx, T)
        mm.mm_set_torque(ctx, mm.make_torque(mm.MM_TORQUE_SOT, p=(0, 1, 0), theta_SH=0.1, fl_ratio=0.3), J)
        g = W.Grid(nx, ny, 1, *cell)
        m0 = [W.m_perp(g, seed=100 + r, tilt=0.3) for r in range(R)]
        for r in range(R):
            mm.mm_set_m(ctx, r, m0[r])
        mm.mm_step(ctx, 7)
        mm.mm_step(ctx, 5)
        for r in range(R):
            o = Solver(oracle_problem(g, mat), m0[r], terms=("exchange", "dmi", "anisotropy", "zeeman", "demag"), T=T[r],
                       seed=int(seeds[r]), dt=1e-14,
                       torque=Torque(kind="sot", J=J[r], p=(0, 1, 0), theta_SH=0.1, fl_ratio=0.3))
            for _ in range(12):
                o.heun_step() if integrator == "heun" else o.dm_step()
            assert np.abs(mm.mm_get_m(ctx, r, m0[r].shape) - o.m).max() <= 1e-5, (r, n)
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("integrator", ["heun", "dm"])
@pytest.mark.parametrize("nx", [12, 16, 20, 24, 28, 32, 36, 44, 52, 60, 64, 72, 80, 96, 108, 128, 140, 160, 192, 212, 240, 256, 260])
def test_stacked_films_with_the_x_pass_in_the_field_kernel(nx, integrator):
    """Two size classes in the stacked shape, rows of every length that has the
    fused kernel (and one above), a temperature and a current per replica, three
    steps against the FP64 oracle."""
    mm = need_gpu()
    from oracle.llg import Solver, Torque
    mat, cell = W.Material(Ms=1.1e6, A=2e-11, alpha=0.05, Ku1=9e5, D=1e-3), (2e-9, 2e-9, 1e-9)
    sizes = [(nx, 5)] * 3 + [(9, 7)]
    M = mm.Material(mat.Ms, mat.A, mat.alpha, mat.Ku1, mat.u, mat.D)
    cfg = mm.make_config(precision=32, integrator=mm.MM_HEUN if integrator == "heun" else mm.MM_DM,
                         demag=mm.MM_DEMAG_EXACT, dt=1e-14)
    seeds = np.arange(1, 5, dtype=np.uint64) * np.uint64(104729)
    T, J = np.linspace(0.0, 300.0, 4), np.linspace(1e11, 3e11, 4)
    ctx = mm.mm_create_batch([mm.make_grid(a, b, 1, *cell) for a, b in sizes], M.s, cfg, seeds)
    try:
        mm.mm_batch_set_shape(ctx, 0)
        mm.mm_set_temperature(ctx, T)
        mm.mm_set_torque(ctx, mm.make_torque(mm.MM_TORQUE_SOT, p=(0, 1, 0), theta_SH=0.1, fl_ratio=0.3), J)
        g = [W.Grid(a, b, 1, *cell) for a, b in sizes]
        m0 = [W.m_perp(g[r], seed=nx + r, tilt=0.3) for r in range(4)]
        for r in range(4):
            mm.mm_set_m(ctx, r, m0[r])
        mm.mm_step(ctx, 3)
        for r in range(4):
            o = Solver(oracle_problem(g[r], mat), m0[r], terms=("exchange", "dmi", "anisotropy", "zeeman", "demag"), T=T[r],
                       seed=int(seeds[r]), dt=1e-14,
                       torque=Torque(kind="sot", J=J[r], p=(0, 1, 0), theta_SH=0.1, fl_ratio=0.3))
            for _ in range(3):
                o.heun_step() if integrator == "heun" else o.dm_step()
            assert np.abs(mm.mm_get_m(ctx, r, m0[r].shape) - o.m).max() <= 1e-5, (r, nx)
    finally:
        mm.mm_destroy(ctx)
