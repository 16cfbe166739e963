"""Grids of many layers, long rows and few rows: the lengths of the demag passes
beyond those of the other tests' grids have kernels of their own too.  Fields
against the FP64 oracle (the bars of the field tests), and the time of a pass
against that of a shorter length: the runtime-planned pass that a length without
a kernel falls to takes 5 to 20 times as long a point."""
import numpy as np
import pytest

import workloads as W
from gpu_util import make_ctx, need_gpu
from test_gpu_columns import MAT, _check, _sizes

pytestmark = pytest.mark.gpu


def _pass_us(mm, shape, name, integrator="rk4"):
    """Shortest mean time of the pass `name` in four steps of the grid."""
    grid = W.Grid(*shape, 3e-9, 3e-9, 3e-9)
    ctx = make_ctx(mm, grid, MAT, precision=32, integrator=integrator)
    try:
        mm.mm_set_m(ctx, 0, W.m_random_sphere(grid, seed=1))
        mm.mm_step(ctx, 2)
        best = np.inf
        for _ in range(3):
            mm.mm_set_profiling(ctx, True)
            mm.mm_step(ctx, 4)
            best = min(best, *[1e3 * e["total_ms"] / e["launches"] for e in mm.mm_get_profile(ctx) if e["name"] == name])
            mm.mm_set_profiling(ctx, False)
        return best
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("prec", [64, 32])
@pytest.mark.parametrize("ny", [7, 8])
@pytest.mark.parametrize("nx", [3, 64])
def test_short_y_lines(nx, ny, prec):
    _check(W.Grid(nx, ny, 5, 2e-9, 2e-9, 2e-9), prec)


@pytest.mark.parametrize("name", ["fft_y_fwd", "fft_y_inv"])
def test_short_y_lines_have_a_kernel(name):
    """Eight rows (16 points) against sixteen (32 points), in half of a pass's
    columns: launches alone, the same kernel."""
    mm = need_gpu()
    assert _pass_us(mm, (64, 8, 6), name) < 1.5 * _pass_us(mm, (64, 16, 6), name)


@pytest.mark.parametrize("cells", [False, True])
@pytest.mark.parametrize("nx", [973, 1023, 1024])
def test_long_rows(nx, cells):
    """The smallest, the largest odd and the largest row of half length 1024."""
    mm = need_gpu()
    from oracle.demag import demag_spectrum, h_demag
    from gpu_util import TERMS, oracle_problem, rel_err
    grid = W.Grid(nx, 3, 1, 2e-9, 2e-9, 1e-9)
    mat = W.with_cells(MAT, W.random_material_cells(grid, nx)) if cells else MAT
    ctx = make_ctx(mm, grid, mat, precision=32)
    try:
        mm.mm_set_m(ctx, 0, W.m_random_sphere(grid, seed=nx))
        m = mm.mm_get_m(ctx, 0, (3,) + grid.shape)
        p = oracle_problem(grid, mat)
        ref = np.where(p.present, h_demag(m, p, demag_spectrum(p.shape, p.d)), 0.0)
        assert rel_err(mm.mm_get_heff(ctx, 0, m.shape, TERMS["demag"]), ref) < 5e-6
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("shape", [(1024, 5, 1), (975, 3, 2)])
def test_stage_state_of_long_rows(shape):
    """Ten RK45 steps replayed from the oracle."""
    mm = need_gpu()
    from gpu_util import oracle_problem
    from oracle.llg import Solver
    grid = W.Grid(*shape, 2e-9, 2e-9, 2e-9)
    m0 = W.m_random_sphere(grid, seed=7)
    o = Solver(oracle_problem(grid, MAT), m0, dt=1e-14, rtol=1e-6)
    dts = [o.rk45_step() for _ in range(10)]
    ctx = make_ctx(mm, grid, MAT, precision=32, dt=1e-14, rtol=1e-6)
    try:
        mm.mm_set_m(ctx, 0, m0)
        mm.mm_step_dt(ctx, dts)
        assert np.abs(mm.mm_get_m(ctx, 0, m0.shape) - o.m).max() <= 1e-5
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("name", ["fft_x_r2c", "fft_x_c2r"])
def test_long_rows_have_a_kernel(name):
    """Rows of 1024 cells against rows of 512 in as many rows: twice the work."""
    mm = need_gpu()
    scale = _pass_us(mm, (511, 600, 1), name)       # (odd: the inverse pass is a launch of its own)
    assert _pass_us(mm, (1023, 600, 1), name) < 3 * scale


LONG_Z = [162, 192, 216, 256, 324, 432, 512, 1024]


@pytest.mark.parametrize("L", LONG_Z)
def test_long_z_lines(L):
    for nz in _sizes(L):
        _check(W.Grid(9, 6, nz, 3e-9, 3e-9, 3e-9), 32)


@pytest.mark.parametrize("L", [162, 192, 216])
def test_long_z_lines_of_many_columns(L):
    """(few and many columns have kernels of their own at 192 and 216 points)"""
    for nz in _sizes(L):
        _check(W.Grid(40, 62, nz, 3e-9, 3e-9, 3e-9), 32)


@pytest.mark.parametrize("L", LONG_Z)
def test_long_z_lines_have_a_kernel(L):
    mm = need_gpu()
    per_point = _pass_us(mm, (64, 64, 64), "fft_conv") / 128
    assert _pass_us(mm, (64, 64, L // 2), "fft_conv") / L < 5 * per_point
