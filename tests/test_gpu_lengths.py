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
