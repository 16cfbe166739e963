"""Fixed steps of single instances: their clock and counters over any order of
calls, and the cost of a step's bookkeeping on large grids."""
import numpy as np
import pytest

import workloads as W
from gpu_util import make_ctx, need_gpu

pytestmark = pytest.mark.gpu

MAT = W.Material(Ms=8.0e5, A=1.3e-11, alpha=0.02)


@pytest.mark.parametrize("integrator", ["heun", "dm", "rk4"])
@pytest.mark.parametrize("shape", [(33, 9, 1), (128, 64, 17)])
def test_clock_and_counters(shape, integrator):
    """t grows by dt a step, rounded each time, over single steps, blocks of them,
    runs to a time, a new state and a restored one."""
    mm = need_gpu()
    dt = 1e-14
    ctx = make_ctx(mm, W.Grid(*shape, 2e-9, 2e-9, 2e-9), MAT, precision=32, integrator=integrator, dt=dt)
    t, n = 0.0, 0

    def check():
        assert mm.mm_get_time(ctx) == (t, dt, n)

    try:
        m0 = W.m_random_sphere(W.Grid(*shape, 2e-9, 2e-9, 2e-9), seed=3)
        mm.mm_set_m(ctx, 0, m0)
        for k in (1, 3, 8, 21):
            mm.mm_step(ctx, k)
            for _ in range(k):
                t, n = t + dt, n + 1
            check()
        blob = mm.mm_get_state(ctx)
        saved = t, n
        mm.mm_run(ctx, 5e-13)
        while t < 5e-13:
            t, n = t + dt, n + 1
        check()
        mm.mm_set_m(ctx, 0, m0)
        mm.mm_step(ctx, 2)
        t, n = t + dt + dt, n + 2
        check()
        mm.mm_set_state(ctx, blob)
        t, n = saved
        check()
        mm.mm_step(ctx, 9)
        for _ in range(9):
            t, n = t + dt, n + 1
        check()
    finally:
        mm.mm_destroy(ctx)


def test_the_corrector_costs_its_bytes():
    """Heun without demag at 8.4 M cells: the corrector moves 48 bytes a cell, the
    predictor 36, both stream; a step's end inside the corrector made it take 1.4
    times as long."""
    mm = need_gpu()
    grid = W.Grid(512, 512, 32, 3e-9, 3e-9, 3e-9)
    ctx = make_ctx(mm, grid, MAT, precision=32, integrator="heun", demag=False)
    try:
        mm.mm_step(ctx, 4)
        best = {}
        for _ in range(4):
            mm.mm_set_profiling(ctx, True)
            mm.mm_step(ctx, 8)
            for e in mm.mm_get_profile(ctx):
                best[e["name"]] = min(best.get(e["name"], np.inf), e["total_ms"] / e["launches"])
            mm.mm_set_profiling(ctx, False)
        assert best["field_heun2"] < 48 / 36 * best["field_heun1"]
    finally:
        mm.mm_destroy(ctx)
