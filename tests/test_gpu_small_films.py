"""Ensembles of one small film size with demag in the stacked shape, which run
blocks of steps per launch (batch_tile.cu): what a caller sees of the clock and
of the launch shape is that of every other ensemble with demag."""
import numpy as np
import pytest

import workloads as W
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

CELL = (2e-9, 2e-9, 1e-9)
MAT = W.Material(Ms=1.1e6, A=2e-11, alpha=0.05, Ku1=9e5)


def _films(mm, n, R, dt, shape=0, integrator=None, T=0.0):
    M = mm.Material(MAT.Ms, MAT.A, MAT.alpha, MAT.Ku1, MAT.u)
    cfg = mm.make_config(precision=32, integrator=mm.MM_HEUN if integrator is None else integrator,
                         demag=mm.MM_DEMAG_EXACT, dt=dt, T=T)
    ctx = mm.mm_create_batch([mm.make_grid(n, n, 1, *CELL)] * R, M.s, cfg)
    ctx._mat = M
    mm.mm_batch_set_shape(ctx, shape, R if shape else 0)
    return ctx


@pytest.mark.parametrize("dt, t_end", [(1e-14, 1e-13), (1e-13, 1e-12), (1e-14, 2e-11)])
@pytest.mark.parametrize("shape", [0, 256])
def test_a_run_to_a_time_steps_while_the_summed_time_is_below_it(shape, dt, t_end):
    """t grows by dt a step, rounded each time, and a step is taken while it is
    below t_end: 11, 10 and 2001 steps here (ten times 1e-14 is below 1e-13)."""
    mm = need_gpu()
    t, n = 0.0, 0
    while t < t_end:
        t, n = t + dt, n + 1
    ctx = _films(mm, 16, 3, dt, shape)
    try:
        mm.mm_run(ctx, t_end)
        assert mm.mm_get_time(ctx) == (t, dt, n)
        mm.mm_run(ctx, t_end)                       # there already
        mm.mm_step(ctx, 5)
        for _ in range(5):
            t += dt
        assert mm.mm_get_time(ctx) == (t, dt, n + 5)
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("R", [4, 256])
def test_the_autotuner_times_what_a_step_runs(R, tmp_path):
    """The stacked shape runs blocks of steps of these films, 5 to 15 times as fast
    as the per-class passes: the autotuner picks it, and the time that it records
    is that of a step (within a factor of 3: three steps a launch, and the clock's
    ramp)."""
    mm = need_gpu()
    import json
    import time
    ctx = _films(mm, 16, R, 1e-14)
    try:
        cache = tmp_path / "shapes"
        assert mm.mm_batch_autotune(ctx, str(cache))[0] == 0
        recorded = list(json.loads(cache.read_text().splitlines()[-1]).values())[0]
        assert recorded["nt"] == 0
        mm.mm_step(ctx, 1024)
        t = time.perf_counter()
        mm.mm_step(ctx, 1024)
        step = 1e3 * (time.perf_counter() - t) / 1024
        assert step / 3 < recorded["ms_per_step"] < 3 * step
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("n, terms, most", [(16, 0, 0.0), (40, 1 | 8 | 16, 1.0), (40, 0, 2.0)])
def test_the_stacked_shape_allocates_what_its_kernels_read(n, terms, most):
    """Blocks of steps need no buffer; the class passes need the spectra and the
    demag field, and the thermal field of a step (12 bytes a cell) where that term is
    on: `most` times 12 bytes a cell beside the spectra, and 4 MB for the modules."""
    mm = need_gpu()
    import torch
    R = 4096
    M = mm.Material(MAT.Ms, MAT.A, MAT.alpha, MAT.Ku1, MAT.u)
    cfg = mm.make_config(precision=32, integrator=mm.MM_HEUN, demag=mm.MM_DEMAG_EXACT, dt=1e-14, terms=terms)
    warm = _films(mm, n, 2, 1e-14)                  # (kernels loaded)
    ctx = mm.mm_create_batch([mm.make_grid(n, n, 1, *CELL)] * R, M.s, cfg)
    try:
        free = torch.cuda.mem_get_info()[0]
        mm.mm_batch_set_shape(ctx, 0)
        taken = free - torch.cuda.mem_get_info()[0]
        spectra = 0 if n == 16 else R * 3 * n * 52 * 8          # rows padded to 96: 49 columns, a pitch of 52
        assert taken <= spectra + most * 12 * R * n * n + (4 << 20)
    finally:
        mm.mm_destroy(warm)
        mm.mm_destroy(ctx)
