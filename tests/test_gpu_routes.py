"""Kernels that the sizes of the other tests do not reach: the middle pass of many
films at every length, the FP64 X passes of more than ten rows per SM (plain,
odd, many materials, the stage state formed inside), the FP64 middle pass of films
wider than ten columns per SM, and retire/refill on the per-class passes.  Against
the FP64 oracle, with the bars of the field, step and trial tests."""
import numpy as np
import pytest

import workloads as W
from gpu_util import TERMS, make_ctx, need_gpu, oracle_problem, rel_err
from test_gpu_columns import LENGTHS, MAT, X_LENGTHS, _sizes
from test_gpu_trials import D1, _compare_outcomes, _context, _run_to_completion, _spec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [32, 36, 48, 54, 64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 256])
def test_middle_pass_of_many_films(L):
    """The smallest and the largest film padded to L, as many as take the kernel of
    ensembles, and one film of another size (a single small size would run blocks
    of steps): the first and the last replica, two Heun steps."""
    mm = need_gpu()
    from oracle.llg import Solver
    for n in _sizes(L):
        R, cell = 2 * 160 * 32 // (n + 1) + 1, (2e-9, 2e-9, 1e-9)
        M = mm.Material(MAT.Ms, MAT.A, MAT.alpha)
        cfg = mm.make_config(precision=32, integrator=mm.MM_HEUN, demag=mm.MM_DEMAG_EXACT, dt=1e-13)
        ctx = mm.mm_create_batch([mm.make_grid(n, n, 1, *cell)] * R + [mm.make_grid(9, 7, 1, *cell)], M.s, cfg)
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
                assert np.abs(mm.mm_get_m(ctx, r, m.shape) - o.m).max() <= 1e-5, (n, r)
        finally:
            mm.mm_destroy(ctx)


def _rows(mm):
    """ny, nz of a grid whose 3 ny nz rows are more than ten per SM."""
    import torch
    nz = 20
    return 10 * torch.cuda.get_device_properties(0).multi_processor_count // (3 * nz) + 1, nz


@pytest.mark.parametrize("kind", ["even", "odd", "cells"])
@pytest.mark.parametrize("L", X_LENGTHS)
def test_fp64_x_passes_of_many_rows(L, kind):
    """Rows padded to L: the demag field, and an RK45 step of the oracle's size,
    whose stage states the forward pass forms."""
    mm = need_gpu()
    from oracle.demag import demag_spectrum, h_demag
    from oracle.llg import Solver
    ny, nz = _rows(mm)
    below = max([v for v in LENGTHS if v % 2 == 0 and v < L])
    nx = {"even": L // 2 - L // 2 % 2, "odd": L // 2 - 1 + L // 2 % 2, "cells": below // 2 + 1}[kind]
    grid = W.Grid(nx, ny, nz, 2e-9, 2e-9, 1e-9)
    mat = W.with_cells(MAT, W.random_material_cells(grid, nx)) if kind == "cells" else MAT
    p = oracle_problem(grid, mat)
    K = demag_spectrum(p.shape, p.d)
    ctx = make_ctx(mm, grid, mat, precision=64, dt=1e-14)
    try:
        mm.mm_set_m(ctx, 0, W.m_random_sphere(grid, seed=nx))
        m = mm.mm_get_m(ctx, 0, (3,) + grid.shape)
        ref = np.where(p.present, h_demag(m, p, K), 0.0)
        assert rel_err(mm.mm_get_heff(ctx, 0, m.shape, TERMS["demag"]), ref) < 1e-11
        if L <= 384 or kind != "cells":             # (odd rows take the same kernel; the oracle is slow)
            o = Solver(p, m, K_hat=K, dt=1e-14, rtol=1e-6)
            mm.mm_step_dt(ctx, [o.rk45_step()])
            assert np.abs(mm.mm_get_m(ctx, 0, m.shape) - o.m).max() <= 1e-11
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("L", [v for v in LENGTHS if 16 <= v <= 512])
def test_fp64_middle_pass_of_wide_films(L):
    mm = need_gpu()
    import torch
    from oracle.demag import demag_spectrum, h_demag
    # columns are half of the padded row and one: the first length of more than ten per SM
    wide = min(2 ** a * 3 ** b for a in range(1, 14) for b in range(8)
               if 2 ** (a - 1) * 3 ** b + 1 > 10 * torch.cuda.get_device_properties(0).multi_processor_count)
    grid = W.Grid(wide // 2, _sizes(L)[0], 1, 2e-9, 2e-9, 1e-9)
    ctx = make_ctx(mm, grid, MAT, precision=64)
    try:
        mm.mm_set_m(ctx, 0, W.m_random_sphere(grid, seed=L))
        m = mm.mm_get_m(ctx, 0, (3,) + grid.shape)
        p = oracle_problem(grid, MAT)
        ref = h_demag(m, p, demag_spectrum(p.shape, p.d))
        assert rel_err(mm.mm_get_heff(ctx, 0, m.shape, TERMS["demag"]), ref) < 1e-11
    finally:
        mm.mm_destroy(ctx)


@pytest.mark.parametrize("integrator", ["dm", "heun"])
def test_retire_refill_on_the_class_passes(integrator):
    """Five trials over two slots of 36x36 films (too large for blocks of steps):
    the thermal field kept from predictor to corrector, idle slots, the stop test
    after the corrector."""
    mm = need_gpu()
    from dataclasses import replace
    grid = W.Grid(36, 36, 1, D1, D1, D1)
    mat = W.Material(Ms=1e6, A=1.5e-11, alpha=0.05, Ku1=1.1e6, u=(0, 0, 1))
    n = 5
    spec = replace(_spec(grid, mat, ("exchange", "anisotropy", "zeeman", "demag"), np.linspace(4e12, 1.2e13, n),
                         np.full(n, 300.0), 1e-13, 0.98, 150), integrator=integrator)
    ctx = _context(mm, spec, 2, mm.MM_DM if integrator == "dm" else mm.MM_HEUN, 1 | 4 | 8 | 16 | 32, True)
    try:
        mm.mm_batch_set_shape(ctx, 0)
        mm.mm_trials_start(ctx, spec.J, spec.T, spec.m_init, axis=spec.axis, threshold=spec.threshold,
                           max_steps=spec.max_steps, base_seed=spec.base_seed, refill=True)
        steps, stopped = _run_to_completion(mm, ctx, n, chunk=50)
        assert stopped.any() and not stopped.all()
        _compare_outcomes(spec, steps, stopped)
    finally:
        mm.mm_destroy(ctx)
