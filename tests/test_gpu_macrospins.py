"""GPU parity of the one-cell replica kernels: step counts around the block of
draws, a replica count that leaves lanes idle, every torque and both
integrators, interfacial DMI (whose ghosts act on a single cell) and, through
the general kernel, bulk DMI; against the FP64 oracle, bar 1e-5 (FP32)."""
import numpy as np
import pytest

import workloads as W
from gpu_util import need_gpu, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Db", [0.0, 1e-3])
@pytest.mark.parametrize("torque", ["none", "sot", "stt"])
@pytest.mark.parametrize("integrator", ["heun", "dm"])
def test_one_cell_blocks_match_oracle(integrator, torque, Db):
    mm = need_gpu()
    from oracle.llg import Solver, Torque
    R, cell = 33, (3e-9, 3e-9, 2e-9)
    mat = W.Material(Ms=1.0e6, A=1.5e-11, alpha=0.1, Ku1=6e5, u=(0.1, 0.0, 1.0), D=2e-3, Db=Db)
    M = mm.Material(mat.Ms, mat.A, mat.alpha, mat.Ku1, mat.u, mat.D, Db=Db)
    cfg = mm.make_config(precision=32, integrator=mm.MM_HEUN if integrator == "heun" else mm.MM_DM,
                         demag=mm.MM_DEMAG_OFF, dt=5e-14)
    seeds = np.arange(1, R + 1, dtype=np.uint64) * np.uint64(104729)
    T, J = np.linspace(0.0, 400.0, R), np.linspace(1e11, 5e11, R)
    ctx = mm.mm_create_batch([mm.make_grid(1, 1, 1, *cell)] * R, M.s, cfg, seeds)
    tq = dict(p=(0.0, 1.0, 0.3), theta_SH=0.2, fl_ratio=0.4, P=0.5, Lambda=1.4, eps_prime=0.1)
    try:
        mm.mm_set_temperature(ctx, T)
        if torque != "none":
            mm.mm_set_torque(ctx, mm.make_torque(mm.MM_TORQUE_SOT if torque == "sot" else mm.MM_TORQUE_STT, **tq), J)
        g = W.Grid(1, 1, 1, *cell)
        m0 = [W.m_random_sphere(g, seed=r) for r in range(R)]
        for r in range(R):
            mm.mm_set_m(ctx, r, m0[r])
        for n in (1, 11, 12, 13):
            mm.mm_step(ctx, n)
        for r in (0, 1, 16, 31, 32):
            o = Solver(oracle_problem(g, mat), m0[r], terms=("exchange", "dmi", "anisotropy", "zeeman"), T=T[r],
                       seed=int(seeds[r]), dt=5e-14, torque=Torque(kind=torque, J=J[r], **tq))
            for _ in range(37):
                o.heun_step() if integrator == "heun" else o.dm_step()
            assert np.abs(mm.mm_get_m(ctx, r, (3, 1, 1, 1)) - o.m).max() <= 1e-5, r
    finally:
        mm.mm_destroy(ctx)
