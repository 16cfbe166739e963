"""Performance cases: what a user of the solver has it do, through its public entry points.

Every pass advances one context by a number of steps (`mm_step`) and reads the
magnetisation into the caller's device buffer (`mm_get_m_device`), the way a
simulation script advances to its next output.  The dynamics go on from pass to
pass, so the first-same-as-last slope of the adaptive integrator is reused as
in a long run.  Adaptive runs have their step capped (`dt_max`), which is also
how a user makes a run reproducible: the controller works, and every step has
the same length.

Covered: the film and block sizes that the paper and this repository's
workloads quote, both precisions, the adaptive and the fixed-step integrators,
one and many materials, zero and finite temperature with spin-orbit torque, and
the replica-batched ensembles.  The learned demag surrogate is left out: a step
with it is slower than one with the exact field on this GPU, and it has to be
trained before it can be used.
"""
import math

import numpy as np
import torch

import paper_2608_15253_gb300 as mm

GAMMA0, MU0, KB = 1.7595e11, 4e-7 * math.pi, 1.380649e-23
HBAR, QE = 1.054571817e-34, 1.602176634e-19

# Ms (A/m), A (J/m), alpha, Ku1 (J/m^3, along z), D (J/m^2), applied B (T)
MATERIALS = {
    "permalloy": (8.0e5, 1.3e-11, 0.02, 0.0, 0.0, (-24.6e-3, 4.3e-3, 0.0)),
    "dmi": (5.8e5, 1.5e-11, 0.1, 8e5, 3e-3, (0.0, 0.0, 0.0)),
    "skyrmion": (5.8e5, 1.5e-11, 0.3, 8e5, 3.5e-3, (0.0, 0.0, 0.2)),
    "perp": (1.1e6, 2e-11, 0.01, 9e5, 0.0, (0.0, 0.0, 0.0)),
}
THETA_SH, SOT_P = 0.1, (0.0, 1.0, 0.0)


def _case(name, kind, nx, ny, nz, cell, material, steps, precision=32, integrator="rk45", grains=False, T=0.0,
          J=0.0, dt=1e-14, R=1, edges="", demag=True):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "dx_nm": cell[0], "dy_nm": cell[1], "dz_nm": cell[2],
         "material": material, "steps": steps, "precision": precision, "integrator": integrator, "grains": grains,
         "T": T, "J": J, "dt": dt, "R": R, "edges": edges, "demag": demag}
    return dict(c, name=name) if name else c


def listed():
    return [
        # standard problem 4's film in double precision, sixteen steps between two samples of <m>
        _case("sp4_film_fp64", "one", 128, 32, 1, (3.90625, 3.90625, 3.0), "permalloy", 16, precision=64),
        # the smallest call: one adaptive step of a small film, its state read after every step
        _case("film_200x50_one_step", "one", 200, 50, 1, (2.5, 2.5, 3.0), "permalloy", 1),
        # relaxation of a skyrmion film
        _case("skyrmion_film_512x512", "one", 512, 512, 1, (2.0, 2.0, 1.0), "skyrmion", 8),
        # a finite-temperature film under spin-orbit torque, fixed-step Heun
        _case("hot_film_256x256_heun", "one", 256, 256, 1, (2.0, 2.0, 1.0), "perp", 32, integrator="heun", T=300.0,
              J=2e11),
        # a small block in double precision, classical RK4
        _case("block_64x64x16_fp64", "one", 64, 64, 16, (3.0, 3.0, 3.0), "permalloy", 4, precision=64,
              integrator="rk4"),
        # a granular block: many materials with absent cells, sizes that are no powers of two
        _case("granular_150x150x24", "one", 150, 150, 24, (3.0, 3.0, 3.0), "permalloy", 4, grains=True),
        # a chiral-magnet block
        _case("dmi_block_256x256x16", "one", 256, 256, 16, (2.0, 2.0, 2.0), "dmi", 4),
        # the paper's largest block
        _case("block_250x250x40", "one", 250, 250, 40, (3.0, 3.0, 3.0), "permalloy", 2),
        # the largest single problem
        _case("vortex_512x512x64", "one", 512, 512, 64, (3.0, 3.0, 3.0), "permalloy", 2),
        # 1024 perpendicular free layers of five sizes at 300 K, a current each
        _case("replicas_1024_uneven", "batch", 0, 0, 1, (2.0, 2.0, 1.0), "perp", 8, integrator="heun", T=300.0,
              J=3e11, R=1024, edges="32,48,64,96,128"),
        # the batching table's row with demag: 256 small films, Depondt-Mertens
        _case("replicas_256_16x16_dm", "batch", 0, 0, 1, (2.0, 2.0, 1.0), "perp", 64, integrator="dm", T=300.0,
              J=3e11, R=256, edges="16"),
        # the batching table's macrospin row: a thousand moments, a thousand steps
        _case("macrospins_1024_dm", "batch", 0, 0, 1, (2.0, 2.0, 1.0), "perp", 1024, integrator="dm", T=300.0, J=3e11,
              R=1024, edges="1", demag=False),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["film", "film", "block", "block", "block", "hot", "double", "batch"])
    if family == "film":
        nx, ny = _logint(rng, 32, 512), _logint(rng, 16, 512)
        cell, mat = rng.choice([((2.0, 2.0, 1.0), "skyrmion"), ((2.5, 2.5, 3.0), "permalloy"),
                                ((3.90625, 3.90625, 3.0), "permalloy")])
        return _case(None, "one", nx, ny, 1, cell, mat, rng.choice([1, 4, 16]), grains=rng.random() < 0.25)
    if family == "block":
        nx, ny, nz = _logint(rng, 32, 512), _logint(rng, 32, 512), _logint(rng, 2, 64)
        while nx * ny * nz > 1 << 22:
            nx, ny, nz = max(32, nx * 3 // 4), max(32, ny * 3 // 4), max(2, nz * 3 // 4)
        cell, mat = rng.choice([((2.0, 2.0, 2.0), "dmi"), ((3.0, 3.0, 3.0), "permalloy")])
        return _case(None, "one", nx, ny, nz, cell, mat, rng.choice([1, 2, 4]),
                     integrator=rng.choice(["rk45", "rk45", "rk4"]), grains=rng.random() < 0.25)
    if family == "hot":
        nx, ny, nz = _logint(rng, 32, 512), _logint(rng, 32, 512), rng.choice([1, 1, 1, 2, 4])
        return _case(None, "one", nx, ny, nz, (2.0, 2.0, 1.0), "perp", rng.choice([4, 8, 32]),
                     integrator=rng.choice(["heun", "dm"]), T=float(rng.randrange(50, 400)),
                     J=rng.uniform(1e11, 3e11))
    if family == "double":
        nx, ny, nz = _logint(rng, 24, 160), _logint(rng, 24, 160), rng.choice([1, 1, 2, 5, 12])
        return _case(None, "one", nx, ny, nz, (3.90625, 3.90625, 3.0), "permalloy", rng.choice([1, 4, 8]),
                     precision=64, integrator=rng.choice(["rk45", "rk45", "heun"]), grains=rng.random() < 0.25)
    edges = rng.choice(["16", "32", "32,64", "48,96", "32,48,64,96,128", "1"])
    one = edges == "1"
    return _case(None, "batch", 0, 0, 1, (2.0, 2.0, 1.0), "perp", rng.choice([256, 1024] if one else [4, 16]),
                 integrator=rng.choice(["heun", "dm"]), T=float(rng.randrange(50, 400)), J=rng.uniform(1e11, 3e11),
                 R=_logint(rng, 64, 8192 if one else 1024), edges=edges, demag=not one)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _edges(c):
    """Replica edge lengths, grouped by size (the order in which they are stored)."""
    pick = [int(e) for e in c["edges"].split(",")]
    return sorted(int(e) for e in np.random.default_rng(3).choice(pick, size=c["R"]))


def _grains(c, gen):
    """Seven kinds of grain with their own Ms, A and Ku1, a few per cent of the cells absent."""
    nz, ny, nx = c["nz"], c["ny"], c["nx"]
    Ms, A, _, _, _, _ = MATERIALS[c["material"]]
    gy, gx = max(2, ny // 12), max(2, nx // 12)
    kind = torch.randint(0, 7, (gy, gx), generator=gen, device="cuda")
    iy = torch.arange(ny, device="cuda") * gy // ny
    ix = torch.arange(nx, device="cuda") * gx // nx
    kind = kind[iy][:, ix].expand(nz, ny, nx)
    f = 0.85 + 0.05 * kind.double()
    hole = torch.rand((nz, ny, nx), generator=gen, device="cuda") < 0.03
    return {"Ms": torch.where(hole, 0.0, Ms * f), "A": A * f, "Ku1": 2e4 * kind.double()}


def _texture(shape, gen, amp=0.02):
    """A few long waves about a uniform direction, and white noise: a magnetic texture on its way to rest."""
    nz, ny, nx = shape
    z = torch.linspace(0, 1, nz, device="cuda").view(nz, 1, 1)
    y = torch.linspace(0, 1, ny, device="cuda").view(1, ny, 1)
    x = torch.linspace(0, 1, nx, device="cuda").view(1, 1, nx)
    out = torch.empty((3, nz, ny, nx), device="cuda")
    lean = torch.tensor([0.3, 0.2, 0.9], device="cuda")
    for d in range(3):
        w = torch.rand((3, 4), generator=gen, device="cuda")
        v = lean[d] * torch.ones((nz, ny, nx), device="cuda")
        for q in range(3):
            ph = 2 * math.pi * (w[q, 0] + (q + 1) * w[q, 1] * x + (q + 1) * w[q, 2] * y + 0.3 * w[q, 3] * z)
            v = v + 0.35 / (q + 1) * torch.cos(ph)
        out[d] = v + amp * torch.randn((nz, ny, nx), generator=gen, device="cuda")
    return out / out.norm(dim=0, keepdim=True)


def _inputs(c, seed):
    """(state: the tensors m of each replica, or of the one grid, per-cell materials, currents)."""
    gen = torch.Generator("cuda").manual_seed(int(seed))
    if c["kind"] == "batch":
        sizes = _edges(c)
        m, q = [], 0
        while q < len(sizes):
            n, r = sizes[q], sizes.count(sizes[q])
            v = torch.tensor([0.0, 0.0, 1.0], device="cuda").view(1, 3, 1, 1, 1) \
                + 0.1 * torch.randn((r, 3, 1, n, n), generator=gen, device="cuda")
            m.append(v / v.norm(dim=1, keepdim=True))
            q += r
        return m, {}, np.linspace(1e11, c["J"], c["R"])
    cells = _grains(c, gen) if c["grains"] else {}
    m = _texture((c["nz"], c["ny"], c["nx"]), gen)
    if c["precision"] == 64:
        m = m.double()
        m /= m.norm(dim=0, keepdim=True)
    if cells:
        m = m * (cells["Ms"] > 0).to(m.dtype)
    return m, cells, np.array([c["J"]])


class Simulation:
    """A context, the stream it runs on and the buffer its state is read into."""

    def __init__(self, ctx, out, steps):
        self.ctx, self.out, self.steps = ctx, out, steps
        self.stream = torch.cuda.Stream()
        mm.mm_set_stream(ctx, self.stream.cuda_stream)

    def __del__(self):
        torch.cuda.synchronize()
        mm.mm_destroy(self.ctx)


def prepare(case, seed):
    c = case
    Ms, A, alpha, Ku, D, B = MATERIALS[c["material"]]
    integrator = {"rk45": mm.MM_RK45, "rk4": mm.MM_RK4, "heun": mm.MM_HEUN, "dm": mm.MM_DM}[c["integrator"]]
    cell = [c[k] * 1e-9 for k in ("dx_nm", "dy_nm", "dz_nm")]
    m, cells, J = _inputs(c, seed)
    batch = c["kind"] == "batch"
    cfg = mm.make_config(precision=c["precision"], integrator=integrator,
                         demag=mm.MM_DEMAG_EXACT if c["demag"] else mm.MM_DEMAG_OFF, dt=c["dt"], dt_max=c["dt"],
                         rtol=1e-6, T=0.0 if batch else c["T"], seed=int(seed))
    mat = mm.Material(Ms, A, alpha, Ku, D=D, cells={k: v.cpu().numpy() for k, v in cells.items()})
    if batch:
        ctx = mm.mm_create_batch([mm.make_grid(e, e, 1, *cell) for e in _edges(c)], mat.s, cfg)
        mm.mm_set_temperature(ctx, np.full(c["R"], c["T"]))
        if c["demag"]:
            mm.mm_batch_set_shape(ctx, 0)      # the shape that the autotuner chooses for these ensembles
        m = torch.cat([v.reshape(-1) for v in m])
    else:
        ctx = mm.mm_create(mm.make_grid(c["nx"], c["ny"], c["nz"], *cell), mat.s, cfg)
        if any(B):
            mm.mm_set_field(ctx, 0, B)
    if c["J"]:
        mm.mm_set_torque(ctx, mm.make_torque(mm.MM_TORQUE_SOT, p=SOT_P, theta_SH=THETA_SH), J)
    s = Simulation(ctx, torch.empty_like(m), c["steps"])
    s.stream.wait_stream(torch.cuda.current_stream())
    mm.mm_set_m_device(ctx, m.data_ptr())
    s.stream.synchronize()
    return s


def run(state):
    mm.mm_step(state.ctx, state.steps)
    mm.mm_get_m_device(state.ctx, state.out.data_ptr())
    torch.cuda.current_stream().wait_stream(state.stream)
    return state.out


def work(case):
    """The state read and written once, the arithmetic of the zero-padded transforms, the tensor product and about
    150 operations per cell for the local field, torque and stage."""
    c = case
    per_step = {"rk45": 6, "rk4": 4, "heun": 2, "dm": 2}[c["integrator"]]
    grids = [(e, e, 1) for e in _edges(c)] if c["kind"] == "batch" else [(c["nx"], c["ny"], c["nz"])]
    flops, cells = 0.0, 0
    for nx, ny, nz in grids:
        cells += nx * ny * nz
        f = 150.0 * nx * ny * nz
        if c["demag"]:
            px, py, pz = 2 * nx, 2 * ny, 2 * nz if nz > 1 else 1
            kx = nx + 1
            f += 6 * (ny * nz * 2.5 * px * math.log2(px) + nz * kx * 5.0 * py * math.log2(py))
            if nz > 1:
                f += 6 * py * kx * 5.0 * pz * math.log2(pz)
            f += (30 if nz > 1 else 16) * py * kx * pz
        flops += f
    return {"bytes": 2.0 * 3 * cells * c["precision"] / 8, "flops": flops * per_step * c["steps"]}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _f(x, y, z):
    x, y, z = x.abs(), y.abs(), z.abs()
    R = (x * x + y * y + z * z).sqrt()

    def asinh(a, b):
        return torch.where(b > 0, torch.asinh(a / torch.where(b > 0, b, 1.0).sqrt()), 0.0)

    r = (2 * x * x - y * y - z * z) * R / 6
    r = r + 0.5 * y * (z * z - x * x) * asinh(y, x * x + z * z) + 0.5 * z * (y * y - x * x) * asinh(z, x * x + y * y)
    return r - x * y * z * torch.atan2(y * z, x * R)


def _g(x, y, z):
    z = z.abs()
    R = (x * x + y * y + z * z).sqrt()

    def asinh(a, b):
        return torch.where(b > 0, torch.asinh(a / torch.where(b > 0, b, 1.0).sqrt()), 0.0)

    def atan(a, b):
        return torch.where(b != 0, torch.atan(a / torch.where(b != 0, b, 1.0)), 0.0)

    r = x * y * z * asinh(z, x * x + y * y) + y * (3 * z * z - y * y) * asinh(x, y * y + z * z) / 6
    r = r + x * (3 * z * z - x * x) * asinh(y, x * x + z * z) / 6
    r = r - z ** 3 * atan(x * y, z * R) / 6 - 0.5 * z * y * y * atan(x * z, y * R) - 0.5 * z * x * x * atan(y * z, x * R)
    return r - x * y * R / 3


def _newell(nx, ny, nz, h):
    """The cell-averaged demagnetising tensor (xx yy zz xy xz yz) on the non-negative displacements: Newell's closed
    form within two cells, tent-weighted Gauss-Legendre quadrature of the dipole kernel beyond."""
    s = max(h)
    h = [v / s for v in h]
    k, j, i = torch.meshgrid(*(torch.arange(n, device="cuda", dtype=torch.float64) for n in (nz, ny, nx)), indexing="ij")
    P = [(i * h[0]).reshape(-1), (j * h[1]).reshape(-1), (k * h[2]).reshape(-1)]
    d = (P[0] ** 2 + P[1] ** 2 + P[2] ** 2).sqrt()
    out = torch.zeros((6, d.numel()), device="cuda", dtype=torch.float64)
    V = 4 * math.pi * h[0] * h[1] * h[2]
    at = (d <= 2.0).nonzero().reshape(-1)
    X, Y, Z = (p[at] for p in P)
    acc = torch.zeros((6, at.numel()), device="cuda", dtype=torch.float64)
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            for e in (-1, 0, 1):
                w = (2.0 if a == 0 else -1.0) * (2.0 if b == 0 else -1.0) * (2.0 if e == 0 else -1.0)
                x, y, z = X + a * h[0], Y + b * h[1], Z + e * h[2]
                acc += w * torch.stack([_f(x, y, z), _f(y, x, z), _f(z, y, x), _g(x, y, z), _g(x, z, y), _g(y, z, x)])
    out[:, at] = acc / V
    for lo, hi, n in ((2.0, 3.0, 16), (3.0, 8.0, 12), (8.0, 32.0, 6), (32.0, 128.0, 4), (128.0, 1e30, 3)):
        at = ((d > lo) & (d <= hi)).nonzero().reshape(-1)
        x, w = np.polynomial.legendre.leggauss(n)
        t1 = np.concatenate([(1 + x) / 2, -(1 + x) / 2])
        w1 = np.concatenate([w * (1 - x) / 4] * 2)
        t = torch.tensor(np.stack([v.ravel() for v in np.meshgrid(t1 * h[0], t1 * h[1], t1 * h[2], indexing="ij")]),
                         device="cuda")
        wt = torch.tensor(np.einsum("i,j,k->ijk", w1 * h[0] ** 2, w1 * h[1] ** 2, w1 * h[2] ** 2).ravel(), device="cuda")
        for part in at.split(max(1, (1 << 25) // wt.numel())):
            r = [P[q][part][:, None] + t[q][None, :] for q in range(3)]
            i2 = 1 / (r[0] ** 2 + r[1] ** 2 + r[2] ** 2)
            w3 = i2 * i2.sqrt() * wt
            w5 = 3 * w3 * i2
            iso = w3.sum(1)
            for q, (a, b) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
                out[q, part] = -((w5 * r[a] * r[b]).sum(1) - (iso if a == b else 0)) / V
    return out.reshape(6, nz, ny, nx)


class _Exact:
    """Field, slope and steps of one problem (or of R films of one size: a leading axis) in 64 bits."""

    def __init__(self, c, shape, cells, J, keys):
        self.c, self.shape, self.keys = c, shape, keys
        Ms, A, self.alpha, Ku, D, B = MATERIALS[c["material"]]
        self.h = [c[k] * 1e-9 for k in ("dx_nm", "dy_nm", "dz_nm")]
        full = lambda v: torch.full(shape, v, device="cuda", dtype=torch.float64)  # noqa: E731
        self.Ms, self.A, self.Ku = (cells.get(k, full(v)) for k, v in (("Ms", Ms), ("A", A), ("Ku1", Ku)))
        self.there = self.Ms > 0
        self.inv = torch.where(self.there, 1 / torch.where(self.there, MU0 * self.Ms, 1.0), 0.0)
        self.D, self.gm = D, GAMMA0 * MU0 / (1 + self.alpha ** 2)
        if c["kind"] == "batch":
            B = (0.0, 0.0, 0.0)
        self.Hext = torch.tensor(B, device="cuda", dtype=torch.float64).view(3, 1, 1, 1) / MU0
        self.sot = None
        if c["J"]:
            base = HBAR * torch.as_tensor(J, device="cuda").view(-1, 1, 1, 1) / (QE * MU0 * shape[0] * self.h[2])
            self.sot = 0.5 * THETA_SH * base * MU0 * self.inv
            self.p = torch.tensor(SOT_P, device="cuda", dtype=torch.float64).view(1, 3, 1, 1, 1)
        self.K = None
        if c["demag"]:
            nz, ny, nx = shape
            self.P = P = (2 * nz if nz > 1 else 1, 2 * ny, 2 * nx)
            N = _newell(nx, ny, nz, self.h)
            self.K = []
            for q, odd in enumerate(((), (), (), (2, 1), (2, 0), (1, 0))):     # odd axes of [z, y, x]
                k = torch.zeros(P, device="cuda", dtype=torch.float64)
                k[:nz, :ny, :nx] = N[q]
                for ax, n in ((0, nz), (1, ny), (2, nx)):
                    if n > 1:
                        src = k.narrow(ax, 1, n - 1).flip(ax)
                        k.narrow(ax, P[ax] - n + 1, n - 1).copy_(-src if ax in odd else src)
                self.K.append(torch.fft.rfftn(k).real.clone())
                del k

    def demag(self, m):
        nz, ny, nx = self.shape
        F = [torch.fft.rfftn(self.Ms * m[:, q], s=self.P, dim=(-3, -2, -1)) for q in range(3)]
        K, out = self.K, torch.empty_like(m)
        for q, row in enumerate(((0, 3, 4), (3, 1, 5), (4, 5, 2))):
            s = K[row[0]] * F[0] + K[row[1]] * F[1] + K[row[2]] * F[2]
            out[:, q] = -torch.fft.irfftn(s, s=self.P, dim=(-3, -2, -1))[:, :nz, :ny, :nx]
        return out

    def field(self, m, noise):
        H = self.Hext.expand_as(m).clone()
        H[:, 2] += 2 * self.Ku * self.inv * m[:, 2]
        diff = []
        for d in range(3):                                    # x, y, z
            ax, n = 4 - d, m.shape[4 - d]
            nbs = []
            for sg in (1, -1):
                nb = torch.roll(m, -sg, ax)
                A2, there2 = torch.roll(self.A, -sg, ax - 2), torch.roll(self.there, -sg, ax - 2).clone()
                there2.narrow(ax - 2, n - 1 if sg > 0 else 0, 1).fill_(False)
                c = torch.where(there2, 2 * self.A * A2 / (self.A + A2), self.A)
                g = m
                if self.D and d < 2:                          # free-edge ghost: m - h (D/2A) (z x n) x m
                    e = torch.zeros_like(m)
                    e[:, d], e[:, 2] = sg * m[:, 2], -sg * m[:, d]
                    g = m - self.h[d] * self.D / (2 * self.A) * e
                nb = torch.where(there2, nb, g)
                nbs.append(nb)
                H += 2 * c * self.inv / self.h[d] ** 2 * (nb - m)
            if self.D and d < 2:
                diff.append((nbs[0] - nbs[1]) / (2 * self.h[d]))
        if self.D:
            f = 2 * self.D * self.inv
            H[:, 0] += f * diff[0][:, 2]
            H[:, 1] += f * diff[1][:, 2]
            H[:, 2] -= f * (diff[0][:, 0] + diff[1][:, 1])
        if self.K is not None:
            H += self.demag(m)
        if noise is not None:
            H += noise
        return H

    def slope(self, m, noise=None, rotation=False):
        H = self.field(m, noise)
        x = torch.linalg.cross
        mH = x(m, H, dim=1)
        a = self.alpha
        k = self.gm * (H + a * mH) if rotation else -self.gm * (mH + a * x(m, mH, dim=1))
        if self.sot is not None:
            hdl = self.sot.unsqueeze(1)
            mp = x(m, self.p.expand_as(m), dim=1)
            k = k + (self.gm * hdl * (mp - a * self.p) if rotation else -self.gm * hdl * (x(m, mp, dim=1) - a * mp))
        return k * self.there

    def noise(self, step):
        c = self.c
        if not c["T"]:
            return None
        n = self.shape[0] * self.shape[1] * self.shape[2]
        M = 0xFFFFFFFF
        key = torch.tensor([[k & M, k >> 32] for k in self.keys], device="cuda")
        x = [torch.arange(n, device="cuda").expand(len(self.keys), n), step & M, step >> 32, 0]
        x = [v if torch.is_tensor(v) else torch.full_like(x[0], v) for v in x]
        k0, k1 = key[:, :1], key[:, 1:]

        def mul(a, b):
            lo, hi = a * (b & 0xFFFF), a * (b >> 16)
            return (hi + (lo >> 16)) >> 16, (lo + ((hi & 0xFFFF) << 16)) & M

        for _ in range(10):
            h0, l0 = mul(0xD2511F53, x[0])
            h1, l1 = mul(0xCD9E8D57, x[2])
            x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
            k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
        u = [((v >> 8) + 1).double() * 2.0 ** -24 for v in x]
        a, b = (-2 * u[0].log()).sqrt(), (-2 * u[2].log()).sqrt()
        g = torch.stack([a * (2 * math.pi * u[1]).cos(), a * (2 * math.pi * u[1]).sin(), b * (2 * math.pi * u[3]).cos()], 1)
        V = self.h[0] * self.h[1] * self.h[2]
        sigma = (2 * self.alpha * KB * c["T"] * self.inv / (MU0 * GAMMA0 * V * c["dt"])).sqrt()
        return sigma * g.reshape(-1, 3, *self.shape)

    def steps(self, m):
        dt, how = self.c["dt"], self.c["integrator"]

        def unit(v):
            n = v.norm(dim=1, keepdim=True)
            return v / torch.where(n > 0, n, 1.0)

        def turn(v, w):                                       # v rotated about w by |w| dt
            n = w.norm(dim=1, keepdim=True)
            e = w / torch.where(n > 0, n, 1.0)
            s, q = (n * dt).sin(), 2 * (n * dt / 2).sin() ** 2
            return v + s * torch.linalg.cross(e, v, dim=1) + q * ((e * v).sum(1, keepdim=True) * e - v)

        m, k1 = unit(m), None
        for n in range(self.c["steps"]):
            if how in ("heun", "dm"):
                th = self.noise(n)
                k1 = self.slope(m, th, how == "dm")
                k2 = self.slope(turn(m, k1) if how == "dm" else m + dt * k1, th, how == "dm")
                m = unit(turn(m, (k1 + k2) / 2) if how == "dm" else m + dt / 2 * (k1 + k2))
            elif how == "rk4":
                k1 = self.slope(m)
                k2 = self.slope(m + dt / 2 * k1)
                k3 = self.slope(m + dt / 2 * k2)
                m = unit(m + dt / 6 * (k1 + 2 * k2 + 2 * k3 + self.slope(m + dt * k3)))
            else:                                             # Dormand & Prince 5(4), first same as last
                k = [self.slope(m) if k1 is None else k1]
                for row in ((1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
                            (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
                            (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
                            (35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84)):
                    y = m + dt * sum(a * v for a, v in zip(row, k))
                    k.append(self.slope(y))
                m, k1 = unit(y), k[6]
        return m


def _splitmix64(x):
    x = (x + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
    x = ((x ^ (x >> 30)) * 0xBF58476D1CE4E5B9) & (2 ** 64 - 1)
    x = ((x ^ (x >> 27)) * 0x94D049BB133111EB) & (2 ** 64 - 1)
    return x ^ (x >> 31)


def exact(case, seed):
    c = case
    m, cells, J = _inputs(c, seed)
    if c["kind"] == "one":
        e = _Exact(c, (c["nz"], c["ny"], c["nx"]), cells, J, [_splitmix64(int(seed))])
        return e.steps(m.double().unsqueeze(0))[0]
    out, r = [], 0
    for v in m:
        n = v.shape[0]
        e = _Exact(c, tuple(v.shape[2:]), {}, J[r:r + n], [_splitmix64(int(seed) + q) for q in range(r, r + n)])
        out.append(e.steps(v.double()).reshape(-1))
        r += n
    return torch.cat(out)
