"""Performance cases: what a program that uses the library has it do, from the
smallest calls to the largest grids, through the package's public entry points.

``listed()`` gives the named cases, ``draw(rng)`` one more of the same ranges;
``prepare(case, seed)`` makes what a program holds before the call (solvers,
fields on the GPU), ``run(state)`` is one pass, ``work(case)`` what a pass cannot
do without, and ``exact(case, seed)`` the same outputs from a plain torch FP64
restatement of the scheme (no library code).

Every field is a seeded smooth state of a developed flow plus white noise.  A
pass starts from that state and hands back the state after the case's steps, so
it can be repeated.  The mixed mode's states carry single-precision increments;
the programs that use it keep their snapshots in float32, and so do its passes.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2004_13887_gb300 as sph

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # The parity configuration: a forced manufactured flow on 32^3 cells in
        # FP64, one step at a time with its residual read back -- a convergence
        # study, where launches and short serial lines count.
        dict(name="mms_32_fp64", kind="step", flow="mms", precision="fp64", nr=32, nt=32, np=32, steps=1,
             source=True, walls=False, wait=True),
        # The paper's low-Mach table: its domain at grid diameter 0.12, odd
        # extents, forcing, and wall velocities that move and are handed over
        # before every step.
        dict(name="walls_14x45x135_fp64", kind="step", flow="paper", precision="fp64", nr=14, nt=45, np=135, steps=1,
             source=True, walls=True, wait=True),
        # The smallest bubble of an ensemble, stepped on its own in mixed
        # precision: latency.
        dict(name="bubble_16x64x64_mixed", kind="step", flow="bubble", precision="mixed", nr=16, nt=64, np=64, steps=4,
             source=False, walls=False, wait=False),
        # The benchmark workload: the rising bubble on 128 x 256 x 256 cells.
        dict(name="bubble_128x256x256_mixed", kind="step", flow="bubble", precision="mixed", nr=128, nt=256, np=256,
             steps=2, source=False, walls=False, wait=False),
        # Thermal 1 on the paper's 100 x 200 x 200 cells: extents that are not
        # powers of two.
        dict(name="thermal_100x200x200_mixed", kind="step", flow="bubble", precision="mixed", nr=100, nt=200, np=200,
             steps=2, source=False, walls=False, wait=False),
        # The benchmark workload in plain FP64.
        dict(name="bubble_128x256x256_fp64", kind="step", flow="bubble", precision="fp64", nr=128, nt=256, np=256,
             steps=1, source=False, walls=False, wait=False),
        # The full sphere with poles and periodic phi, mixed precision: the
        # largest grid.
        dict(name="shell_64x512x1024_mixed", kind="step", flow="shell", precision="mixed", nr=64, nt=512, np=1024,
             steps=2, source=False, walls=False, wait=False),
        # A coarse full sphere in FP64: cyclic lines.
        dict(name="shell_32x128x256_fp64", kind="step", flow="shell", precision="fp64", nr=32, nt=128, np=256, steps=1,
             source=False, walls=False, wait=False),
        # Backward: the adjoint of one step on a small bubble, as in a gradient
        # check ...
        dict(name="adjoint_16x32x32", kind="adjoint", flow="bubble", nr=16, nt=32, np=32),
        # ... and on the gradient workload's 96 x 192 x 192 cells.
        dict(name="adjoint_96x192x192", kind="adjoint", flow="bubble", nr=96, nt=192, np=192),
        # An ensemble of independent bubbles on uneven grids, batched launches
        # in one CUDA graph.
        dict(name="ensemble_12_mixed", kind="batch", flow="bubble", count=12, grids=20041389, fused=True, replays=1),
        # The stand-alone block-tridiagonal solve on systems the caller
        # assembled.
        dict(name="lines_1024x128", kind="lines", nlines=1024, n=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extent(rng, lo, hi):
    """a length of lo..hi cells: any, or a multiple of 16 as most grids have"""
    n = _log_int(rng, lo, hi)
    return max(lo, min(hi, 16 * round(n / 16))) if rng.random() < 0.5 and hi >= 32 else n


def draw(rng):
    """one more case: the listed ones' kinds over their ranges of sizes"""
    what = rng.choice(["bubble_mixed", "bubble_mixed", "bubble_fp64", "mms", "walls", "shell", "adjoint", "batch",
                       "lines"])
    step = dict(kind="step", steps=rng.choice([1, 2, 3]), source=False, walls=False, wait=False)
    if what.startswith("bubble"):
        return dict(step, flow="bubble", precision=what.split("_")[1], nr=_extent(rng, 8, 128),
                    nt=_extent(rng, 24, 256), np=_extent(rng, 24, 256))
    if what == "mms":
        return dict(step, flow="mms", precision=rng.choice(["fp64", "mixed"]), source=True, wait=True, steps=1,
                    nr=_extent(rng, 5, 48), nt=_extent(rng, 6, 64), np=_extent(rng, 7, 64))
    if what == "walls":
        return dict(step, flow="paper", precision="fp64", source=True, walls=True, wait=True, steps=1,
                    nr=_extent(rng, 6, 24), nt=_extent(rng, 8, 64), np=_extent(rng, 24, 160))
    if what == "shell":
        if rng.random() < 0.5:
            return dict(step, flow="shell", precision="mixed", nr=_extent(rng, 8, 64), nt=_extent(rng, 32, 512),
                        np=rng.choice([_extent(rng, 64, 700), 256, 512, 1024]))
        return dict(step, flow="shell", precision="fp64", nr=_extent(rng, 8, 48), nt=_extent(rng, 16, 160),
                    np=_extent(rng, 32, 320))
    if what == "adjoint":
        return dict(kind="adjoint", flow=rng.choice(["bubble", "bubble", "shell"]), nr=_extent(rng, 6, 64),
                    nt=_extent(rng, 10, 128), np=_extent(rng, 12, 128))
    if what == "batch":
        return dict(kind="batch", flow="bubble", count=rng.randint(3, 12), grids=rng.randrange(1 << 30),
                    fused=rng.random() < 0.5, replays=1)
    n = _log_int(rng, 3, 512)
    return dict(kind="lines", n=n, nlines=_log_int(rng, 8, 131072 // n))


K = 2                   # Picard iterations a step, as in every workload


# ---------------------------------------------------------------------------
# grids, constants and fields

class Grid:
    """a sector [r1,r2] x [t1,t2] x [p1,p2] of nr x nt x np uniform cells"""

    def __init__(self, n, r, t, p, periodic=False):
        self.nr, self.nt, self.np = n
        (self.r1, self.r2), (self.t1, self.t2), (self.p1, self.p2) = r, t, p
        self.periodic = periodic
        self.npf = self.np + (not periodic)

    def shapes(self):
        nr, nt, n = self.nr, self.nt, self.np
        return [(nr, nt, n), (nr + 1, nt, n), (nr, nt + 1, n), (nr, nt, self.npf), (nr, nt, n)]

    def wall_shape(self, c, d):
        return tuple(s for a, s in enumerate(self.shapes()[1 + c]) if a != d)

    def axes(self, f):
        """the unit-interval coordinates of field f along each axis, broadcastable"""
        out = []
        for a, n in enumerate((self.nr, self.nt, self.np)):
            face = f == 1 + a
            m = self.shapes()[f][a]
            x = (torch.arange(m, dtype=F64, device=DEV) + (0.0 if face else 0.5)) / n
            out.append(x.reshape([-1 if b == a else 1 for b in range(3)]))
        return out


AIR = dict(gamma=1000.0 / 713.0, cv=713.0, Pr=0.71, mu=1.846e-5, pinf=0.0, omega=0.0)
GAS = dict(gamma=1.6, cv=1.0, Pr=1.0, mu=1.0, pinf=0.0, g=0.0, omega=0.0)   # the manufactured flows' unit gas


def _setting(flow, n):
    """(grid, constants, background p and T of nr + 2 values, time step, speed,
    pressure and temperature scales) of a flow"""
    nr = n[0]
    if flow == "bubble":
        half = 10.0 / 6371.0
        grid = Grid(n, (6371e3, 6381e3), (math.pi / 2 - half, math.pi / 2 + half), (math.pi - half, math.pi + half))
        dr, cp, Rg, g = (grid.r2 - grid.r1) / nr, 1000.0, 287.0, 9.80665
        exner = 1.0 - g * (np.arange(-1, nr + 1) + 0.5) * dr / (cp * 300.0)
        T = 300.0 * exner
        p = np.empty(nr + 2)       # discretely hydrostatic: the rest state is an equilibrium
        p[0] = 1e5 * exner[0] ** (cp / Rg)
        for m in range(1, nr + 2):
            p[m] = p[m - 1] * (1.0 - g * dr / (2 * Rg * T[m - 1])) / (1.0 + g * dr / (2 * Rg * T[m]))
        return grid, SimpleNamespace(**AIR, g=g), (p, T), 1.0, 3.0, 5.0, 0.5
    if flow == "shell":
        grid = Grid(n, (6371e3, 6381e3), (0.0, math.pi), (0.0, 2 * math.pi), periodic=True)
        return grid, SimpleNamespace(**AIR, g=0.0), (np.full(nr + 2, 1e5), np.full(nr + 2, 300.0)), 1.0, 0.035, 5.0, 5e-3
    T0 = 6250.0 / 0.6
    bg = (np.full(nr + 2, 6250.0), np.full(nr + 2, T0))
    if flow == "paper":
        grid = Grid(n, (1.0, 2.0), (math.pi / 4, 3 * math.pi / 4), (math.pi / 4, 7 * math.pi / 4))
    else:
        grid = Grid(n, (637.1, 638.1), (math.pi / 4, 3 * math.pi / 4), (0.0, math.pi / 2))
    return grid, SimpleNamespace(**GAS), bg, 1e-3, 1.0, 1.0, 1.0


def _fields(grid, scales, gen, at_walls=False, noise=1e-3):
    """five smooth seeded fields of the given scales (p, u, T) plus white noise;
    velocities vanish on every wall and pole unless at_walls"""
    out = []
    cpu = torch.Generator().manual_seed(int(torch.randint(1 << 31, (1,), generator=gen, device=DEV).item()))
    for f, shape in enumerate(grid.shapes()):
        x = grid.axes(f)
        v = torch.zeros(shape, dtype=F64, device=DEV)
        for _ in range(3):
            a = torch.randn(1, generator=cpu).item()
            m = torch.randint(0, 3, (3,), generator=cpu).tolist()
            ph = (torch.rand(3, generator=cpu) * 2 * math.pi).tolist()
            term = a
            for q in range(3):
                wave = 2 if q == 2 and grid.periodic else 1
                term = term * torch.cos(wave * math.pi * m[q] * x[q] + ph[q])
            v += term
        v *= 1 + noise * torch.randn(shape, dtype=F64, device=DEV, generator=gen)
        if 1 <= f <= 3 and not at_walls:
            for q in range(3):
                if not (q == 2 and grid.periodic):
                    v *= torch.sin(math.pi * x[q])
        out.append(v * (scales[1] if 1 <= f <= 3 else scales[0] if f == 0 else scales[2]))
    if not at_walls:
        out[1][0] = out[1][-1] = 0.0
        out[2][:, 0] = out[2][:, -1] = 0.0
        if not grid.periodic:
            out[3][:, :, 0] = out[3][:, :, -1] = 0.0
    return out


def _walls(grid, U, scale, gen):
    """wall velocities at t^n (U's own normal faces) and t^{n+1}: {(c, d, s): tensor}"""
    now, then = {}, {}
    for c in range(3):
        for d in range(3):
            for s in range(2):
                if c == d:
                    w = U[1 + c].select(d, s * (U[1 + c].shape[d] - 1)).contiguous()
                else:
                    w = U[1 + c].select(d, s * (U[1 + c].shape[d] - 1)).contiguous() * 0.5
                now[(c, d, s)] = w
                then[(c, d, s)] = w + 1e-3 * scale * torch.randn(w.shape, dtype=F64, device=DEV, generator=gen)
    return now, then


def _inputs(flow, n, seed, source=False, walls=False):
    grid, par, bg, dt, u, p, T = _setting(flow, n)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    U = _fields(grid, (p, u, T), gen, at_walls=walls)
    if flow == "bubble":        # the warm anomaly: a Gaussian in the lower half of the sector
        amp, size, alt = (torch.rand(3, generator=gen, device=DEV, dtype=F64) * torch.tensor([0.8, 0.1, 0.1], device=DEV)
                          + torch.tensor([0.2, 0.15, 0.25], device=DEV)).tolist()
        x = grid.axes(4)
        U[4] = 0.02 * U[4] + amp * torch.exp(-((x[0] - alt) ** 2 + 4 * (x[1] - 0.5) ** 2 + 4 * (x[2] - 0.5) ** 2)
                                             / size ** 2)
    S = _fields(grid, (10 * p, u, 10 * T), gen, at_walls=True) if source else None
    W = _walls(grid, U, u, gen) if walls else None
    return SimpleNamespace(grid=grid, par=par, bg=bg, dt=dt, U=U, S=S, W=W)


def _batch_grids(case):
    """the uneven grids of an ensemble: nr in {16, 32, 48, 64}, nt and np in {64, 128, 192, 256}"""
    rng = np.random.default_rng(case["grids"])
    return [(int(rng.choice([16, 32, 48, 64])), int(rng.choice([64, 128, 192, 256])),
             int(rng.choice([64, 128, 192, 256]))) for _ in range(case["count"])]


def _systems(case, seed):
    """diagonally dominant 3x3-block tridiagonal lines, as I + tau/2 D is"""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    nl, n = case["nlines"], case["n"]
    A, B, C = (0.2 * torch.randn((nl, n, 3, 3), dtype=F64, device=DEV, generator=gen) for _ in range(3))
    B += 2.0 * torch.eye(3, dtype=F64, device=DEV)
    return A, B, C, torch.randn((nl, n, 3), dtype=F64, device=DEV, generator=gen)


# ---------------------------------------------------------------------------
# what a program has in hand, and a pass

def _solver(p, precision, stream=None):
    s = sph.Solver(p.grid, p.par, precision=sph.SPH_PREC_MIXED if precision == "mixed" else sph.SPH_PREC_FP64,
                   stream=stream)
    s.set_background(*p.bg)
    return s


def prepare(case, seed):
    if case["kind"] == "lines":
        return SimpleNamespace(kind="lines", systems=_systems(case, seed))
    if case["kind"] == "batch":
        ps = [_inputs("bubble", n, seed * 64 + q) for q, n in enumerate(_batch_grids(case))]
        solvers = [_solver(p, "mixed", torch.cuda.Stream()) for p in ps]
        for s, p in zip(solvers, ps):
            s.set_state(p.U)
        torch.cuda.synchronize()
        batch = sph.Batch(solvers)
        batch.capture(1.0, K, 2, fused=case["fused"])
        return SimpleNamespace(kind="batch", ps=ps, solvers=solvers, batch=batch, replays=case["replays"],
                               out=[s.empty() for s in solvers])
    if case["kind"] == "adjoint":
        p = _inputs(case["flow"], (case["nr"], case["nt"], case["np"]), seed)
        gen = torch.Generator(device=DEV).manual_seed(seed + 1)
        lam = _fields(p.grid, (1.0, 1.0, 1.0), gen)
        s = _solver(p, "fp64")
        return SimpleNamespace(kind="adjoint", p=p, solver=s, lam=lam)
    p = _inputs(case["flow"], (case["nr"], case["nt"], case["np"]), seed, case["source"], case["walls"])
    s = _solver(p, case["precision"])
    return SimpleNamespace(kind="step", p=p, solver=s, steps=case["steps"], wait=case["wait"],
                           mixed=case["precision"] == "mixed", out=s.empty())


def run(state):
    if state.kind == "lines":
        return sph.block_thomas_noalloc(*state.systems)
    if state.kind == "batch":
        for s, p in zip(state.solvers, state.ps):
            s.set_state(p.U)
            state.batch.stream.wait_stream(s.stream)
        state.batch.launch(state.replays)
        state.batch.status()
        return [[f.float() for f in s.get_state(out=o)] for s, o in zip(state.solvers, state.out)]
    p, s = state.p, state.solver
    if state.kind == "adjoint":
        s.set_state(p.U)
        return s.step_adjoint(p.dt, K, state.lam)
    s.set_state(p.U)
    residual = None
    for _ in range(state.steps):
        if p.W is not None:
            s.set_bc(*p.W)
        if state.wait:      # a study that looks at every step's residual
            residual = s.step(p.dt, K, p.S, residual=True)
        else:
            s.step_async(p.dt, K, p.S)
    if not state.wait:
        s.status()
    out = s.get_state(out=state.out)
    if state.mixed:
        return [f.float() for f in out]
    return out if residual is None else list(out) + [residual.astype(np.float32)]


def _points(case):
    if case["kind"] == "batch":
        return sum(a * b * c for a, b, c in _batch_grids(case))
    return case["nr"] * case["nt"] * case["np"]


def work(case):
    """The state (five doubles a point) read and written once a step's state
    hand-over, the forcing read; about 1000 operations a point for an
    iteration's operator and 900 for its line solves, three times that for the
    adjoint of an iteration beside the forward it needs."""
    if case["kind"] == "lines":
        m = case["nlines"] * case["n"]
        return {"bytes": 8.0 * 33 * m, "flops": 190.0 * m}
    n = _points(case)
    if case["kind"] == "adjoint":
        return {"bytes": 8.0 * 15 * n, "flops": 4.0 * K * 1900 * n}
    steps = 2 * case["replays"] if case["kind"] == "batch" else case["steps"]
    return {"bytes": 8.0 * (10 + 5 * bool(case.get("source"))) * n, "flops": float(K * steps * 1900 * n)}


# ---------------------------------------------------------------------------
# the scheme in plain torch, FP64: Picard iterations of
#   R = -(U^k - U^n) - dt [N(Ubar) + G - S],  Ubar = (U^k + U^n)/2,
#   (I + dt/2 D_r)(I + dt/2 D_theta)(I + dt/2 D_phi) x = R,  U^{k+1} = U^k + x
# on the MAC grid, with D_d and N frozen at Ubar.

def exact(case, seed):
    if case["kind"] == "lines":
        A, B, C, d = (v.movedim(1, 0) for v in _systems(case, seed))
        return torch.stack(_thomas(A, B, C, d.unsqueeze(-1)), 1).squeeze(-1)
    if case["kind"] == "batch":
        out = []
        for q, n in enumerate(_batch_grids(case)):
            p = _inputs("bubble", n, seed * 64 + q)
            U = p.U
            for _ in range(2 * case["replays"]):
                U = _Ref(p).step(U)[0]
            out.append(U)
        return out
    if case["kind"] == "adjoint":
        if _points(case) > 600_000:      # autograd would keep some hundreds of fields an iteration
            return None
        p = _inputs(case["flow"], (case["nr"], case["nt"], case["np"]), seed)
        gen = torch.Generator(device=DEV).manual_seed(seed + 1)
        lam = _fields(p.grid, (1.0, 1.0, 1.0), gen)
        U = [u.clone().requires_grad_(True) for u in p.U]
        out = _Ref(p).step(U)[0]
        return list(torch.autograd.grad(out, U, lam))
    p = _inputs(case["flow"], (case["nr"], case["nt"], case["np"]), seed, case["source"], case["walls"])
    U, res = p.U, None
    with torch.no_grad():
        for _ in range(case["steps"]):
            U, res = _Ref(p).step(U)
    return list(U) + [res] if case["wait"] and case["precision"] == "fp64" else list(U)


def _thomas(A, B, C, d):
    """block Thomas over the first axis; A, B, C (n, lines, b, b), d (n, lines, b, k)"""
    one = B.shape[-1] == 1
    E, g = [], []
    for m in range(B.shape[0]):
        S, y = (B[m], d[m]) if m == 0 else (B[m] - A[m] @ E[-1], d[m] - A[m] @ g[-1])
        r = torch.cat([C[m], y], -1)
        r = r / S if one else torch.linalg.solve_ex(S, r)[0]
        E.append(r[..., :B.shape[-1]])
        g.append(r[..., B.shape[-1]:])
    x = [g[-1]]
    for m in range(B.shape[0] - 2, -1, -1):
        x.append(g[m] - E[m] @ x[-1])
    return x[::-1]


def _cyclic(A, B, C, d):
    """the same with A[0] coupling to the last cell and C[-1] to the first"""
    n = B.shape[0]
    z = torch.zeros_like(B[0])
    e = torch.stack([A[0]] + [z] * (n - 3) + [C[n - 2]])
    s = _thomas(A[:-1], B[:-1], C[:-1], torch.cat([d[:-1], e], -1))
    k = d.shape[-1]
    y0, Z0, y1, Z1 = s[0][..., :k], s[0][..., k:], s[-1][..., :k], s[-1][..., k:]
    S = B[-1] - C[-1] @ Z0 - A[-1] @ Z1
    r = d[-1] - C[-1] @ y0 - A[-1] @ y1
    last = r / S if B.shape[-1] == 1 else torch.linalg.solve_ex(S, r)[0]
    return [v[..., :k] - v[..., k:] @ last for v in s] + [last]


def _ax(v, a):
    return v.reshape([-1 if b == a else 1 for b in range(3)])


class _Ref:
    def __init__(self, p):
        self.p, g = p, p.grid
        self.n = (g.nr, g.nt, g.np)
        self.per = (False, False, g.periodic)
        lo, hi = (g.r1, g.t1, g.p1), (g.r2, g.t2, g.p2)
        self.h = [(b - a) / n for a, b, n in zip(lo, hi, self.n)]
        cen = [a + (torch.arange(n, dtype=F64, device=DEV) + 0.5) * h for a, n, h in zip(lo, self.n, self.h)]
        fac = [a + torch.arange(n + 1, dtype=F64, device=DEV) * h for a, n, h in zip(lo, self.n, self.h)]
        self.rc, self.rf = _ax(cen[0], 0), _ax(fac[0], 0)
        sin_f = torch.sin(fac[1])
        if g.t1 < 1e-14:
            sin_f[0] = 0.0
        if abs(g.t2 - math.pi) < 1e-14:
            sin_f[-1] = 0.0
        self.sc, self.sf = _ax(torch.sin(cen[1]), 1), _ax(sin_f, 1)
        self.cc, self.cf = _ax(torch.cos(cen[1]), 1), _ax(torch.cos(fac[1]), 1)
        bp, bT = (torch.as_tensor(v, dtype=F64, device=DEV) for v in p.bg)
        self.pref, self.Tref = _ax(bp[1:-1], 0), _ax(bT[1:-1], 0)
        self.dbp, self.dbT = _ax(bp[2:] - bp[:-2], 0), _ax(bT[2:] - bT[:-2], 0)
        f2 = fac[0] ** 2
        self.lapT = _ax((f2[1:] * (bT[2:] - bT[1:-1]) - f2[:-1] * (bT[1:-1] - bT[:-2])) / (cen[0] ** 2 * self.h[0] ** 2), 0)
        Rg = p.par.cv * (p.par.gamma - 1)
        rho = (bp + p.par.pinf) / (Rg * bT)
        # the background's hydrostatic residual on the interior r-faces
        self.ehyd = _ax((bp[2:-1] - bp[1:-2]) / (self.h[0] * 0.5 * (rho[1:-2] + rho[2:-1])) + p.par.g, 0)
        self.Rg, self.kappa = Rg, p.par.mu * p.par.gamma * p.par.cv / p.par.Pr
        w = p.W
        self.wall = {k: 0.5 * (w[0][k] + w[1][k]) for k in w[0]} if w else {}

    # ---- moves between centres and faces, ghosts
    def lohi(self, u, a):
        """the values of a face field on the two a-faces of every cell"""
        if self.per[a]:
            return u, torch.roll(u, -1, a)
        return u.narrow(a, 0, self.n[a]), u.narrow(a, 1, self.n[a])

    def sides(self, f, a):
        """the two cells of every unknown a-face (interior, or all when periodic)"""
        if self.per[a]:
            return torch.roll(f, 1, a), f
        m = f.shape[a] - 1
        return f.narrow(a, 0, m), f.narrow(a, 1, m)

    def inner(self, u, a):
        return u if self.per[a] else u.narrow(a, 1, u.shape[a] - 2)

    def nb_c(self, f, a):
        """neighbours of a centre field along a: zero-gradient ghosts"""
        if self.per[a]:
            return torch.roll(f, 1, a), torch.roll(f, -1, a)
        n = f.shape[a]
        return (torch.cat([f.narrow(a, 0, 1), f.narrow(a, 0, n - 1)], a),
                torch.cat([f.narrow(a, 1, n - 1), f.narrow(a, n - 1, 1)], a))

    def nb_v(self, u, c, a):
        """neighbours of velocity component c along a transverse direction:
        ghost = 2 wall - interior"""
        if self.per[a]:
            return torch.roll(u, 1, a), torch.roll(u, -1, a)
        n = u.shape[a]
        gh = []
        for s in range(2):
            e = u.narrow(a, s * (n - 1), 1)
            w = self.wall.get((c, a, s))
            gh.append(-e if w is None else 2 * w.unsqueeze(a) - e)
        return (torch.cat([gh[0], u.narrow(a, 0, n - 1)], a), torch.cat([u.narrow(a, 1, n - 1), gh[1]], a))

    def mid(self, u, a):
        lo, hi = self.lohi(u, a)
        return 0.5 * (lo + hi)

    # ---- everything frozen at Ubar
    def freeze(self, U):
        P, V, T = U[0], U[1:4], U[4]
        par, h = self.p.par, self.h
        q = SimpleNamespace(V=V, P=P, T=T)
        q.Pb, q.Tb = P + self.pref + par.pinf, T + self.Tref
        q.rho = q.Pb / (self.Rg * q.Tb)
        q.beta = (par.gamma - 1) * q.Tb / q.Pb
        q.drho = (P * self.Tref - (self.pref + par.pinf) * T) / (self.Rg * self.Tref * q.Tb)
        q.uc = [self.mid(V[a], a) for a in range(3)]
        lh = [self.lohi(V[a], a) for a in range(3)]
        q.lh = lh
        r, s = self.rc, self.sc
        cot = self.cc / s
        m = (1.0, 1 / r, 1 / (r * s))          # metric factors of the three derivatives at centres
        d = [(lh[a][1] - lh[a][0]) / h[a] * m[a] for a in range(3)]
        q.G = [d[0], d[1] + q.uc[0] / r, d[2] + q.uc[0] / r + q.uc[1] * cot / r]
        def der(c, a):                          # centred derivative along a of the centre average of component c
            lo, hi = self.nb_v(V[c], c, a)
            return self.mid(hi - lo, c) * 0.5 / h[a] * m[a]
        q.x = [der(1, 0) + der(0, 1), der(2, 0) + der(0, 2), der(2, 1) + der(1, 2)]
        q.s = [q.x[0] - q.uc[1] / r, q.x[1] - q.uc[2] / r, q.x[2] - q.uc[2] * cot / r]
        f2 = self.rf ** 2
        q.div = [(f2[1:] * lh[0][1] - f2[:-1] * lh[0][0]) / (r * r * h[0]),
                 (self.sf[:, 1:] * lh[1][1] - self.sf[:, :-1] * lh[1][0]) / (r * s * h[1]), d[2]]
        return q

    def rows_c(self, q, a, isT):
        """p- or T-row of D_a at the centres: advection, T weights (m-1, m, m+1),
        the two u_a couplings split as (a, g0, g1, w0, w1)"""
        par, h, r, s = self.p.par, self.h, self.rc, self.sc
        g1 = par.gamma - 1
        vis = par.mu * q.beta if isT else par.mu * g1
        al = g1 * q.Tb if isT else par.gamma * q.Pb
        dif = self.kappa * (q.beta if isT else g1)
        al = al + 2.0 / 3.0 * vis * (q.G[0] + q.G[1] + q.G[2])
        if a == 0:
            f0, f1, m, k = self.rf[:-1] ** 2, self.rf[1:] ** 2, 1.0 / h[0], 1 / (r * r)
            lin = -vis * (q.G[1] + q.G[2]) / r
        elif a == 1:
            f0, f1, m, k = self.sf[:, :-1], self.sf[:, 1:], 1 / (r * h[1]), 1 / s
            lin = -vis * (2 * q.G[2] * self.cc / s - q.s[0]) * 0.5 / r
        else:
            f0 = f1 = torch.ones((), dtype=F64, device=DEV)
            m, k = 1 / (r * s * h[2]), 1.0
            lin = vis * (q.s[1] + q.s[2] * self.cc / s) * 0.5 / r
        m0 = 2 * vis * q.G[a] * m
        adv, dd = 0.5 * q.uc[a] * m, -dif * m * m * k
        return adv, (dd * f0, -dd * (f0 + f1), dd * f1), al, (-f0 * k * m, f1 * k * m), (m0 + lin, -m0 + lin), dif

    def rows_f(self, q, a):
        """normal-velocity row of D_a on its unknown faces: p weight, u weights"""
        par, h = self.p.par, self.h
        r0, r1 = self.sides(q.rho, a)
        ir = 2 / (r0 + r1)
        if a == 0:
            f, c2 = self.rf, self.rc ** 2
            m = 1 / h[0]
            nu = -par.mu * ir * m * m
            lap, gd = nu / f[1:-1] ** 2, nu / 3.0
            w = (lap * c2[:-1] + gd * f[:-2] ** 2 / c2[:-1],
                 -lap * (c2[:-1] + c2[1:]) - gd * f[1:-1] ** 2 * (1 / c2[1:] + 1 / c2[:-1]),
                 lap * c2[1:] + gd * f[2:] ** 2 / c2[1:])
        elif a == 1:
            f, c1 = self.sf, self.sc
            m = 1 / (self.rc * h[1])
            nu = -par.mu * ir * m * m
            lap, gd = nu / f[:, 1:-1], nu / 3.0
            w = (lap * c1[:, :-1] + gd * f[:, :-2] / c1[:, :-1],
                 -lap * (c1[:, :-1] + c1[:, 1:]) - gd * f[:, 1:-1] * (1 / c1[:, 1:] + 1 / c1[:, :-1]),
                 lap * c1[:, 1:] + gd * f[:, 2:] / c1[:, 1:])
        else:
            m = 1 / (self.rc * self.sc * h[2])
            lap = -4.0 / 3.0 * par.mu * ir * m * m
            w = (lap, -2 * lap, lap)
        adv = 0.5 * self.inner(q.V[a], a) * m
        return ir * m, (w[0] - adv, w[1], w[2] + adv), ir

    def rows_s(self, q, c, a):
        """row of component c along a transverse direction a on its unknown faces"""
        par, h = self.p.par, self.h
        r0, r1 = self.sides(q.rho, c)
        ir = 2 / (r0 + r1)
        u0, u1 = self.sides(q.uc[a], c)
        r = self.rf[1:-1] if c == 0 else self.rc
        s = self.sf[:, 1:-1] if c == 1 else self.sc
        if a == 0:
            m, k, f0, f1 = 1 / h[0], 1 / (r * r), self.rf[:-1] ** 2, self.rf[1:] ** 2
        elif a == 1:
            m, k, f0, f1 = 1 / (r * h[1]), 1 / s, self.sf[:, :-1], self.sf[:, 1:]
        else:
            m, k = 1 / (r * s * h[2]), 1.0
            f0 = f1 = torch.ones((), dtype=F64, device=DEV)
        adv, lap = 0.25 * (u0 + u1) * m, -par.mu * ir * m * m * k
        return -adv + lap * f0, -lap * (f0 + f1), adv + lap * f1

    def rhs(self, q, D, S):
        """R = -D - dt (N(Ubar) + G - S); zero on the wall faces"""
        par, h, r, s = self.p.par, self.h, self.rc, self.sc
        V, out, div = q.V, [], q.div[0] + q.div[1] + q.div[2]
        cross = sum(a * b for a, b in zip(q.s, q.x))
        for isT in (False, True):
            acc = -par.mu * (q.beta if isT else par.gamma - 1) * cross
            for a in range(3):
                adv, wT, al, _, wv, dif = self.rows_c(q, a, isT)
                tl, th = self.nb_c(q.T, a)
                fl, fh = (tl, th) if isT else self.nb_c(q.P, a)
                acc = acc + adv * (fh - fl) + wT[0] * tl + wT[1] * q.T + wT[2] * th
                acc = acc + wv[0] * q.lh[a][0] + wv[1] * q.lh[a][1]
                if a == 0:
                    acc = acc + adv * (self.dbT if isT else self.dbp) - dif * self.lapT
            out.append(al * div + acc)
        N = [out[0]]
        for c in range(3):
            wp, wu, ir = self.rows_f(q, c)
            p0, p1 = self.sides(q.P, c)
            u = self.inner(V[c], c)
            if self.per[c]:
                um, up = torch.roll(V[c], 1, c), torch.roll(V[c], -1, c)
            else:
                um, up = V[c].narrow(c, 0, V[c].shape[c] - 2), V[c].narrow(c, 2, V[c].shape[c] - 2)
            acc = wp * (p1 - p0) + wu[0] * um + wu[1] * u + wu[2] * up
            for a in range(3):
                if a != c:
                    w = self.rows_s(q, c, a)
                    lo, hi = (self.inner(v, c) for v in self.nb_v(V[c], c, a))
                    acc = acc + w[0] * lo + w[1] * u + w[2] * hi
            at = lambda f: (lambda z: 0.5 * (z[0] + z[1]))(self.sides(f, c))          # noqa: E731
            jump = lambda f: (lambda z: z[1] - z[0])(self.sides(f, c))                # noqa: E731
            mu, om = par.mu * ir, par.omega
            if c == 0:
                rf = self.rf[1:-1]
                b = at(q.drho) / at(q.rho)
                Q = q.div[1] + q.div[2]
                acc = acc + (1 - b) * self.ehyd + par.g * b - (at(q.uc[1]) ** 2 + at(q.uc[2]) ** 2) / rf
                acc = acc + 2 * mu * u / rf ** 2 - 2 * om * s * at(q.uc[2]) - mu / 3 * jump(Q) / h[0] + 2 * mu * at(Q) / rf
            elif c == 1:
                sf, cf = self.sf[:, 1:-1], self.cf[:, 1:-1]
                acc = acc + u * at(q.uc[0]) / r - at(q.uc[2]) ** 2 * cf / sf / r + mu * u / (r * sf) ** 2
                acc = acc - 2 * om * cf * at(q.uc[2]) - mu / 3 * jump(q.div[0] + q.div[2]) / (r * h[1])
                acc = acc - mu * (2 / (r * r * h[1]) * jump(q.uc[0]) - 2 * cf / (r * sf) ** 2 * at(q.div[2] * r * s))
            else:
                m = 1 / (r * s * h[2])
                acc = acc + u * (at(q.uc[1]) * self.cc / s + at(q.uc[0])) / r + mu * u / (r * s) ** 2
                acc = acc + 2 * om * (self.cc * at(q.uc[1]) + s * at(q.uc[0])) - mu / 3 * m * jump(q.div[0] + q.div[1])
                acc = acc - mu * (2 * m / r * jump(q.uc[0]) + 2 * self.cc / (r * s) * m * jump(q.uc[1]))
            N.append(acc)
        N.append(out[1])
        R = []
        for f in range(5):
            c = f - 1 if 1 <= f <= 3 else None
            pick = (lambda v: self.inner(v, c)) if c is not None else (lambda v: v)
            R.append(-pick(D[f]) - self.p.dt * (N[f] - (0 if S is None else pick(S[f]))))
        return R

    def sweep(self, q, a, R):
        """(I + dt/2 D_a) x = R; velocities on their unknown faces"""
        hh, n, per = 0.5 * self.p.dt, self.n[a], self.per[a]
        full = lambda v, like: v.expand_as(like) if torch.is_tensor(v) else torch.full_like(like, v)   # noqa: E731
        z = torch.zeros_like(q.rho)
        A, B, C = ([[z] * 3 for _ in range(3)] for _ in range(3))
        for row, isT in ((0, False), (1, True)):
            adv, wT, al, gd, wv, _ = self.rows_c(q, a, isT)
            v0, v1 = al * gd[0] + wv[0], al * gd[1] + wv[1]
            A[row][1], B[row][1], C[row][1] = (full(w, z) for w in wT)
            if isT:
                A[1][1], C[1][1] = A[1][1] - adv, C[1][1] + adv
            else:
                A[0][0], C[0][0] = -adv, adv
            A[row][2], B[row][2] = v0, v1
        wp, wu, _ = self.rows_f(q, a)
        def cells(v):            # a value on face m + 1, in cell m's row (the last cell of a walled line has none)
            return torch.roll(v, -1, a) if per else torch.cat([v, torch.zeros_like(z.narrow(a, 0, 1))], a)
        wp, wu = cells(full(wp, self.sides(z, a)[0])), [cells(v) for v in wu]
        A[2][2], B[2][0], B[2][2], C[2][0], C[2][2] = wu[0], -wp, wu[1], wp, wu[2]
        stack = lambda M: torch.stack([torch.stack(r, -1) for r in M], -2).movedim(a, 0) * hh           # noqa: E731
        A, B, C = stack(A), stack(B), stack(C)
        B = B + torch.eye(3, dtype=F64, device=DEV)
        if not per:              # zero-gradient ghosts of p and T; no face beyond the walls
            keep2 = torch.tensor([1.0, 1.0, 0.0], dtype=F64, device=DEV)
            fold = torch.zeros((n, 1, 1, 1, 1), dtype=F64, device=DEV)
            first, last = fold.clone(), fold.clone()
            first[0], last[-1] = 1.0, 1.0
            pt = torch.outer(keep2, keep2)
            B = B + first * A * pt + last * C * pt
            no_u = torch.ones((3, 3), dtype=F64, device=DEV)
            no_u[:2, 2] = 0.0
            B = B * (1 - last) + last * B * no_u
            A, C = A * (1 - first), C * (1 - last)
        d = torch.stack([R[0], R[4], cells(R[1 + a])], -1).movedim(a, 0)
        lines = lambda M: M.reshape(n, -1, 3, 3)                                                        # noqa: E731
        x = (_cyclic if per else _thomas)(lines(A), lines(B), lines(C), d.reshape(n, -1, 3, 1))
        x = torch.stack(x).reshape(d.shape).movedim(0, a)
        out = [x[..., 0], None, None, None, x[..., 1]]
        u = x[..., 2]
        out[1 + a] = torch.roll(u, 1, a) if per else u.narrow(a, 0, n - 1)
        for c in range(3):
            if c == a:
                continue
            w = [(hh * v).movedim(a, 0) for v in self.rows_s(q, c, a)]
            shape = w[1].shape
            lo, di, up = w[0].reshape(n, -1), 1 + w[1].reshape(n, -1), w[2].reshape(n, -1)
            if not per:          # tangential no-slip ghosts: - interior
                di = torch.cat([di[:1] - lo[:1], di[1:-1], di[-1:] - up[-1:]])
                lo = torch.cat([torch.zeros_like(lo[:1]), lo[1:]])
                up = torch.cat([up[:-1], torch.zeros_like(up[:1])])
            one = lambda v: v.reshape(n, -1, 1, 1)                                                      # noqa: E731
            y = (_cyclic if per else _thomas)(one(lo), one(di), one(up), one(R[1 + c].movedim(a, 0).reshape(n, -1)))
            out[1 + c] = torch.stack(y).reshape(shape).movedim(0, a)
        return out

    def spread(self, x, c):
        """values on unknown faces, zero on the wall faces"""
        if self.per[c]:
            return x
        e = torch.zeros_like(x.narrow(c, 0, 1))
        return torch.cat([e, x, e], c)

    def step(self, Un):
        """(U^{n+1}, the RMS over unknowns of the last increment of each field)"""
        Uk = list(Un)
        if self.p.W:
            for c in range(3):
                ends = [self.p.W[1][(c, c, s)].unsqueeze(c) for s in range(2)]
                Uk[1 + c] = torch.cat([ends[0], self.inner(Uk[1 + c], c), ends[1]], c)
        for _ in range(K):
            q = self.freeze([0.5 * (a + b) for a, b in zip(Un, Uk)])
            x = self.rhs(q, [b - a for a, b in zip(Un, Uk)], self.p.S)
            for a in range(3):
                x = self.sweep(q, a, x)
            res = [torch.sqrt(torch.mean(v.detach() ** 2)).item() for v in x]
            Uk = [u + (self.spread(v, f - 1) if 1 <= f <= 3 else v) for f, (u, v) in enumerate(zip(Uk, x))]
        return Uk, np.array(res)
