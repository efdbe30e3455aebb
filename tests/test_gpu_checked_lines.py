"""The bounds-checked build over the line solvers that need many lines: the mixed
mode's many-lines kernels (r, theta and phi lines, walled and cyclic, rows that are
multiples of 4 cells and not, with a last warp partly filled), alone and batched, and
the FP64 sweeps and their transposes with a lane per line and side (more than 4864
lines).  The violation count must stay zero."""
import math

import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import Grid, Params, cases
from paper_2004_13887_gb300 import _build
from tests.gpu_helpers import perturbed, solver_for, to_dev

pytestmark = pytest.mark.gpu

PAR = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)


@pytest.fixture(scope="module")
def checked():
    path = _build.build(checked=True)
    prev = sph.use_library(path)
    assert sph.bounds_report()[0] == 0
    yield
    sph.restore_library(prev)


def _solver(n, periodic, prec):
    g = Grid(*n, 1.0, 1.3, 0.4, 2.7, 0.0, 2 * math.pi if periodic else 1.5, periodic=periodic)
    U = perturbed(g.zeros(), [0.1, 0.05, 0.05, 0.05, 0.1], 5, g)
    s = solver_for(g, PAR, (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0)), U, precision=prec)
    return g, U, s


@pytest.mark.parametrize("n,periodic", [((33, 35, 4), False), ((33, 35, 5), True), ((33, 35, 37), False),
                                        ((33, 35, 36), True), ((4, 33, 35), True), ((33, 5, 35), False)])
def test_many_lines(checked, n, periodic):
    g, U, s = _solver(n, periodic, sph.SPH_PREC_MIXED)
    n0 = s.launches
    s.step(0.01, 1)
    assert s.launches - n0 > 6   # a sweep of two launches among the step's stages
    for d in range(3):
        s.sweep(d, 0.01, to_dev(perturbed(g.zeros(), [1.0] * 5, 7 + d, g)))
    s.close()
    count, first = sph.bounds_report()
    assert count == 0, (n, count, first)


def test_batched_many_lines(checked):
    import torch
    solvers = []
    for n, seed in (((16, 64, 128), 1), ((32, 48, 64), 2)):   # 11264 r lines, 4096 theta lines
        c = cases.bubble(n, seed=seed, dt=1.0)
        s = sph.Solver(c.grid, c.par, precision=sph.SPH_PREC_MIXED, stream=torch.cuda.Stream())
        s.set_background(*c.bg)
        s.set_state(to_dev(c.init))
        solvers.append(s)
    torch.cuda.synchronize()
    b = sph.Batch(solvers)
    b.capture(1.0, 1, 2, fused=True)
    b.launch(1)
    b.status()
    b.close()
    for s in solvers:
        s.close()
    count, first = sph.bounds_report()
    assert count == 0, (count, first)


@pytest.mark.parametrize("n,periodic", [((3, 70, 72), False), ((70, 3, 72), False), ((70, 72, 3), False), ((70, 72, 4), True)])
def test_fp64_lane_per_line(checked, n, periodic):
    g, U, s = _solver(n, periodic, sph.SPH_PREC_FP64)
    s.step(0.01, 1)
    for d in range(3):
        s.sweep(d, 0.01, to_dev(perturbed(g.zeros(), [1.0] * 5, 7 + d, g)))
    s.set_state(U)
    s.step_adjoint(0.01, 1, to_dev(perturbed(g.zeros(), [1.0] * 5, 9, g)))
    s.close()
    count, first = sph.bounds_report()
    assert count == 0, (n, count, first)
