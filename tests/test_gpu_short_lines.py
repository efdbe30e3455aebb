"""The mixed mode's many-lines sweeps where they are taken for lengths the
partitioned solver does not have (from 1024 lines of 4 cells): phi lines of 4 to 9
cells, whose two sides meet within one group of 4 cells or next to one, and lengths
around later groups, walled and cyclic; the shortest r and theta lines.  Every case
has at least 1024 lines in the direction it is meant for and the sweep's launches are
counted, so that a case that another solver took fails -- or, with lines of 2 and 3
cells, one that the one-thread-per-line solver did not.

Bounds: 1e-5 of each field's largest value against the oracle for a sweep, as for
every FP32 line solve, and for a step 1e-4 of the change."""
import math

import numpy as np
import pytest

import oracle
import paper_2004_13887_gb300 as sph
from inputs import Grid, Params
from tests.gpu_helpers import perturbed, rel_err, solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu

PAR = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)


def _case(n, periodic):
    g = Grid(*n, 1.0, 1.3, 0.4, 2.7, 0.0, 2 * math.pi if periodic else 1.5, periodic=periodic)
    U = perturbed(g.zeros(), [0.1, 0.05, 0.05, 0.05, 0.1], 5, g)
    bg = (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0))
    return g, bg, U, perturbed(U, [1e-2] * 5, 6, g)


def _launches(s, d, dt, rhs):
    n0 = s.launches
    x = to_host(s.sweep(d, dt, to_dev(rhs)))
    return x, s.launches - n0


GRIDS = [((33, 35, n), p, 2) for n in (3, 4, 5, 6, 7, 8, 9, 36, 37) for p in (False, True)]
GRIDS += [((33, 35, 2), False, 2)]
GRIDS += [((n, 33, 35), p, 0) for n, p in ((2, False), (3, True), (4, False), (5, False), (18, True))]
GRIDS += [((33, n, 35), p, 1) for n, p in ((2, False), (3, True), (4, False), (5, False), (18, True))]


@pytest.mark.parametrize("n,periodic,d", GRIDS)
def test_sweep_and_step(n, periodic, d):
    g, bg, U, it = _case(n, periodic)
    dt = 0.01
    s = solver_for(g, PAR, bg, U, precision=sph.SPH_PREC_MIXED)
    s.set_iterate(it)
    rhs = perturbed(g.zeros(), [1.0] * 5, 7 + d, g)
    x, taken = _launches(s, d, dt, rhs)
    s.set_line_solver(sph.SPH_LINES_THOMAS)
    many = n[d] >= 4   # (two launches)
    assert taken == _launches(s, d, dt, rhs)[1] + many, "another solver was taken"
    s.set_line_solver(sph.SPH_LINES_PARTITIONED)
    ref = oracle.sweep(g, PAR, U, it, dt, d, rhs, bg=bg)
    for q in range(5):
        assert rel_err(x[q], ref[q]) <= 1e-5, (n, d, q, rel_err(x[q], ref[q]))
    s.set_state(U)
    s.step(dt, 2)
    V = to_host(s.get_state())
    ref, _ = oracle.step(g, PAR, U, dt, 2, bg=bg)
    for q in range(5):
        change = np.max(np.abs(ref[q] - U[q]))
        assert np.max(np.abs(V[q] - ref[q])) <= 1e-4 * change, (n, q)
    s.close()
