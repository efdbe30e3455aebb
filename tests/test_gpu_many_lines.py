"""The mixed mode's many-lines sweeps (one lane per line and side) at the edges of
their layouts: the shortest lines, lengths whose halves differ, phi lengths around
the groups of 4 cells (aligned and not), a split that leaves one side empty, line
counts that leave a warp partly filled, walled and cyclic; and lengths that the
partitioned solver also takes, with line counts on both sides of the switch
(10240).  Bounds as for every FP32 line solve: 1e-5 of each field's largest value
against the oracle; the step's residual (sums of squares of the last increments)
1e-3 relative."""
import math

import numpy as np
import pytest

import oracle
import paper_2004_13887_gb300 as sph
from inputs import Grid, Params
from tests.gpu_helpers import perturbed, rel_err, solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu

PAR = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)
GRIDS = [((2, 2, 2), False), ((3, 5, 7), False), ((5, 2, 8), False), ((4, 3, 9), False), ((7, 9, 37), False),
         ((6, 11, 40), False), ((33, 35, 5), False), ((2, 3, 3), True), ((5, 7, 4), True), ((3, 9, 5), True),
         ((4, 34, 36), True), ((9, 10, 50), True),
         ((16, 32, 320), False), ((16, 32, 319), False), ((32, 320, 32), False), ((32, 319, 32), True)]


@pytest.mark.parametrize("n,periodic", GRIDS)
def test_sweeps_and_step(n, periodic):
    g = Grid(*n, 1.0, 1.3, 0.4, 2.7, 0.0, 2 * math.pi if periodic else 1.5, periodic=periodic)
    U = perturbed(g.zeros(), [0.1, 0.05, 0.05, 0.05, 0.1], 5, g)
    bg = (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0))
    it = perturbed(U, [1e-2] * 5, 6, g)
    dt = 0.01
    s = solver_for(g, PAR, bg, U, precision=sph.SPH_PREC_MIXED)
    s.set_iterate(it)
    for d in range(3):
        rhs = perturbed(g.zeros(), [1.0] * 5, 7 + d, g)
        x = to_host(s.sweep(d, dt, to_dev(rhs)))
        ref = oracle.sweep(g, PAR, U, it, dt, d, rhs, bg=bg)
        for q in range(5):
            assert rel_err(x[q], ref[q]) <= 1e-5, (n, d, q, rel_err(x[q], ref[q]))
    s.set_state(U)
    res = s.step(dt, 2, residual=True)
    V = to_host(s.get_state())
    ref, rres = oracle.step(g, PAR, U, dt, 2, bg=bg)
    for q in range(5):
        assert abs(res[q] - rres[q]) <= 1e-3 * rres[q], (n, q, res[q], rres[q])
        change = np.max(np.abs(ref[q] - U[q]))
        assert np.max(np.abs(V[q] - ref[q])) <= 1e-4 * change, (n, q)
