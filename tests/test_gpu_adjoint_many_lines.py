"""The step adjoint with more lines than the FP64 sweeps split over lanes (4864 on 152
SMs), along each direction and on a ring: the transposed solves with a lane per line
and side against the one-thread-per-line ones.  Bound: 1e-11 of each field's largest
value (two transposed solves a direction, 1e-12 each as for the sweeps' parity, through
two iterations)."""
import math

import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import Grid, Params
from tests.gpu_helpers import perturbed, rel_err, solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu

PAR = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)


@pytest.mark.parametrize("n,periodic", [((3, 70, 72), False), ((8, 70, 72), True), ((70, 5, 72), False), ((70, 72, 4), False),
                                        ((70, 72, 3), True), ((70, 72, 6), True)])
def test_transposed_solves(n, periodic):
    g = Grid(*n, 1.0, 1.3, 0.4, 2.7, 0.0, 2 * math.pi if periodic else 1.5, periodic=periodic)
    U = perturbed(g.zeros(), [0.1, 0.05, 0.05, 0.05, 0.1], 5, g)
    bg = (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0))
    lam = perturbed(g.zeros(), [1.0] * 5, 9, g)
    out = []
    for which in (sph.SPH_LINES_PARTITIONED, sph.SPH_LINES_THOMAS):
        s = solver_for(g, PAR, bg, U)
        s.set_line_solver(which)
        out.append(to_host(s.step_adjoint(0.01, 2, to_dev(lam))))
        s.close()
    for q in range(5):
        assert rel_err(out[0][q], out[1][q]) <= 1e-11, (n, q, rel_err(out[0][q], out[1][q]))
