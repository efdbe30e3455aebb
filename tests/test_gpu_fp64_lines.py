"""The FP64 line solves around the edges of their two layouts (one lane per line
and side for many lines, a 3x3 column per lane for few): the shortest lines, odd
lengths whose two sides differ by a cell, line counts that leave a warp partly
filled, and line counts on both sides of the switch, walled and cyclic.  Bound:
the parity tests' 1e-12 of each field's largest value against the oracle."""
import math

import numpy as np
import pytest

import oracle
from inputs import Grid, Params
from tests.gpu_helpers import perturbed, rel_err, solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu

PAR = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)
# (nr, nt, np), periodic: 5040 lines of the long pairs lie above the switch (4864 on 152 SMs)
GRIDS = [((2, 2, 2), False), ((2, 3, 33), False), ((3, 70, 72), False), ((70, 5, 72), False), ((70, 72, 4), False),
         ((5, 3, 3), True), ((3, 11, 4), True), ((70, 72, 3), True), ((70, 72, 6), True), ((9, 17, 31), True)]


@pytest.mark.parametrize("n,periodic", GRIDS)
def test_fp64_sweeps_at_layout_edges(n, periodic):
    g = Grid(*n, 1.0, 1.3, 0.4, 2.7, 0.0, 2 * math.pi if periodic else 1.5, periodic=periodic)
    U = perturbed(g.zeros(), [0.1, 0.05, 0.05, 0.05, 0.1], 5, g)
    bg = (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0))
    it = perturbed(U, [1e-2] * 5, 6, g)
    dt = 0.01
    s = solver_for(g, PAR, bg, U)
    s.set_iterate(it)
    for d in range(3):
        rhs = perturbed(g.zeros(), [1.0] * 5, 7 + d, g)
        x = to_host(s.sweep(d, dt, to_dev(rhs)))
        ref = oracle.sweep(g, PAR, U, it, dt, d, rhs, bg=bg)
        for q in range(5):
            assert rel_err(x[q], ref[q]) <= 1e-12, (n, d, q, rel_err(x[q], ref[q]))
