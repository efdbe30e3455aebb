"""The mixed mode's right-hand side, one thread a cell with its lower faces: rows
whose last tile is partly empty, tiles that touch the walls and inner ones, walled
and periodic phi, both below and above a tile's width, against the oracle.

Bound: as for any right-hand side of the mixed mode, 1e-5 of the field's maximum
(about 60 FP32 terms a row, each rounded to 2^-24 of values up to a few times the
row's) plus twice the oracle's own evaluation-order noise.
"""
import math

import numpy as np
import pytest

import oracle
import paper_2004_13887_gb300 as sph
from oracle import Grid, Params
from tests.gpu_helpers import perturbed, solver_for, to_host
from tests.test_gpu_parity import rhs_midpoint

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,periodic,tile", [
    ((2, 2, 2), False, None), ((6, 7, 31), False, None), ((7, 6, 33), False, (1, 1)), ((6, 9, 130), False, None),
    ((6, 8, 129), True, None), ((7, 9, 96), True, (2, 2)), ((8, 11, 17), False, (4, 2)), ((6, 6, 4), True, (1, 1))])
def test_rhs_of_cells(n, periodic, tile):
    sph.build()
    oracle.build()
    par = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)
    g = Grid(*n, 1.0, 1.3, 0.9, 2.1, 0.0, 2 * math.pi if periodic else 1.2, periodic=periodic)
    Un = perturbed(g.zeros(), [0.1, 0.05, 0.05, 0.05, 0.1], 5, g)
    Uk = perturbed(Un, [1e-2] * 5, 6, g)
    bg = (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0))
    s = solver_for(g, par, bg, Un, precision=sph.SPH_PREC_MIXED)
    if tile:
        s.set_tile(*tile)
    s.set_iterate(Uk)
    R = to_host(s.rhs(0.01))
    ref = oracle.rhs(g, par, Un, Uk, 0.01, bg=bg)
    mid = rhs_midpoint(g, par, bg, Un, Uk, 0.01, None)
    for q in range(5):
        noise = float(np.max(np.abs(mid[q] - ref[q])))
        err = float(np.max(np.abs(R[q] - ref[q])))
        assert err <= 1e-5 * float(np.max(np.abs(ref[q]))) + 2 * noise, (q, err)
    s.close()
