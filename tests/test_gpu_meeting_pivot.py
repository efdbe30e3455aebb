"""A zero pivot where the two sides of a transverse scalar line meet is reported like
any other.  Walled phi lines of two cells, fluid at rest, negative density: the line's
matrix is [[1 - 3k, k], [k, 1 - 3k]], k = h 2 mu / (2 |rho| (r sin dphi)^2), singular at k
= 1/4, which no side's own pivot (1 - 3k) shows.  dt is stepped in its last bits around
that value on several lines; a solve that gives a value that is not finite must
have raised SPH_ERR_SINGULAR, and some step has to hit it."""
import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import Grid, Params
from tests.gpu_helpers import solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu

SINGULAR = -4   # SPH_ERR_SINGULAR
PAR = Params(gamma=1.4, cv=2.5, Pr=1.3, mu=0.05, pinf=0.0, g=0.0, omega=0.0)


@pytest.mark.parametrize("prec", [sph.SPH_PREC_FP64, sph.SPH_PREC_MIXED])
def test_zero_pivot_between_the_sides(prec):
    g = Grid(33, 35, 2, 1.0, 1.3, 0.4, 2.7, 0.0, 1.5, periodic=False)
    rho = 20.0 / (PAR.cv * (PAR.gamma - 1.0) * -30.0)
    s = solver_for(g, PAR, (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, -30.0)), g.zeros(), precision=prec)
    rhs = g.zeros()
    rhs[1][1:-1, :, 0] = 1.0   # excites the vanishing eigenvalue's vector (1, 1)
    rhs = to_dev(rhs)
    ulp = 2.0 ** -24 if prec == sph.SPH_PREC_MIXED else 2.0 ** -53
    hits = 0
    for i, j in ((3, 4), (8, 11), (15, 17), (21, 6), (27, 30), (31, 22)):
        r, th = g.r1 + i * g.dr, g.t1 + (j + 0.5) * (g.t2 - g.t1) / g.nt
        m = g.np / ((g.p2 - g.p1) * r * np.sin(th))
        dt0 = 2.0 * 0.25 * -rho / (PAR.mu * m * m)
        for k in range(-12, 13):
            try:
                x = to_host(s.sweep(2, dt0 * (1.0 + k * ulp), rhs))
            except sph.SphError as e:
                assert e.code == SINGULAR, (e.code, i, j, k)
                hits += 1
                continue
            assert all(np.isfinite(f).all() for f in x), (i, j, k)
    assert hits > 0
    s.close()
