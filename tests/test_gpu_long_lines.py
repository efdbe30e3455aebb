"""The many-lines solver of the mixed mode on long stiff lines: smooth and noisy
right-hand sides, strong conduction and sound speed along the line, lengths the
partitioned solver does not take.  Its rows and its two-sided elimination may not be
less accurate than the one-sided solver with a thread per line.

Bound: 1.5 times that solver's error against the FP64 mode over the same lines, the
largest and the relative L2 norm of each field's (both make the same number of
roundings of values of the same size, in another order; the errors over 1155 lines
vary by less)."""
import math

import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import Grid, Params, cases
from tests.gpu_helpers import perturbed, rel_err, solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu

PAR = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)


def _shell(n):
    g = Grid(*n, 1.0, 1.3, 0.4, 2.7, 0.0, 1.5, periodic=False)
    U = perturbed(g.zeros(), [0.1, 0.05, 0.05, 0.05, 0.1], 5, g)
    return g, PAR, (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0)), U, 0.01


def _sector(n):
    c = cases.sector_mms(n, with_source=False)
    return c.grid, c.par, c.bg, c.init, c.dt


def _errors(x, ref):
    return [max(rel_err(a, b) for a, b in zip(x, ref)),
            max(float(np.linalg.norm(a - b) / np.linalg.norm(b)) for a, b in zip(x, ref))]


@pytest.mark.parametrize("smooth", [True, False])
@pytest.mark.parametrize("make,n,d", [(_shell, (200, 33, 35), 0), (_shell, (512, 33, 35), 0), (_sector, (512, 33, 35), 0),
                                      (_shell, (33, 301, 35), 1), (_shell, (33, 35, 300), 2), (_shell, (33, 35, 701), 2)])
def test_no_less_accurate_than_one_sided(make, n, d, smooth):
    g, par, bg, U, dt = make(n)
    it = perturbed(U, [1e-2] * 5, 6, g)
    rhs = perturbed(g.zeros(), [1e-2] * 5, 11, g)
    for q in (0, 4) if smooth else ():
        m = np.cos(math.pi * np.arange(n[d]) / n[d])
        rhs[q] += 1.0 + m.reshape([-1 if a == d else 1 for a in range(3)])
    xs, launches = [], []
    for prec, which in ((sph.SPH_PREC_FP64, None), (sph.SPH_PREC_MIXED, sph.SPH_LINES_THOMAS),
                        (sph.SPH_PREC_MIXED, sph.SPH_LINES_PARTITIONED)):
        s = solver_for(g, par, bg, U, precision=prec)
        if which is not None:
            s.set_line_solver(which)
        s.set_iterate(it)
        n0 = s.launches
        xs.append(to_host(s.sweep(d, dt, to_dev(rhs))))
        launches.append(s.launches - n0)
        s.close()
    assert launches[2] == launches[1] + 1, "the many-lines kernels (two launches) were not taken"
    for one, two in zip(_errors(xs[1], xs[0]), _errors(xs[2], xs[0])):
        assert two <= 1.5 * one, (one, two)
