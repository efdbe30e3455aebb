"""Cyclic phi lines of the mixed mode close their ring in FP64: the last unknown's
3x3 (scalar) system and every increment y - Z X are FP64, and the increment reaches
the FP64 state without a rounding to FP32 -- for the one-thread-per-line solver and
the many-lines one alike."""
import math

import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import Grid, Params
from tests.gpu_helpers import perturbed, solver_for, to_host

pytestmark = pytest.mark.gpu

PAR = Params(gamma=1.4, cv=2.5, Pr=0.7, mu=0.05, pinf=2.0, g=0.3, omega=0.4)


@pytest.mark.parametrize("np_", [5, 36, 37])
@pytest.mark.parametrize("which", [sph.SPH_LINES_PARTITIONED, sph.SPH_LINES_THOMAS])
def test_increment_is_not_rounded(np_, which):
    g = Grid(33, 35, np_, 1.0, 1.3, 0.4, 2.7, 0.0, 2 * math.pi, periodic=True)
    bg = (np.full(g.nr + 2, 20.0), np.full(g.nr + 2, 30.0))
    # from the rest state one iteration's result is the phi sweep's increment itself
    s = solver_for(g, PAR, bg, g.zeros(), precision=sph.SPH_PREC_MIXED)
    s.set_line_solver(which)
    s.step(0.01, 1, perturbed(g.zeros(), [1.0] * 5, 3, g))
    for q, f in enumerate(to_host(s.get_state())):
        if q in (1, 2):   # (walls at rest)
            f = f[1:-1] if q == 1 else f[:, 1:-1]
        # the cells beside the ring's seam (Z X fades along the line, below FP64's
        # last bit of y in the end): a value of 40 or more bits falls on one of
        # FP32's 24 by chance about once in 2^16
        f = f[:, :, [0, -1]]
        rounded = float(np.mean(f.astype(np.float32).astype(np.float64) == f))
        assert rounded <= 1e-2, (q, rounded)
    s.close()
