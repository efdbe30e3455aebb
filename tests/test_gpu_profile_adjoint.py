"""Stage timing with an adjoint in the timed span: the record reads back as finite,
non-negative times, for both FP64 line solvers, and the context goes on working."""
import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import cases
from tests.gpu_helpers import perturbed, solver_for, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [sph.SPH_LINES_PARTITIONED, sph.SPH_LINES_THOMAS])
def test_profile_over_an_adjoint(which):
    c = cases.sector_mms((6, 7, 8))
    s = solver_for(c.grid, c.par, c.bg, c.init)
    s.set_line_solver(which)
    lam = to_dev(perturbed(c.grid.zeros(), [1.0] * 5, 9, c.grid))
    s.profile(True)
    s.step_adjoint(c.dt, 2, lam)
    rec = s.profile_read()
    # two iterations forward less the last, two again in reverse: 3 of every stage
    for k in ("coef", "rhs", "sweep_r", "sweep_theta", "sweep_phi"):
        ms, n = rec[k]
        assert np.isfinite(ms) and 0.0 < ms < 1e3 and n == 3, (k, ms, n)
    s.profile(False)
    s.step(c.dt, 2)
    s.close()
