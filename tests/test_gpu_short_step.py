"""FP64 steps of any positive length: below the smallest change FP64 holds, a step, a
sweep and the adjoint leave what they are given (D is finite, so I + h D is I to
the last bit), whatever the line solver."""
import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import cases
from tests.gpu_helpers import perturbed, solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [sph.SPH_LINES_PARTITIONED, sph.SPH_LINES_THOMAS])
@pytest.mark.parametrize("dt", [1e-50, 1e-70, 1e-110, 1e-200])
def test_tiny_step(dt, which):
    c = cases.sector_mms((6, 7, 8))
    s = solver_for(c.grid, c.par, c.bg, c.init)
    s.set_line_solver(which)
    s.step(dt, 2)
    for q, f in enumerate(to_host(s.get_state())):
        assert np.max(np.abs(f - c.init[q])) <= 1e-15 * np.max(np.abs(c.init[q])), q
    rhs = perturbed(c.grid.zeros(), [1.0] * 5, 3, c.grid)
    for d in range(3):
        for a, b in zip(to_host(s.sweep(d, dt, to_dev(rhs))), rhs):
            assert np.max(np.abs(a - b)) <= 1e-14, d
    for a, b in zip(to_host(s.step_adjoint(dt, 2, to_dev(rhs))), rhs):
        assert np.max(np.abs(a - b)) <= 1e-14
    s.close()
