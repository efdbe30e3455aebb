"""The wall faces of u_phi at the high end of walled phi lines in the mixed mode:
a step keeps whatever normal velocity the state holds there, and a sweep's
increment is zero there whatever its output buffer held before -- for every
line solver and for lengths the partitioned solver takes and does not."""
import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import cases
from tests.gpu_helpers import perturbed, solver_for, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_", [16, 18, 64])
@pytest.mark.parametrize("which", [sph.SPH_LINES_PARTITIONED, sph.SPH_LINES_PARTITIONED_NARROW, sph.SPH_LINES_THOMAS])
def test_high_phi_wall_face(np_, which):
    c = cases.bubble((6, 8, np_), seed=3, dt=0.1)
    U = [f.copy() for f in c.init]
    U[3][:, :, 0], U[3][:, :, -1] = 0.01, 0.02
    s = solver_for(c.grid, c.par, c.bg, U, precision=sph.SPH_PREC_MIXED)
    s.set_line_solver(which)
    rhs = to_dev(perturbed(c.grid.zeros(), [1.0] * 5, 4, c.grid))
    for d in (0, 1, 2):   # r and theta sweeps leave other values in the shared work buffers
        x = to_host(s.sweep(d, c.dt, rhs))
        assert np.all(x[3][:, :, 0] == 0.0) and np.all(x[3][:, :, -1] == 0.0), (np_, d)
    s.step(c.dt, 2)
    V = to_host(s.get_state())
    assert np.all(V[3][:, :, 0] == 0.01) and np.all(V[3][:, :, -1] == 0.02), np_
