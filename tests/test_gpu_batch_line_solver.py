"""Batched launches below the line count from which r and theta lines share the
many-lines kernels: every context keeps the partitioned layout it was set to, in
launches of its own along all three directions, and steps like on its own; above that
count a context's choice is left for its phi lines."""
import numpy as np
import pytest

import paper_2004_13887_gb300 as sph
from inputs import cases
from tests.gpu_helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


def _solver(c, which):
    import torch
    s = sph.Solver(c.grid, c.par, precision=sph.SPH_PREC_MIXED, stream=torch.cuda.Stream())
    s.set_background(*c.bg)
    s.set_state(to_dev(c.init))
    s.set_line_solver(which)
    return s


def _replay(cs, which):
    """launches of one replay of two steps of one iteration, and the states after it"""
    import torch
    solvers = [_solver(c, w) for c, w in zip(cs, which)]
    torch.cuda.synchronize()
    b = sph.Batch(solvers)
    b.capture(1.0, 1, 2, fused=True)
    n0 = solvers[0].launches
    b.launch(1)
    b.status()
    n = solvers[0].launches - n0
    out = [to_host(s.get_state()) for s in solvers]
    b.close()
    for s in solvers:
        s.close()
    return n, out


ALL = [sph.SPH_LINES_PARTITIONED, sph.SPH_LINES_PARTITIONED_WARP, sph.SPH_LINES_PARTITIONED_NARROW]
STAGES = 4   # averages, coefficients, right-hand side, the residual's sums


@pytest.mark.parametrize("which", [ALL[:1] * 2, ALL[:2], ALL[1:], [ALL[2], ALL[0]]])
def test_few_lines_keep_their_layouts(which):
    cs = [cases.bubble((64, 64, 64), seed=s, dt=1.0) for s in (1, 2)]   # 8192 lines a direction
    n, out = _replay(cs, which)
    # two steps; block and scalar lines of every layout in three directions
    assert n == 2 * (STAGES + 3 * 2 * len(set(which)))
    for c, w, got in zip(cs, which, out):
        s = _solver(c, w)
        for _ in range(2):
            s.step(1.0, 1)
        for f, (a, b) in enumerate(zip(got, to_host(s.get_state()))):
            scale = float(np.max(np.abs(b - c.init[f]))) or 1.0
            assert float(np.max(np.abs(a - b))) <= 1e-5 * scale, (w, f)
        s.close()


@pytest.mark.parametrize("which", [ALL[:1] * 2, ALL[1:]])
def test_many_lines_share_r_and_theta(which):
    cs = [cases.bubble(n, seed=1, dt=1.0) for n in ((64, 64, 192), (64, 64, 64))]   # 16384 lines along r and theta
    n, _ = _replay(cs, which)
    # one pair of launches along r and one along theta; phi lines of two lengths
    assert n == 2 * (STAGES + 2 * 2 + 2 * 2)
