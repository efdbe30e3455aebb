"""Wall data handed over as device arrays (one kernel) give the step that host
arrays give, bit for bit: all walls, some of them, one time level only, strided
tensors, tensors written on a side stream, and sets that grow and shrink between
calls; then none."""
import numpy as np
import pytest
import torch

import paper_2004_13887_gb300 as sph
from inputs import cases
from tests.gpu_helpers import solver_for

pytestmark = pytest.mark.gpu


def _dev(walls, stream=None):
    if walls is None:
        return None
    with torch.cuda.stream(stream or torch.cuda.current_stream()):
        out = {}
        for n, (key, a) in enumerate(walls.items()):
            t = torch.from_numpy(np.ascontiguousarray(a)).cuda()
            if n % 2 and t.dim() == 2:                      # the same values, strided
                t = torch.stack([t, t + 1.0], dim=-1)[..., 0]
            out[key] = t
        return out


@pytest.mark.parametrize("precision", [sph.SPH_PREC_FP64, sph.SPH_PREC_MIXED])
def test_device_walls_equal_host_walls(precision):
    sph.build()
    w = cases.paper_mms(1e-2, n=(4, 5, 7))
    a, b = (solver_for(w.grid, w.par, w.bg, w.init, precision=precision) for _ in range(2))
    w0, w1 = w.walls(0.0), w.walls(w.dt)
    keys = list(w1)
    few = {k: w1[k] for k in keys[1::3]}
    other = {k: w0[k] for k in keys[::4]}
    for n, (x, y) in enumerate([(few, None), (w0, w1), (None, few), (other, few), (w1, w0), ({}, {}), (None, None)]):
        a.set_bc(x, y)
        stream = torch.cuda.Stream() if n % 2 else None
        with torch.cuda.stream(stream or torch.cuda.current_stream()):
            b.set_bc(_dev(x), _dev(y))
        a.step(w.dt, 2, w.source(0.5 * w.dt))
        b.step(w.dt, 2, w.source(0.5 * w.dt))
        for q, (u, v) in enumerate(zip(a.get_state(device=False), b.get_state(device=False))):
            assert np.array_equal(u, v), (n, q)
