"""The tables a context derives from its grid and background are complete when the
call that makes them returns: work on any other stream (a batch replayed on its
own) may read them at once, so nothing may still be queued on the context's
stream then."""
import pytest

import paper_2004_13887_gb300 as sph
from inputs import cases
from tests.gpu_helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [sph.SPH_PREC_FP64, sph.SPH_PREC_MIXED])
def test_tables_are_done_on_return(prec):
    import torch
    c = cases.bubble((64, 128, 16), seed=1, dt=1.0)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        s = sph.Solver(c.grid, c.par, precision=prec, stream=st)
        assert st.query(), "create left work queued"
        for _ in range(3):
            s.set_background(*c.bg)
            assert st.query(), "set_background left work queued"
        s.close()


def test_batch_after_a_new_background():
    """A replay right after a change of background steps with the new one."""
    import torch
    c = cases.bubble((16, 64, 64), seed=1, dt=1.0)
    other = (c.bg[0] * 1.01, c.bg[1] * 1.02)
    out = []
    for late in (False, True):
        s = sph.Solver(c.grid, c.par, precision=sph.SPH_PREC_MIXED, stream=torch.cuda.Stream())
        s.set_background(*(c.bg if late else other))
        s.set_state(to_dev(c.init))
        torch.cuda.synchronize()
        b = sph.Batch([s])
        b.capture(c.dt, 2, 2, fused=True)
        if late:
            s.set_background(*other)
        b.launch(1)
        b.status()
        out.append([f.clone() for f in s.get_state()])
        b.close()
        s.close()
    for q in range(5):
        assert torch.equal(out[0][q], out[1][q]), q
