"""The stand-alone block-tridiagonal solve on systems of very large and very small
numbers: scaling the blocks and the right-hand side by powers of two scales the
solution exactly as long as the blocks' inverses and the solution are in FP64's
range, in both of its forms."""
import numpy as np
import pytest

import paper_2004_13887_gb300 as sph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nl", [5, 7144, 7145, 20001])   # 16 lanes a line, one thread a line (from 7145 on 152 SMs)
@pytest.mark.parametrize("blocks,sol", [(330, 100), (-330, -100), (330, -300), (-330, 300), (0, 600), (0, -600)])
def test_power_of_two_scales(nl, blocks, sol):
    import torch
    n = 6
    rng = np.random.default_rng(nl)
    A, B, C = (0.2 * rng.standard_normal((nl, n, 3, 3)) for _ in range(3))
    B += 2.0 * np.eye(3)
    d = rng.standard_normal((nl, n, 3))
    dev = lambda *a: [torch.from_numpy(v).cuda() for v in a]
    ref = sph.block_thomas_noalloc(*dev(A, B, C, d)).cpu().numpy()
    x = sph.block_thomas_noalloc(*dev(*[np.ldexp(v, blocks) for v in (A, B, C)], np.ldexp(d, blocks + sol))).cpu().numpy()
    assert np.array_equal(x, np.ldexp(ref, sol))
