"""The stand-alone block-tridiagonal solve around the edges of its two forms (16
lanes a line up to 8192 lines, one thread a line above): one line, odd line
counts, one- and two-block lines, both sides of the switch, and a zero pivot that
must fill its own line with NaN and leave the line sharing its warp alone.  Bound:
1e-12 of the largest value against dense LU (the systems are diagonally dominant)."""
import numpy as np
import pytest

import paper_2004_13887_gb300 as sph

pytestmark = pytest.mark.gpu


def _system(nl, n, seed):
    rng = np.random.default_rng(seed)
    A, B, C = (0.2 * rng.standard_normal((nl, n, 3, 3)) for _ in range(3))
    B += 2.0 * np.eye(3)
    return A, B, C, rng.standard_normal((nl, n, 3))


def _dense(A, B, C, d):
    n = B.shape[0]
    M = np.zeros((3 * n, 3 * n))
    for m in range(n):
        M[3 * m:3 * m + 3, 3 * m:3 * m + 3] = B[m]
        if m:
            M[3 * m:3 * m + 3, 3 * m - 3:3 * m] = A[m]
        if m + 1 < n:
            M[3 * m:3 * m + 3, 3 * m + 3:3 * m + 6] = C[m]
    return np.linalg.solve(M, d.reshape(-1)).reshape(n, 3)


def _solve(*a):
    import torch
    return sph.block_thomas_noalloc(*[torch.from_numpy(v).cuda() for v in a]).cpu().numpy()


@pytest.mark.parametrize("nl,n", [(1, 1), (1, 2), (2, 5), (3, 1), (7, 33), (1025, 4), (8191, 2), (8192, 3), (8193, 3)])
def test_against_dense_lu(nl, n):
    s = _system(nl, n, nl + n)
    x = _solve(*s)
    for l in sorted({0, 1, nl // 2, nl - 2, nl - 1} & set(range(nl))):
        ref = _dense(*[v[l] for v in s])
        assert np.max(np.abs(x[l] - ref)) <= 1e-12 * np.max(np.abs(ref)), (nl, n, l)


@pytest.mark.parametrize("nl", [6, 8200])
def test_zero_pivot_stays_in_its_line(nl):
    n = 4
    A, B, C, d = _system(nl, n, 3)
    B[2, 0] = 0.0
    x = _solve(A, B, C, d)
    assert np.isnan(x[2]).all()
    for l in (0, 1, 3, nl - 1):
        ref = _dense(A[l], B[l], C[l], d[l])
        assert np.max(np.abs(x[l] - ref)) <= 1e-12 * np.max(np.abs(ref)), l
