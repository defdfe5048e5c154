"""FP32 ELL product, block-Jacobi update and direction step of the refinement
solver at the edges of their batches: one to 33 slots per row around the
batch of eight, row counts around the four rows of a direction step, and
block sizes with a register budget of their own.  The solution is checked by
its true residual in FP64: after stopping at ||r|| <= tol ||b|| the residual
recomputed on the host differs by the rounding of one product only, at most
(K + 2) eps ||A||_inf ||x||_inf sqrt(n)."""
import numpy as np
import pytest

from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


def _banded(n, half, seed):
    """Symmetric, strictly diagonally dominant, 2*half+1 diagonals."""
    g = np.random.default_rng(seed)
    a = np.zeros((n, n))
    for k in range(1, min(half, n - 1) + 1):
        a[np.arange(n - k), np.arange(k, n)] = -g.uniform(0.1, 1.0, n - k)
    a += a.T
    a[np.arange(n), np.arange(n)] = 1.0 - a.sum(axis=1)
    rows, cols = np.nonzero(a)
    ptr = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(rows, minlength=n), out=ptr[1:])
    return (ptr, cols.astype(np.int32), a[rows, cols]), a


@pytest.mark.parametrize("prec", [0, 1, 4, 5, 8, 16, 32])
@pytest.mark.parametrize("n,half", [(1, 0), (2, 1), (7, 3), (34, 3), (255, 4), (257, 8), (515, 16)])
@pytest.mark.parametrize("fmt", ["ell", "hyb"])
def test_refinement_at_batch_edges(gk, n, half, prec, fmt):
    A, dense = _banded(n, half, 100 * n + half)
    b = np.random.default_rng(n).uniform(-1, 1, n)
    M = gk.Matrix(to_dev(A[0]), to_dev(A[1]), to_dev(A[2]), fmt=fmt)
    S = gk.Solver(M, gk.Precond(M, prec) if prec else None, "ir_cg", max_iters=5000, reduction_factor=1e-11)
    x = to_dev(np.zeros(n))
    st = gk.solve(S, to_dev(b), x)
    xh = to_np(x)
    assert st.stop_reason == gk.STOP_CONVERGED
    eps = np.finfo(np.float64).eps
    slack = (2 * half + 3) * eps * np.abs(dense).sum(axis=1).max() * np.abs(xh).max() * np.sqrt(n)
    assert np.linalg.norm(b - dense @ xh) <= 1e-11 * np.linalg.norm(b) + 2 * slack
