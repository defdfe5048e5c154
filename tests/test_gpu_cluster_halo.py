"""The one-cluster form of CG and BiCGSTAB with each CTA's rows and halo in its
shared memory: sizes around the 16 CTAs' row shares (ragged and empty last
CTAs, 1 to 8 rows per thread), and matrices whose halo does not fit, which
keep the form with the direction vector read across the cluster.  Against the
graph form and the oracle's SpMV."""
import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


def _solve(gk, A, b, kind, prec, **crit):
    M = gk.Matrix(*[to_dev(a) for a in A])
    S = gk.Solver(M, gk.Precond(M, prec) if prec else None, kind, max_iters=4000, reduction_factor=1e-10, **crit)
    x = to_dev(np.zeros(b.size))
    return gk.solve(S, to_dev(b), x), to_np(x)


def _check(gk, orc, A, kind, prec):
    n = A[0].size - 1
    b = orc.spmv(A, W.uniform_vector(n, 21))
    s1, x1 = _solve(gk, A, b, kind, prec)
    s2, x2 = _solve(gk, A, b, kind, prec)
    s0, _ = _solve(gk, A, b, kind, prec, check_every=-1)
    assert s1.form == gk.FORM_CLUSTER and s0.form == gk.FORM_GRAPH
    assert s1.stop_reason == s0.stop_reason == gk.STOP_CONVERGED and s1.device_error == 0
    slack = max(2, s0.iters * 3 // 100) if kind == "cg" else max(3, s0.iters // 4)
    assert abs(s1.iters - s0.iters) <= slack, (s1.iters, s0.iters)
    assert np.linalg.norm(b - orc.spmv(A, x1)) <= 1.5e-10 * np.linalg.norm(b)
    assert s1.iters == s2.iters and np.array_equal(x1, x2)


@pytest.mark.parametrize("shape", [(1, 1), (3, 5), (1, 17), (63, 65), (64, 64), (17, 241), (90, 91), (128, 128)])
@pytest.mark.parametrize("kind,prec", [("cg", None), ("cg", 1), ("bicgstab", 1)])
def test_row_shares(gk, orc, shape, kind, prec):
    _check(gk, orc, W.varcoef2d(np.exp(0.5 * np.random.default_rng(3).standard_normal(shape))), kind, prec)


@pytest.mark.parametrize("shape", [(128, 129), (181, 181)])
def test_row_shares_cg_only(gk, orc, shape):
    _check(gk, orc, W.varcoef2d(np.exp(0.5 * np.random.default_rng(4).standard_normal(shape))), "cg", 1)


@pytest.mark.parametrize("kind,n", [("cg", 32768), ("bicgstab", 16000)])
def test_scattered_columns(gk, orc, kind, n):
    """Ten random columns per row: nearly every other row is in the halo."""
    rng = np.random.default_rng(5)
    rows = np.repeat(np.arange(n), 10)
    cols = rng.integers(0, n, rows.size)
    r, c = np.concatenate([rows, cols]), np.concatenate([cols, rows])
    off = r != c
    rp, col, val = W._coo_to_csr(n, r[off], c[off], np.full(int(off.sum()), -0.02))
    d = np.arange(n)
    row_of = np.repeat(d, np.diff(rp))
    A = W._coo_to_csr(n, np.concatenate([row_of, d]), np.concatenate([col.astype(np.int64), d]),
                      np.concatenate([val, np.full(n, 2.0)]))
    _check(gk, orc, A, kind, 1)
