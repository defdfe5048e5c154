"""BiCGSTAB's mid-size form: the whole solve in one cooperative launch (one
CTA per SM, grid-wide reductions through sequence-numbered words), chosen by
default without a preconditioner or with scalar Jacobi on 32,769 rows to
1,024 rows per CTA (155,648 on 152 SMs), rows of at most 64 entries.
Checked against the graph form and the oracle's SpMV (Section 3.1, criteria
of Section 2.5)."""
import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


def _solve(gk, A, b, x0=None, prec=None, **crit):
    n = A[0].size - 1
    M = gk.Matrix(to_dev(A[0]), to_dev(A[1]), to_dev(A[2]), fmt="csr")
    S = gk.Solver(M, gk.Precond(M, prec) if prec else None, "bicgstab", **crit)
    x = to_dev(np.zeros(n) if x0 is None else x0)
    return gk.solve(S, to_dev(b), x), to_np(x)


def _convdiff(ny, nx):
    """workloads.convdiff2d on a ragged ny x nx grid, the rows scaled by a
    varying factor so that the Jacobi diagonal is not constant."""
    offs = [(-1, 0), (0, -1), (0, 0), (0, 1), (1, 0)]
    rp, c, v = W._from_offsets((ny, nx), offs, [-1.0, -1.5, 4.5, -1.0, -1.0])
    scale = 1.0 + 0.5 * np.sin(np.arange(ny * nx))
    return rp, c, v * np.repeat(scale, np.diff(rp))


# 32,769 = 3 * 10,923 is the smallest size; 1 row per thread to 38,912 rows,
# 2 to 77,824, 4 above (152 SMs); ragged last CTAs
@pytest.mark.parametrize("shape", [(3, 10923), (150, 259), (151, 259), (277, 281), (394, 395)])
@pytest.mark.parametrize("prec", [None, 1])
def test_against_graph_form(gk, orc, shape, prec):
    """Same stop reason, iterations within max(3, 25 %) (BiCGSTAB's count is
    sensitive to rounding), two SpMVs per full iteration, the true residual
    from the oracle's SpMV within the tolerance's bar; run to run
    bit-identical."""
    A = _convdiff(*shape)
    n = A[0].size - 1
    b = orc.spmv(A, W.uniform_vector(n, 14))
    crit = dict(prec=prec, max_iters=20000, reduction_factor=1e-10)
    s1, x1 = _solve(gk, A, b, **crit)
    s2, x2 = _solve(gk, A, b, **crit)
    s0, _ = _solve(gk, A, b, check_every=-1, **crit)
    assert s1.form == gk.FORM_GRID and s0.form == gk.FORM_GRAPH
    assert s1.stop_reason == s0.stop_reason == gk.STOP_CONVERGED
    assert abs(s1.iters - s0.iters) <= max(3, s0.iters // 4), (s1.iters, s0.iters)
    assert s1.spmvs in (2 * s1.iters + 2, 2 * s1.iters + 1)
    assert s1.device_error == 0
    assert np.linalg.norm(b - orc.spmv(A, x1)) <= 1.5e-10 * np.linalg.norm(b)
    assert s1.iters == s2.iters and np.array_equal(x1, x2)


def test_exits(gk, orc):
    """A = c I converges at the first half step (one SpMV in the iteration);
    exact initial guess, zero right-hand side, iteration limits, NaN: as the
    graph form."""
    n = 40000
    b = W.uniform_vector(n, 15)
    s1, x1 = _solve(gk, W.scaled_identity(n, 2.5), b, max_iters=50, reduction_factor=1e-10)
    assert s1.form == gk.FORM_GRID and s1.stop_reason == gk.STOP_CONVERGED
    assert s1.iters == 1 and s1.spmvs == 3
    np.testing.assert_allclose(x1, b / 2.5, rtol=1e-14)
    A = _convdiff(200, 200)
    xs = W.uniform_vector(n, 16)
    bb = orc.spmv(A, xs)
    for c in (dict(b=bb, x0=xs), dict(b=np.zeros(n)), dict(b=bb, max_iters=0), dict(b=bb, max_iters=3),
              dict(b=np.full(n, np.nan), max_iters=50), dict(b=np.full(n, np.inf), max_iters=50)):
        bv, x0 = c.pop("b"), c.pop("x0", None)
        c.setdefault("reduction_factor", 1e-10)
        s1, x1 = _solve(gk, A, bv, x0=x0, **c)
        s0, x0g = _solve(gk, A, bv, x0=x0, check_every=-1, **c)
        assert s1.form == gk.FORM_GRID
        assert (s1.stop_reason, s1.iters, s1.spmvs) == (s0.stop_reason, s0.iters, s0.spmvs), c
        if s1.stop_reason != gk.STOP_NAN:
            np.testing.assert_allclose(x1, x0g, rtol=0, atol=1e-11 * max(1.0, np.abs(x0g).max()))


def test_selection(gk):
    """Below 32,769 rows, above 1,024 rows per CTA, with block Jacobi or a
    Time criterion: the graph form."""
    edge = _convdiff(128, 256)  # 32,768 rows
    assert _solve(gk, edge, W.uniform_vector(32768, 1), max_iters=3)[0].form == gk.FORM_GRAPH
    A = _convdiff(200, 200)
    b = W.uniform_vector(40000, 2)
    assert _solve(gk, A, b, max_iters=3)[0].form == gk.FORM_GRID
    assert _solve(gk, A, b, max_iters=3, prec=4)[0].form == gk.FORM_GRAPH
    assert _solve(gk, A, b, max_iters=3, time_limit_s=5.0)[0].form == gk.FORM_GRAPH
    big = _convdiff(400, 500)
    assert _solve(gk, big, W.uniform_vector(200000, 3), max_iters=3)[0].form == gk.FORM_GRAPH


@pytest.mark.parametrize("side,staged", [(33, True), (53, False)])
def test_27_point_staged_and_not(gk, orc, side, staged):
    """27-point stencils: on 33^3 a CTA's rows fit shared memory, on 53^3
    (26,000 entries per CTA) they do not."""
    A = W.stencil27(side)
    b = W.uniform_vector(side ** 3, 13)
    crit = dict(prec=1, max_iters=2000, reduction_factor=1e-10)
    s1, x1 = _solve(gk, A, b, **crit)
    s0, _ = _solve(gk, A, b, check_every=-1, **crit)
    assert s1.form == gk.FORM_GRID
    assert s1.stop_reason == s0.stop_reason == gk.STOP_CONVERGED
    assert abs(s1.iters - s0.iters) <= max(3, s0.iters // 4), (s1.iters, s0.iters)
    assert np.linalg.norm(b - orc.spmv(A, x1)) <= 1.5e-10 * np.linalg.norm(b)
