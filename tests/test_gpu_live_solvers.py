"""Several handles alive at once.  The one-launch solvers and the batched ones
ask for as much dynamic shared memory as their own system needs, and the limit
on it belongs to the kernel: a handle made for a smaller system afterwards
must not take away what the larger one's launches need."""
import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


def _grid5(ny, nx, upwind):
    offs = [(-1, 0), (0, -1), (0, 0), (0, 1), (1, 0)]
    return W._from_offsets((ny, nx), offs, [-1.0, -1.5, 4.5, -1.0, -1.0] if upwind else [-1.0, -1.0, 4.0, -1.0, -1.0])


def _scattered(n, seed):
    """A few random columns a row: halos that do not fit shared memory."""
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(n), 10)
    cols = rng.integers(0, n, rows.size)
    r, c = np.concatenate([rows, cols, np.arange(n)]), np.concatenate([cols, rows, np.arange(n)])
    v = np.where(r == c, 2.0, -0.02)
    key, first = np.unique(r * n + c, return_index=True)
    return W._coo_to_csr(n, key // n, key % n, v[first])


def _solver(gk, A, kind, prec):
    M = gk.Matrix(*[to_dev(a) for a in A])
    return gk.Solver(M, gk.Precond(M, 1) if prec else None, kind, max_iters=30, reduction_factor=1e-10)


def _x(gk, S, b):
    x = to_dev(np.zeros(b.size))
    return gk.solve(S, to_dev(b), x), to_np(x)


@pytest.mark.parametrize("kind", ["cg", "bicgstab"])
@pytest.mark.parametrize("prec", [False, True])
@pytest.mark.parametrize("form,large,small", [
    ("grid", (201, 199), (200, 199)), ("grid", (256, 256), (230, 230)), ("grid", (300, 305), (270, 300)),
    ("cluster", (64, 64), (60, 60)), ("cluster", (120, 130), (100, 130)), ("cluster", (20, 20), (19, 20))])
def test_a_smaller_solver_made_later(gk, kind, prec, form, large, small):
    A = _grid5(*large, kind == "bicgstab")
    b = W.uniform_vector(A[0].size - 1, 5)
    S1 = _solver(gk, A, kind, prec)
    st, want = _x(gk, S1, b)
    assert st.form == (gk.FORM_GRID if form == "grid" else gk.FORM_CLUSTER)
    S2 = _solver(gk, _grid5(*small, kind == "bicgstab"), kind, prec)
    again, got = _x(gk, S1, b)
    assert again.form == st.form and again.iters == st.iters and np.array_equal(got, want)
    _x(gk, S2, W.uniform_vector(small[0] * small[1], 6))


def test_a_smaller_solver_made_later_across_the_cluster(gk):
    """The kernels that read the direction vector across the cluster."""
    A = _scattered(32768, 7)
    b = W.uniform_vector(32768, 8)
    S1 = _solver(gk, A, "cg", True)
    st, want = _x(gk, S1, b)
    assert st.form == gk.FORM_CLUSTER
    S2 = _solver(gk, _scattered(30000, 9), "cg", True)
    _, got = _x(gk, S1, b)
    assert np.array_equal(got, want)
    _x(gk, S2, W.uniform_vector(30000, 6))


@pytest.mark.parametrize("kind", ["cg", "bicgstab", "ir_cg"])
def test_a_smaller_batch_made_later(gk, kind):
    large = W.batch_varcoef2d(40, seed=5)
    small = W.batch_varcoef2d(7, seed=6)
    B1, B2 = (gk.Batch(p, *[to_dev(a) for a in A]) for p, A in (large, small))
    b1, b2 = (to_dev(W.uniform_vector(int(p[-1]), 7)) for p, _ in (large, small))

    def solve(B, b, iters):
        x = to_dev(np.zeros(b.numel()))
        B.solve(b, x, kind, max_iters=iters, reduction_factor=1e-10)
        return to_np(x)

    want = solve(B1, b1, 2000)
    solve(B2, b2, 2000)
    assert np.array_equal(solve(B1, b1, 2000), want)
    assert solve(B1, b1, 1999).shape == want.shape  # other criteria: planned anew
    solve(B2, b2, 1999)
    assert np.array_equal(solve(B1, b1, 2000), want)
