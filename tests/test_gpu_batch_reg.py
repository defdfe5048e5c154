"""Batched refinement with each system's rows in registers: block sizes that
give 1 to 8 rows per thread, 5 and up to 8 entries a row (and wider systems,
which keep the shared-memory form), ragged sizes, other vectors on the same
handle.  Every system meets the FP64 criterion against its own operator."""
import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


def _systems(sizes, width, seed):
    """Block-diagonal SPD systems: a diagonal and (width - 1) / 2 random
    neighbours to either side, symmetric, diagonally dominant."""
    rng = np.random.default_rng(seed)
    rows, cols, vals, ptr = [], [], [], np.concatenate([[0], np.cumsum(sizes)])
    for r0, n in zip(ptr[:-1], sizes):
        i = np.arange(n)
        diag = np.full(n, 0.1)
        for d in range(1, (width + 1) // 2):
            v = -rng.uniform(0.5, 1.5, n)
            k = i[: max(n - d, 0)]
            for a, b in ((k, k + d), (k + d, k)):
                rows.append(r0 + a)
                cols.append(r0 + b)
                vals.append(v[k])
            diag[k] -= v[k]
            diag[k + d] -= v[k]
        rows.append(r0 + i)
        cols.append(r0 + i)
        vals.append(diag)
    n = int(ptr[-1])
    return ptr, W._coo_to_csr(n, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals))


@pytest.mark.parametrize("threads", [32, 64, 128, 256])
@pytest.mark.parametrize("width", [5, 7, 9])
@pytest.mark.parametrize("jacobi", [True, False])
def test_every_system_meets_the_criterion(gk, orc, threads, width, jacobi):
    sizes = [1, 2, 31, 32, 33, 64, 65, 127, 129, 255, 256, 257, 500, 512, 513, 1000, 1024]
    ptr, A = _systems(sizes, width, 7)
    n = int(ptr[-1])
    B = gk.Batch(ptr, *[to_dev(a) for a in A])
    B.set_threads([threads] * gk.BATCH_CLASSES, "ir_cg", jacobi)
    for seed in (1, 2):  # other vectors on the same handle
        b = W.uniform_vector(n, seed)
        x = to_dev(np.zeros(n))
        st = B.solve(to_dev(b), x, "ir_cg", jacobi=jacobi, max_iters=20000, reduction_factor=1e-11)
        assert np.all(st["stop_reason"] == gk.STOP_CONVERGED), st["stop_reason"]
        r = b - orc.spmv(A, to_np(x))
        for s in range(len(sizes)):
            rs, bs = r[ptr[s]:ptr[s + 1]], b[ptr[s]:ptr[s + 1]]
            assert np.linalg.norm(rs) <= 1.5e-11 * np.linalg.norm(bs), (s, sizes[s])
        x2 = to_dev(np.zeros(n))
        st2 = B.solve(to_dev(b), x2, "ir_cg", jacobi=jacobi, max_iters=20000, reduction_factor=1e-11)
        assert np.array_equal(to_np(x), to_np(x2)) and np.array_equal(st["iters"], st2["iters"])
