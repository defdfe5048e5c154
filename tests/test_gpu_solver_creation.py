"""Generating solvers: what it costs a program that makes one per step, and
that it leaves other threads alone."""
import threading
import time

import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,side", [(k, s) for k in ("cg", "bicgstab", "fcg", "gmres") for s in (8, 64, 128)
                                       if (k, s) != ("gmres", 128)])  # whose basis is too large for a shared chunk
def test_generation_of_small_solvers(gk, kind, side):
    """A solver of a small system was made and destroyed in 35 to 60 us while
    the operator's arrays kept its chunk of memory mapped, in 500 to 600 where
    nothing did.  The bar lies between, for the median of 30."""
    import torch
    M = gk.Matrix(*[to_dev(a) for a in W.poisson2d(side)])
    P = gk.Precond(M, 1)
    took = []
    for _ in range(33):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        S = gk.Solver(M, P, kind, max_iters=10, reduction_factor=1e-10)
        del S
        took.append(time.perf_counter() - t0)
    assert sorted(took[3:])[15] <= 250e-6, sorted(took[3:])


@pytest.mark.parametrize("kind,side", [("cg", 30), ("bicgstab", 30), ("cg", 200), ("bicgstab", 200)])
def test_generated_while_another_thread_captures(gk, kind, side):
    import torch
    M = gk.Matrix(*[to_dev(a) for a in W.poisson2d(side)])
    acc = torch.zeros(8, device="cuda:0")
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    begun, go_on, failed = threading.Event(), threading.Event(), []

    def capture():
        try:
            with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                acc.add_(1.0)
                begun.set()
                go_on.wait()
                acc.add_(1.0)
        except Exception as e:  # noqa: BLE001
            failed.append(e)
            begun.set()

    t = threading.Thread(target=capture)
    t.start()
    begun.wait()
    try:
        S = gk.Solver(M, None, kind, max_iters=2000, reduction_factor=1e-8)
    finally:
        go_on.set()
        t.join()
    assert not failed, failed
    graph.replay()
    torch.cuda.synchronize()
    assert acc.tolist() == [2.0] * 8
    x = to_dev(np.zeros(side * side))
    assert gk.solve(S, to_dev(W.uniform_vector(side * side, 1)), x).stop_reason == gk.STOP_CONVERGED
    assert np.all(np.isfinite(to_np(x)))
