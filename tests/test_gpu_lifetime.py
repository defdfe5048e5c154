"""Handles destroyed while work that uses them is still running: their arrays
come from the stream-ordered pool, which hands freed memory out again at
once: the destroying call waits for the device, or frees them in the order of
the default stream where they were used on no other."""
import threading

import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu

BUSY = 100_000_000  # cycles of torch's sleep kernel: tens of milliseconds ahead of the apply


def _operator(gk, A, fmt="csr"):
    return gk.Matrix(*[to_dev(a) for a in A], fmt=fmt)


@pytest.mark.parametrize("what", ["csr", "csr_merge", "ell", "hyb", "jacobi", "block jacobi"])
def test_destroyed_with_an_apply_in_flight(gk, orc, what):
    """An apply waits in a busy stream when its handle goes; then another
    operator of the same size, with other columns and values, is made on a
    second stream.  The first apply's result is the first operator's."""
    import torch
    ny, nx = 300, 401
    n = ny * nx
    A = W.varcoef2d(np.exp(0.5 * np.random.default_rng(1).standard_normal((ny, nx))))
    B = W.varcoef2d(np.exp(0.5 * np.random.default_rng(2).standard_normal((nx, ny))))
    b_dev = [to_dev(a) for a in B]
    x = to_dev(W.uniform_vector(n, 3))
    fmt = what if "jacobi" not in what else "csr"
    M = _operator(gk, A, fmt)
    P = gk.Precond(M, 1 if what == "jacobi" else 8) if "jacobi" in what else None
    want = torch.empty_like(x)
    gk.precond_apply(P, x, want) if P else gk.apply(M, x, want)
    if not P:
        assert np.allclose(to_np(want), orc.spmv(A, to_np(x)), rtol=0, atol=1e-10)
    y = torch.full_like(x, float("nan"))
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(BUSY)
        gk.precond_apply(P, x, y) if P else gk.apply(M, x, y)
        done.record()
    assert not done.query()  # else nothing is tested
    P = None
    M = None
    assert done.query()  # the destroying call has waited
    with torch.cuda.stream(s2):
        other = gk.Matrix(*b_dev, fmt=fmt)
        Q = gk.Precond(other, 8)
    torch.cuda.synchronize()
    assert np.array_equal(to_np(y), to_np(want))
    del Q


@pytest.mark.parametrize("what", ["csr", "csr_merge", "ell", "hyb", "jacobi", "block jacobi"])
@pytest.mark.parametrize("same", [True, False])
def test_destroyed_with_an_apply_in_flight_on_the_default_stream(gk, what, same):
    """As above on the default stream, in whose order the arrays are freed;
    the next operators are made on it or on another stream."""
    import torch
    ny, nx = 300, 401
    n = ny * nx
    A, B = (W.varcoef2d(np.exp(0.5 * np.random.default_rng(k).standard_normal(s))) for k, s in
            ((1, (ny, nx)), (2, (nx, ny))))
    b_dev = [to_dev(a) for a in B]
    x = to_dev(W.uniform_vector(n, 3))
    fmt = what if "jacobi" not in what else "csr"
    M = _operator(gk, A, fmt)
    P = gk.Precond(M, 1 if what == "jacobi" else 8) if "jacobi" in what else None
    want = torch.empty_like(x)
    gk.precond_apply(P, x, want) if P else gk.apply(M, x, want)
    y = torch.full_like(x, float("nan"))
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    torch.cuda._sleep(BUSY)
    gk.precond_apply(P, x, y) if P else gk.apply(M, x, y)
    done.record()
    P = None
    M = None
    assert not done.query()  # freed in order, without a wait
    with torch.cuda.stream(torch.cuda.default_stream() if same else torch.cuda.Stream()):
        others = [gk.Matrix(*b_dev, fmt=fmt) for _ in range(2)]
        Q = [gk.Precond(o, 8) for o in others]
    torch.cuda.synchronize()
    assert np.array_equal(to_np(y), to_np(want))
    del Q, others


def test_destroyed_while_another_thread_captures(gk):
    """The wait does not disturb a capture in another thread's stream."""
    import torch
    A = W.poisson2d(40)
    M = _operator(gk, A)
    x = to_dev(W.uniform_vector(1600, 4))
    y = torch.empty_like(x)
    gk.apply(M, x, y)
    want = to_np(y)
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
    M = None
    go_on.set()
    t.join()
    assert not failed, failed
    graph.replay()
    torch.cuda.synchronize()
    assert acc.tolist() == [2.0] * 8
    M = _operator(gk, A)
    gk.apply(M, x, y)
    assert np.array_equal(to_np(y), want)
