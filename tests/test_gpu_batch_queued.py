"""Batched solves without a status read-back return before they have run: the
vectors of each are those of its own call, whatever the caller does next."""
import numpy as np
import pytest

import workloads as W
from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["cg", "bicgstab", "ir_cg"])
def test_queued_solves_keep_their_vectors(gk, kind):
    import torch
    ptr, A = W.batch_varcoef2d(30, seed=8)
    n = int(ptr[-1])
    B = gk.Batch(ptr, *[to_dev(a) for a in A])
    bs = [to_dev(W.uniform_vector(n, k)) for k in (1, 2, 3)]
    crit = dict(max_iters=4000, reduction_factor=1e-10)
    want = []
    for b in bs:
        x = to_dev(np.zeros(n))
        B.solve(b, x, kind, **crit)
        want.append(to_np(x))
    xs = [to_dev(np.zeros(n)) for _ in bs]
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(20_000_000)  # the calls return while the stream is busy
        for b, x in zip(bs, xs):
            B.solve(b, x, kind, status=False, **crit)
    assert not s.query()
    torch.cuda.synchronize()
    for x, w in zip(xs, want):
        assert np.array_equal(to_np(x), w)
