"""GK_CSR at the edges of its two rules for a slice's chain of loads: 16 slots
loaded ahead in small matrices (row lengths around multiples of 16 up to the
longest slice, 256, and row counts on both sides of the 16 slices per SM at
which the rule ends), and a few long slices among many short ones taken by
four warps each.  Every row of up to 256 entries is summed in increasing
column order throughout, so the products equal the oracle's bit for bit; the
advanced form adds one product and one sum, each rounded once; a longer row
and the fused dot product are sums of N terms in another order, off by at most
N eps times the sum of magnitudes on either side."""
import numpy as np
import pytest

from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu


def _csr(lengths, ncols, seed):
    g = np.random.default_rng(seed)
    ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    start = g.integers(0, ncols - int(lengths.max()) + 1, lengths.size)
    col = np.repeat(start - ptr[:-1], lengths) + np.arange(ptr[-1])
    return ptr, col.astype(np.int32), g.uniform(-1, 1, int(ptr[-1]))


@pytest.mark.parametrize("longest", [1, 8, 9, 15, 16, 17, 31, 32, 33, 48, 255, 256])
@pytest.mark.parametrize("n", [300, 1023])
def test_rows_around_the_batch(gk, orc, longest, n):
    lengths = np.random.default_rng(longest).integers(0, longest + 1, n)
    lengths[n // 2] = longest
    A = _csr(lengths, n, n + longest)
    x = np.random.default_rng(1).uniform(-1, 1, n)
    M = gk.Matrix(to_dev(A[0]), to_dev(A[1]), to_dev(A[2]), fmt="csr")
    y = to_dev(np.full(n, np.nan))
    gk.apply(M, to_dev(x), y)
    ref = orc.spmv(A, x)
    assert np.array_equal(to_np(y), ref)
    y0 = np.random.default_rng(2).uniform(-1, 1, n)
    ya = to_dev(y0)
    gk.apply_adv(2.0, M, to_dev(x), 0.5, ya)
    want = 2.0 * ref + 0.5 * y0
    assert np.all(np.abs(to_np(ya) - want) <= np.finfo(np.float64).eps * (np.abs(2.0 * ref) + np.abs(0.5 * y0)))


@pytest.mark.parametrize("slices", [-1, 0, 1])
def test_both_sides_of_the_line(gk, orc, slices):
    import torch
    n = 32 * (16 * torch.cuda.get_device_properties(0).multi_processor_count + slices)
    lengths = np.random.default_rng(5).integers(0, 21, n)
    A = _csr(lengths, n, 6)
    x = np.random.default_rng(7).uniform(-1, 1, n)
    M = gk.Matrix(to_dev(A[0]), to_dev(A[1]), to_dev(A[2]), fmt="csr")
    y = to_dev(np.full(n, np.nan))
    gk.apply(M, to_dev(x), y)
    assert np.array_equal(to_np(y), orc.spmv(A, x))


@pytest.mark.parametrize("longest", [65, 79, 80, 81, 255, 256])
@pytest.mark.parametrize("count", [1, 31, 33])
@pytest.mark.parametrize("very_long", [0, 600])
def test_few_long_slices(gk, orc, longest, count, very_long):
    import torch
    n = 32 * (16 * torch.cuda.get_device_properties(0).multi_processor_count + 40) + 5
    g = np.random.default_rng(longest + count)
    lengths = g.integers(0, 7, n)
    rows = g.choice(n, count + 1, replace=False)
    lengths[rows[:count]] = longest - np.arange(count) % 3
    if very_long:
        lengths[rows[count]] = very_long
    A = _csr(lengths, n, n)
    x = g.uniform(-1, 1, n)
    M = gk.Matrix(to_dev(A[0]), to_dev(A[1]), to_dev(A[2]), fmt="csr")
    y = to_dev(np.full(n, np.nan))
    gk.apply(M, to_dev(x), y)
    ref, got = orc.spmv(A, x), to_np(y)
    eps = np.finfo(np.float64).eps
    assert np.array_equal(got[lengths <= 256], ref[lengths <= 256])
    assert np.all(np.abs(got - ref) <= 2 * 600 * eps * 600)
    u = g.uniform(-1, 1, n)
    z, dot = to_dev(np.full(n, np.nan)), to_dev(np.zeros(1))
    gk.apply_dot(M, to_dev(x), z, to_dev(u), dot)
    assert np.array_equal(to_np(z)[lengths <= 256], ref[lengths <= 256])
    assert abs(to_np(dot)[0] - u @ to_np(z)) <= 2 * n * eps * (np.abs(u) @ np.abs(ref) + 1.0)
