"""Creation of the CSR operator on the device: the copy, the checks of the
caller's arrays, the length-sorted slices, the hybrid split.  Plans are
checked through gk_matrix_get_info against numpy, and through the applies
against the oracle's ordered SpMV, at the edges of the passes' tiles (32 rows
of a warp, 1,024 rows of a block) and of the row-length classes (256 entries
of a slice, 512 of a piece)."""
import numpy as np
import pytest

from helpers import to_dev, to_np

pytestmark = pytest.mark.gpu

LENGTHS = {
    "short": (0, 1, 7),
    "slice edge": (0, 3, 255, 256),
    "long": (0, 5, 256, 257, 511, 512, 513, 1024, 1030),
}


def _csr(n, lengths, seed, n_cols=1100):
    rng = np.random.default_rng(seed)
    lens = rng.choice(lengths, size=n)
    if max(lengths) > 256:  # mostly short rows, so that the matrix stays small
        lens[rng.random(n) < 0.95] = 5
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    col = np.concatenate([np.sort(rng.choice(n_cols, size=k, replace=False)) for k in lens] or [[]]).astype(np.int32)
    return (rp, col, rng.standard_normal(col.size)), lens, n_cols


def _hyb(lens, n):
    """The smallest width minimising 12 K n + 16 overflow."""
    cost = [k * n * 12 + np.maximum(lens - k, 0).sum() * 16 for k in range(int(lens.max(initial=0)) + 1)]
    K = int(np.argmin(cost))
    return K, int((lens > K).sum()), int(np.maximum(lens - K, 0).sum())


@pytest.mark.parametrize("kind", list(LENGTHS))
@pytest.mark.parametrize("n", [1, 31, 33, 1023, 1024, 1025, 2500])
@pytest.mark.parametrize("host", [False, True])
def test_plans_and_applies(gk, orc, kind, n, host):
    A, lens, n_cols = _csr(n, LENGTHS[kind], n)
    arrays = A if host else [to_dev(a) for a in A]
    x = np.random.default_rng(n + 1).standard_normal(n_cols)
    want, bound = orc.spmv_accurate(A, x)
    ordered = orc.spmv(A, x)
    for fmt in ("csr", "csr_merge", "hyb", "auto"):
        M = gk.Matrix(*arrays, n_cols=n_cols, fmt=fmt)
        info = M.info()
        if fmt == "csr":
            assert info["long_rows"] == int((lens > 256).sum())
            assert info["split_rows"] == int((lens > 512).sum())
            assert info["short_items"] == (int((lens <= 256).sum()) + 31) // 32
        if fmt == "hyb":
            assert (info["ell_width"], info["tail_rows"], info["tail_nnz"]) == _hyb(lens, n)
        y = to_dev(np.full(n, np.nan))
        gk.apply(M, to_dev(x), y)
        y = to_np(y)
        assert np.all(np.abs(y - want) <= 1e-13 * bound + 1e-300), fmt
        if fmt == "csr":  # rows of up to 256 entries are summed in the oracle's order
            assert np.array_equal(y[lens <= 256], ordered[lens <= 256])


@pytest.mark.parametrize("n", [40, 1100])
@pytest.mark.parametrize("where", [0, 31, 32, 127, 128, 129])
@pytest.mark.parametrize("host", [False, True])
def test_bad_columns(gk, n, where, host):
    """A column out of range, unsorted or repeated at entry `where`, and again
    in the last row: refused, and the first bad row is named."""
    rows = np.arange(n)
    col = np.stack([rows % 7, 10 + rows % 5, 20 + rows], 1).astype(np.int32).ravel()
    rp = (3 * np.arange(n + 1)).astype(np.int32)
    val = np.ones(col.size)
    where = min(where, col.size - 1)
    before = np.int32(-1) if where % 3 == 0 else col[where - 1]  # of the same row
    for bad in (np.int32(-1), np.int32(n + 20), before):
        c = col.copy()
        c[where] = bad
        c[-1] = -5
        arrays = [rp, c, val] if host else [to_dev(a) for a in (rp, c, val)]
        with pytest.raises(gk.GkError) as e:
            gk.Matrix(*arrays, n_cols=n + 20)
        assert e.value.code == 5 and f"row {where // 3}:" in str(e.value), (bad, str(e.value))


def test_bad_row_pointers(gk):
    """Refused in the order first pointer, first decrease, last pointer; the
    entries are not read then."""
    n = 3000
    good = np.arange(n + 1, dtype=np.int32)
    col = np.zeros(n, np.int32)
    val = np.ones(n)
    for change, text in (((0, 1), "rowptr[0] = 1"), ((1500, 5000), "decreases at row 1500"),
                         ((2000, -7), "decreases at row 1999"), ((n, n - 1), f"rowptr[n_rows] = {n - 1}")):
        rp = good.copy()
        rp[change[0]] = change[1]
        with pytest.raises(gk.GkError) as e:
            gk.Matrix(to_dev(rp), to_dev(col), to_dev(val), n_cols=n)
        assert e.value.code == 5 and text in str(e.value), str(e.value)
