"""GPU assembly at the edges of its kernels' ranges, bit for bit against the oracle:
rows at the sizes where the row sorts change (8, 16, 32, 64 and 4096 entries), runs of
equal rows that start, end and break anywhere in a warp, ignored entries, slices and
tiles at and beyond what a numeric tile's shared memory holds, INSERT and ADD.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_08646_gb300 import binding as B  # noqa: E402

DEV = "cuda"


def t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def check(n, m, i, j, seed):
    i, j = np.asarray(i, np.int32), np.asarray(j, np.int32)
    rng = np.random.default_rng(seed)
    v = rng.standard_normal(i.size)
    A = B.Mat.from_coo(n, m, t(i), t(j))
    O = oracle.coo_symbolic(n, m, i, j)
    for mode in (B.INSERT, B.ADD, B.INSERT):
        A.set_values(t(v), mode=mode)
        oracle.coo_numeric(O, v, mode=mode)
        rp, col, val = (x.cpu().numpy() for x in A.csr())
        perm, jmap = (x.cpu().numpy() for x in A.coo_maps())
        assert np.array_equal(rp, O.row_ptr) and np.array_equal(col, O.col)
        assert np.array_equal(perm, O.perm) and np.array_equal(jmap, O.jmap)
        assert val.tobytes() == O.val.tobytes()
        v = v * 1.7
    x = rng.standard_normal(m)
    y = A.mult(t(x)).cpu().numpy()              # the sliced copy's values too
    Oabs = oracle.CSR(O.nrows, O.ncols, O.row_ptr, O.col, O.perm, O.jmap, O.ncoo, np.abs(O.val))
    assert np.all(np.abs(y - oracle.spmv(O, x)) <= 1e-12 * oracle.spmv(Oabs, np.abs(x)) + 1e-300)
    A.close()


def rows_of(counts, m, rng, distinct):
    """One row per count, its entries over `distinct` columns, in random order."""
    i = np.repeat(np.arange(len(counts)), counts)
    j = rng.integers(0, min(distinct, m), i.size) * (m // min(distinct, m))
    p = rng.permutation(i.size)
    return i[p], j[p]


@pytest.mark.parametrize("top", [1, 8, 9, 16, 17, 32, 33, 64, 65, 100, 1000, 4096, 4097])
@pytest.mark.parametrize("distinct", [3, 5000])
def test_row_sort_classes(top, distinct):
    rng = np.random.default_rng(top)
    counts = [0, 1, top, 0, min(top, 7)] + list(rng.integers(0, min(top, 70) + 1, 60)) + [top, 0]
    m = 5000
    i, j = rows_of(counts, m, rng, distinct)
    check(len(counts), m, i, j, top)


@pytest.mark.parametrize("run", [1, 2, 7, 8, 31, 32, 33, 129])
def test_runs_of_equal_rows(run):
    """COO entries in runs of one row, with ignored entries among them."""
    rng = np.random.default_rng(run)
    i = np.repeat(rng.integers(0, 41, 400), run)
    j = (i + rng.integers(-3, 4, i.size)) % 41
    i[rng.random(i.size) < 0.1] = -1
    j[rng.random(i.size) < 0.1] = -1
    check(41, 41, i, j, run)


@pytest.mark.parametrize("width,dup", [(1, 1), (5, 3), (27, 4), (32, 3), (33, 1), (31, 4), (40, 2)])
def test_numeric_tiles_of_slices(width, dup):
    """Bands of `width` columns, every entry given `dup` times: slices of up to 1280
    nonzeros (1024 fit a tile) and 3968 COO entries (3072 fit)."""
    n = 333
    r = np.arange(n)
    i = np.repeat(r, width)
    j = i + np.tile(np.arange(width), n) - width // 2
    j = np.where((j >= 0) & (j < n), j, i)
    i, j = np.tile(i, dup), np.tile(j, dup)
    p = np.random.default_rng(width).permutation(i.size)
    check(n, n, i[p], j[p], width)


def test_long_segments_and_empty_tiles():
    """A nonzero of more terms than a tile holds, beside empty rows."""
    i = np.concatenate([np.full(3500, 2), np.arange(100), np.full(9, 99)])
    j = np.concatenate([np.full(3500, 2), np.arange(100), np.arange(9)])
    check(130, 130, i, j, 5)
