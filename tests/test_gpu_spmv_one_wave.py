"""GPU MatMult where its form changes: the one-wave form (alike slices, wide ones, or narrow
ones that stream from HBM) on operators stacked on top of one another -- more rows than x has
elements: an absent pattern entry's stand-in read has to stay inside x -- and the general form on
the other side of the rule's lines (uneven slices, too few, too many or small ones, operators side
by side).  |y - y*| <= 1e-12 sum |a||x| per row against the oracle; the general form without
patterns gives the same bits.
"""
import itertools

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_08646_gb300 import binding as B  # noqa: E402

DEV = "cuda"


def t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def stencil(shape, corners):
    """Rows and columns of the 27-point (corners) or 7-point stencil on a grid."""
    g = np.arange(int(np.prod(shape))).reshape(shape)
    i, j = [], []
    for off in itertools.product((-1, 0, 1), repeat=3):
        if corners or sum(map(abs, off)) <= 1:
            i.append(g[tuple(slice(max(0, -o), s - max(0, o)) for o, s in zip(off, shape))].ravel())
            j.append(g[tuple(slice(max(0, o), s - max(0, -o)) for o, s in zip(off, shape))].ravel())
    return g.size, np.concatenate(i), np.concatenate(j)


def stacked(shape, corners, down, right):
    n, i, j = stencil(shape, corners)
    return (down * n, right * n, np.concatenate([i + k * n for k in range(down) for _ in range(right)]),
            np.concatenate([j + k * n for _ in range(down) for k in range(right)]))


def uneven():
    """27-point rows above as many diagonal rows."""
    n, i, j = stencil((56, 56, 56), True)
    g = np.arange(n, 2 * n)
    return 2 * n, 2 * n, np.concatenate([i, g]), np.concatenate([j, g])


CASES = {
    "wide, tall": (True, lambda: stacked((56, 56, 56), True, 2, 1)),
    "wide, square": (True, lambda: stacked((62, 63, 64), True, 1, 1)),
    "wide, too few slices": (False, lambda: stacked((48, 48, 48), True, 2, 1)),
    "wide, too many slices": (False, lambda: stacked((105, 104, 104), True, 1, 1)),
    "streaming, tall": (True, lambda: stacked((125, 126, 127), False, 2, 1)),
    "narrow and in cache, tall": (False, lambda: stacked((49, 50, 51), False, 2, 1)),
    "side by side": (False, lambda: stacked((53, 54, 55), False, 1, 2)),
    "uneven": (False, uneven),
}


@pytest.mark.parametrize("name", list(CASES))
def test_forms(name):
    one_wave, make = CASES[name]
    nr, nc, i, j = make()
    i, j = i.astype(np.int32), j.astype(np.int32)
    rng = np.random.default_rng(nr)
    v, x = rng.standard_normal(i.size), rng.standard_normal(nc)
    A = B.Mat.from_coo(nr, nc, t(i), t(j))
    A.set_values(t(v))
    s, dev = A.slices(), torch.cuda.get_device_properties(0)
    ns, entries = s["nslices"], s["entries"]
    assert A.plan()["kernel"] == B.SPMV_SELL and s["pattern_slices"] == ns
    # the form by its rule: alike slices, width, then waves of slices or bytes and reach
    even = 8 * np.bincount(i // 32).max() * ns <= 9 * i.size
    width, wave = entries / (32 * ns), 2 * dev.multi_processor_count * 16
    far = np.abs(i.astype(np.int64) - j).max() >= 8192
    streams = 4 * (8 * entries + 20 * nr) >= 7 * dev.L2_cache_size
    assert one_wave == bool(even and (1.5 * wave <= ns < 7 * wave if width >= 24
                                      else 6 <= width <= 12 and far and streams))
    O = oracle.coo_symbolic(nr, nc, i, j)
    oracle.coo_numeric(O, v)
    Oabs = oracle.CSR(O.nrows, O.ncols, O.row_ptr, O.col, O.perm, O.jmap, O.ncoo, np.abs(O.val))
    y = A.mult(t(x)).cpu().numpy()
    assert np.all(np.abs(y - oracle.spmv(O, x)) <= 1e-12 * oracle.spmv(Oabs, np.abs(x)) + 1e-300)
    A.set_slice_patterns(False)
    assert np.array_equal(A.mult(t(x)).cpu().numpy(), y)
    A.close()
