"""GPU MatMult on rectangular matrices in the two-CTAs-an-SM form: operators stacked on top of
one another (more rows than x has elements: an absent pattern entry's stand-in read has to stay
inside x) and side by side.  |y - y*| <= 1e-12 sum |a||x| per row against the oracle; the form
without patterns, which reads present entries only, gives the same bits.
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


# slices that end with an operator, slices that hold rows of two, three operators, side by side
@pytest.mark.parametrize("shape, corners, down, right", [
    ((48, 48, 48), True, 2, 1), ((49, 50, 51), False, 2, 1), ((38, 37, 39), False, 3, 1),
    ((53, 54, 55), False, 1, 2)])
def test_rectangular(shape, corners, down, right):
    n, i0, j0 = stencil(shape, corners)
    i = np.concatenate([i0 + k * n for k in range(down) for _ in range(right)]).astype(np.int32)
    j = np.concatenate([j0 + k * n for _ in range(down) for k in range(right)]).astype(np.int32)
    nr, nc = down * n, right * n
    rng = np.random.default_rng(n)
    v, x = rng.standard_normal(i.size), rng.standard_normal(nc)
    A = B.Mat.from_coo(nr, nc, t(i), t(j))
    A.set_values(t(v))
    s, sms = A.slices(), torch.cuda.get_device_properties(0).multi_processor_count
    assert A.plan()["kernel"] == B.SPMV_SELL and s["pattern_slices"] == s["nslices"]
    # the form's rule: a wave of two CTAs an SM, 16 slices each, and a mean width of 6
    assert (s["nslices"] + 15) // 16 >= 2 * sms and s["entries"] >= 6 * 32 * s["nslices"]
    O = oracle.coo_symbolic(nr, nc, i, j)
    oracle.coo_numeric(O, v)
    Oabs = oracle.CSR(O.nrows, O.ncols, O.row_ptr, O.col, O.perm, O.jmap, O.ncoo, np.abs(O.val))
    y = A.mult(t(x)).cpu().numpy()
    assert np.all(np.abs(y - oracle.spmv(O, x)) <= 1e-12 * oracle.spmv(Oabs, np.abs(x)) + 1e-300)
    A.set_slice_patterns(False)
    assert np.array_equal(A.mult(t(x)).cpu().numpy(), y)
    A.close()
