"""GPU MatMult where its kernel changes -- the two-CTAs-an-SM form from one wave of slices
and a mean slice width of 6 on -- and CSR-vector row products in length order: windows of
512 rows (MatMult) and blocks (solves) that end anywhere, equal and extreme lengths, empty
rows.  |y - y*| <= 1e-12 sum |a||x| per row against the oracle; a row's own sum does not
depend on the order rows are dealt in.
"""
import numpy as np
import pytest

import oracle
from paper_2406_08646_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_08646_gb300 import binding as B  # noqa: E402

DEV = "cuda"


def t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def check(A, n, i, j, v, seed):
    O = oracle.coo_symbolic(n, n, i, j)
    oracle.coo_numeric(O, v)
    Oabs = oracle.CSR(O.nrows, O.ncols, O.row_ptr, O.col, O.perm, O.jmap, O.ncoo, np.abs(O.val))
    x = np.random.default_rng(seed).standard_normal(n)
    y = A.mult(t(x)).cpu().numpy()
    assert np.all(np.abs(y - oracle.spmv(O, x)) <= 1e-12 * oracle.spmv(Oabs, np.abs(x)) + 1e-300)
    return O, x, y


# 152 SMs: one wave of the form is 304 CTAs of 16 slices, 155,648 rows
@pytest.mark.parametrize("shape", [(53, 54, 54), (54, 53, 55), (54, 54, 55), (395, 400), (61, 67, 71)])
def test_sliced_forms(shape):
    ea, eb = W.grid_edges(shape)
    k = 10.0 ** np.random.default_rng(5).uniform(-1, 1, ea.shape[0])
    n = int(np.prod(shape))
    i, j, v = W.edge_coo(ea, eb, k)
    A = B.Mat.from_coo(n, n, t(i), t(j))
    A.set_values(t(v))
    _, x, y = check(A, n, i, j, v, n)
    A.set_slice_patterns(False)      # column indices: the other form, the same sums
    assert np.array_equal(A.mult(t(x)).cpu().numpy(), y)
    A.close()


@pytest.mark.parametrize("n", [31, 511, 512, 513, 1025, 2500])
@pytest.mark.parametrize("kernel", [1, 2, 4, 8])
def test_rows_in_length_order(n, kernel):
    rng = np.random.default_rng(n)
    deg = np.minimum(rng.integers(0, 9, n) ** 2, n - 1)
    deg[rng.random(n) < 0.1] = 0
    a = np.repeat(np.arange(n), deg)
    b = (a + 1 + rng.integers(0, n - 1, a.size)) % n
    k = rng.uniform(0.1, 1.0, a.size)
    own = np.arange(n)
    i = np.concatenate([a, b, a, b, own]).astype(np.int32)
    j = np.concatenate([a, b, b, a, own]).astype(np.int32)
    v = np.concatenate([k, k, -k, -k, np.full(n, 0.3)])
    A = B.Mat.from_coo(n, n, t(i), t(j))
    A.set_values(t(v))
    A.set_plan(kernel=kernel)
    O, x, _ = check(A, n, i, j, v, n)
    for rows in (0, 32, 96):         # blocks of the solves' table
        A.set_plan(spmv_rows=rows, kernel=kernel)
        xs, r = A.solve(t(x), rtol=1e-10)
        _, ro = oracle.pcg(O, x, rtol=1e-10)
        assert r["status"] == B.OK
        assert abs(r["iterations"] - ro["iterations"]) <= max(2, 0.01 * ro["iterations"])
        assert np.linalg.norm(x - oracle.spmv(O, xs.cpu().numpy())) <= 1.05e-10 * np.linalg.norm(x)
    A.close()
