"""GPU numeric COO stage without a sliced copy: tiles from 512 nonzeros down to one warp's, by the
number of nonzeros and the mean number of entries of one, with lengths that vary around it (tiles
that fit shared memory beside ones that do not); and patterns of few rows, whose entries cannot
fit the row counts.  Bits of the oracle's sums in increasing COO index.
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


@pytest.mark.parametrize("mean", [1, 4, 5, 9, 24, 36, 71, 73, 150, 900])
@pytest.mark.parametrize("n", [1, 31, 777])
def test_vector_tiles(n, mean):
    rng = np.random.default_rng(100 * n + mean)
    i = rng.integers(0, n, n * mean)
    i = np.concatenate([i, rng.integers(0, max(1, n // 20), n * mean // 4)]).astype(np.int32)
    v = rng.standard_normal(i.size) * 10.0 ** rng.uniform(-3, 3, i.size)
    y0 = rng.standard_normal(n)
    V = B.Vec(n, t(i))
    for mode in (B.INSERT, B.ADD):
        y = V.set_values(t(v), t(y0), mode).cpu().numpy()
        assert y.tobytes() == oracle.vec_set_values_coo(n, i, v, mode, y0).tobytes(), mode
    V.close()


@pytest.mark.parametrize("n, m", [(1, 4096), (1, 4097), (3, 12289), (7, 40000)])
def test_few_rows(n, m):
    rng = np.random.default_rng(m)
    i, j = rng.integers(0, n, m).astype(np.int32), rng.integers(-1, n, m).astype(np.int32)
    v = rng.standard_normal(m)
    A = B.Mat.from_coo(n, n, t(i), t(j))
    A.set_values(t(v))
    O = oracle.coo_symbolic(n, n, i, j)
    oracle.coo_numeric(O, v)
    got = [x.cpu().numpy() for x in (*A.csr(), *A.coo_maps())]
    want = [O.row_ptr, O.col, O.val, O.perm, O.jmap]
    assert all(np.array_equal(g, w[:g.size]) for g, w in zip(got, want))
    A.close()
