"""GPU: which systems the automatic choice gives to teams of CTAs, on both sides of its lines --
rows whose lengths differ from place to place (the longest run of slices against the mean), and
matrices without column patterns by their size -- and the solution either way: residual and
oracle iteration counts as in the phase kernels' tests.
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


def stencil27(side):
    g = np.arange(side ** 3).reshape((side,) * 3)
    i, j, v = [], [], []
    for off in itertools.product((-1, 0, 1), repeat=3):
        i.append(g[tuple(slice(max(0, -o), side - max(0, o)) for o in off)].ravel())
        j.append(g[tuple(slice(max(0, o), side - max(0, -o)) for o in off)].ravel())
        v.append(np.full(i[-1].size, -1.0 if any(off) else 26.5))
    return g.size, np.concatenate(i), np.concatenate(j), np.concatenate(v)


def uneven(side, extra):
    """27-point rows followed by diagonal ones."""
    n, i, j, v = stencil27(side)
    d = np.arange(n, n + extra)
    return n + extra, np.concatenate([i, d]), np.concatenate([j, d]), np.concatenate([v, np.full(extra, 2.0)])


def scattered(n):
    """Nine entries a row, eight of them anywhere."""
    rng, a = np.random.default_rng(n), np.arange(n)
    i, j, v = [a], [a], [np.full(n, 8.2)]
    for _ in range(4):
        p = rng.permutation(n)
        i += [a, p]
        j += [p, a]
        v += [np.full(n, -1.0)] * 2
    return n, np.concatenate(i), np.concatenate(j), np.concatenate(v)


@pytest.mark.parametrize("team, make", [
    (True, lambda: uneven(48, 0)), (True, lambda: uneven(48, 60000)), (False, lambda: uneven(48, 300000)),
    (True, lambda: scattered(400000)), (False, lambda: scattered(520000))])
def test_choice(team, make):
    n, i, j, v = make()
    i, j = i.astype(np.int32), j.astype(np.int32)
    A = B.Mat.from_coo(n, n, t(i), t(j))
    A.set_values(t(v))
    assert A.plan()["kernel"] == B.SPMV_SELL
    b = np.random.default_rng(n).standard_normal(n)
    c0 = B.launch_count()
    x, r = A.solve(t(b), rtol=1e-10)
    assert (B.launch_count() - c0 == 2) == team
    O = oracle.coo_symbolic(n, n, i, j)
    oracle.coo_numeric(O, v)
    _, ro = oracle.pcg(O, b, rtol=1e-10)
    assert r["status"] == B.OK
    assert abs(r["iterations"] - ro["iterations"]) <= max(2, 0.01 * ro["iterations"])
    assert np.linalg.norm(b - oracle.spmv(O, x.cpu().numpy())) <= 1.05e-10 * np.linalg.norm(b)
    A.close()
