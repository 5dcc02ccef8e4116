"""GPU: batches of a few large systems on one shared grid of CTAs -- equal and unlike systems,
parts that keep their matrix and parts that stream it, more CTAs than a system has slices,
empty systems, column indices -- against the oracle with the bars of the batches' tests; the
statuses of every system on its own; reruns bit for bit.
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


def batch_of(shapes, seed):
    rng = np.random.default_rng(seed)
    I, J, V, rows, ncoo = [], [], [], [], []
    for s in shapes:
        n = int(np.prod(s))
        i, j, v = np.zeros(0, np.int32), np.zeros(0, np.int32), np.zeros(0)
        if n:
            ea, eb = W.grid_edges(s)
            i, j, v = W.edge_coo(ea, eb, 10.0 ** rng.uniform(-1, 1, ea.shape[0]))
        I.append(i), J.append(j), V.append(v), rows.append(n), ncoo.append(i.size)
    b = rng.standard_normal(sum(rows))
    A = B.Mat.from_coo_batched(rows, ncoo, t(np.concatenate(I)), t(np.concatenate(J)))
    v = np.concatenate(V)
    A.set_values(t(v))
    off = np.concatenate([[0], np.cumsum(rows)])
    gi = np.concatenate([np.where(i >= 0, i + o, -1) for i, o in zip(I, off)]).astype(np.int32)
    gj = np.concatenate([np.where(j >= 0, j + o, -1) for j, o in zip(J, off)]).astype(np.int32)
    O = oracle.coo_symbolic(int(off[-1]), int(off[-1]), gi, gj)
    oracle.coo_numeric(O, v)
    return A, O, off, b, v, gi, gj


BATCHES = {
    "2 equal": [(200, 150)] * 2,
    "9 equal": [(150, 160)] * 9,
    "64 equal": [(80, 75)] * 64,
    "streaming": [(430, 420)] * 2,
    "3D": [(40, 41, 42), (42, 41, 40), (41, 40, 42)],
    "unlike, tiny and empty": [(400, 300), (7, 5), (0, 5), (300, 310), (33, 1), (50, 60, 30)],
    "flat, wide span": [(4000, 30), (30, 4000)],
}


@pytest.mark.parametrize("name", list(BATCHES))
def test_parity(name):
    A, O, off, b, *_ = batch_of(BATCHES[name], len(name))
    assert A.plan()["kernel"] == B.SPMV_SELL
    c0 = B.launch_count()
    x, rs = A.solve_batched(t(b), rtol=1e-10)
    assert B.launch_count() - c0 == 2
    xo, ros = oracle.pcg_batched(O, off, b, rtol=1e-10)
    xg = x.cpu().numpy()
    resid = b - oracle.spmv(O, xg)
    for s, (r, ro) in enumerate(zip(rs, ros)):
        sl = slice(off[s], off[s + 1])
        assert r["status"] == B.OK and abs(r["iterations"] - ro["iterations"]) <= max(
            2, 0.01 * ro["iterations"]), (s, r, ro)
        assert np.linalg.norm(resid[sl]) <= 1.05e-10 * np.linalg.norm(b[sl])
        assert np.linalg.norm(xg[sl] - xo[sl]) <= 1e-6 * np.linalg.norm(xo[sl])
    x2, rs2 = A.solve_batched(t(b), rtol=1e-10)
    assert torch.equal(x, x2) and rs == rs2
    A.set_slice_patterns(False)
    x3, _ = A.solve_batched(t(b), rtol=1e-10)
    assert torch.equal(x, x3)
    x4, r4 = A.solve_batched(t(b), x=t(xg), rtol=1e-9, nonzero_guess=True)
    assert all(r["status"] == B.OK and r["iterations"] == 0 for r in r4) and torch.equal(x4, x)
    A.close()


def test_statuses():
    A, O, off, b, v, gi, gj = batch_of([(150, 150), (140, 160), (150, 149), (90, 250)], 3)
    b[off[1]:off[2]] = 0.0
    b[off[2] + 5] = np.nan
    x, rs = A.solve_batched(t(b), x=torch.ones(b.size, dtype=torch.float64, device=DEV),
                            rtol=1e-9, nonzero_guess=True)
    assert [r["status"] for r in rs] == [B.OK, B.OK, B.ERR_NAN, B.OK]
    assert rs[1]["iterations"] == 0 and torch.count_nonzero(x[off[1]:off[2]]) == 0
    b[off[2] + 5] = 1.0
    _, rs = A.solve_batched(t(b), maxit=3)
    assert [r["status"] for r in rs] == [B.ERR_MAXIT, B.OK, B.ERR_MAXIT, B.ERR_MAXIT]
    _, rs = A.solve_batched(t(b), timeout_ns=1)
    assert [r["status"] for r in rs] == [B.ERR_TIMEOUT, B.OK, B.ERR_TIMEOUT, B.ERR_TIMEOUT]
    assert all(r["iterations"] <= 1 for r in rs)
    w = v.copy()
    w[(gi == off[1] - 1) & (gj == off[1] - 1)] = 0.0          # a missing diagonal in system 0
    own = (gi >= off[3]) & (gi != gj)
    w[own] *= 40.0                                             # system 3: not positive definite
    A.set_values(t(w))
    _, rs = A.solve_batched(t(b), rtol=1e-9)
    assert [r["status"] for r in rs] == [B.ERR_NOT_SPD, B.OK, B.OK, B.ERR_BREAKDOWN]
    A.set_values(t(v))
    _, rs = A.solve_batched(t(b), rtol=1e-9)
    assert [r["status"] for r in rs] == [B.OK] * 4
    A.close()
