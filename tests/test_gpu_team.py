"""GPU parity of the one-launch CG on a team of CTAs (the automatic choice for one
system): the edges of its ranges -- less than one slice, one slice, clusters of every
size, the change from cluster to grid, windows or a span too wide for them, a matrix
that stays in shared memory and one that streams -- against the oracle, with the bars
of the phase kernels' tests; statuses; reruns and column patterns bit for bit.
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


def make(n, i, j, v):
    i, j, v = np.asarray(i, np.int32), np.asarray(j, np.int32), np.asarray(v, np.float64)
    A = B.Mat.from_coo(n, n, t(i), t(j))
    A.set_values(t(v))
    O = oracle.coo_symbolic(n, n, i, j)
    oracle.coo_numeric(O, v)
    return A, O


def grid(shape, seed):
    ea, eb = W.grid_edges(shape)
    k = 10.0 ** np.random.default_rng(seed).uniform(-1, 1, ea.shape[0])
    return (int(np.prod(shape)), *W.edge_coo(ea, eb, k))


def coupled(n, step):
    """A tridiagonal matrix whose rows also reach `step` rows away: its span."""
    g = np.arange(n)
    i, j, v = [g], [g], [np.full(n, 4.5)]
    for s in (1, step):
        a = g[:max(0, n - s)]
        i += [a, a + s]
        j += [a + s, a]
        v += [np.full(a.size, -1.0)] * 2
    return n, np.concatenate(i), np.concatenate(j), np.concatenate(v)


CASES = {
    "1 row": lambda: grid((1, 1), 1),
    "31 rows": lambda: grid((31, 1), 2),
    "32 rows": lambda: grid((8, 4), 3),
    "33 rows": lambda: grid((11, 3), 4),
    "3 slices, ragged": lambda: grid((7, 13), 5),
    "15 slices": lambda: grid((24, 20), 6),
    "17 slices": lambda: grid((32, 17), 7),
    "cluster, 3D": lambda: grid((16, 15, 17), 8),
    "cluster, its largest": lambda: grid((110, 111), 9),
    "grid, its smallest": lambda: grid((113, 112), 10),
    "grid, 3D": lambda: grid((40, 41, 39), 11),
    "grid, the matrix streams": lambda: grid((601, 700), 12),
    "cluster, wide span": lambda: coupled(9000, 4500),
    "grid, wide span": lambda: coupled(50001, 25000),
    "grid, span over the 16-bit offsets": lambda: coupled(80000, 40000),
}


@pytest.mark.parametrize("name", list(CASES))
def test_parity(name):
    n, i, j, v = CASES[name]()
    A, O = make(n, i, j, v)
    b = np.random.default_rng(n).standard_normal(n)
    c0 = B.launch_count()
    x, r = A.solve(t(b), rtol=1e-10)
    # the call's arguments and one solver kernel (CSR row products, which the sliced copy's
    # padding leaves to the smallest matrices, run on the phase kernels)
    sliced = A.plan()["kernel"] == B.SPMV_SELL
    assert sliced or n < 64
    assert (B.launch_count() - c0 == 2) == sliced
    xo, ro = oracle.pcg(O, b, rtol=1e-10)
    assert r["status"] == B.OK and ro["status"] == oracle.OK
    assert abs(r["iterations"] - ro["iterations"]) <= max(2, 0.01 * ro["iterations"])
    assert abs(r["rnorm0"] - ro["rnorm0"]) <= 1e-12 * ro["rnorm0"]
    xg = x.cpu().numpy()
    assert np.linalg.norm(b - oracle.spmv(O, xg)) <= 1.05e-10 * np.linalg.norm(b)
    assert np.linalg.norm(xg - xo) <= 1e-6 * np.linalg.norm(xo)
    x2, r2 = A.solve(t(b), rtol=1e-10)
    assert torch.equal(x, x2) and r == r2
    A.set_slice_patterns(False)
    x3, r3 = A.solve(t(b), rtol=1e-10)
    assert torch.equal(x, x3) and r3["iterations"] == r["iterations"]
    A.close()


@pytest.mark.parametrize("shape", [(20, 20), (120, 130)])  # a cluster, the grid
def test_statuses(shape):
    n, i, j, v = grid(shape, 21)
    A, O = make(n, i, j, v)
    b = np.random.default_rng(3).standard_normal(n)
    z = torch.zeros(n, dtype=torch.float64, device=DEV)
    x, r = A.solve(z, x=torch.ones_like(z), nonzero_guess=True)
    assert r["status"] == B.OK and r["iterations"] == 0 and torch.count_nonzero(x) == 0
    x, r = A.solve(t(b), maxit=7)
    xo, ro = oracle.pcg(O, b, maxit=7)
    assert r["status"] == B.ERR_MAXIT and r["iterations"] == 7
    assert np.linalg.norm(x.cpu().numpy() - xo) <= 1e-10 * np.linalg.norm(xo)
    x, r = A.solve(t(b), timeout_ns=1)
    assert r["status"] == B.ERR_TIMEOUT and r["iterations"] == 1 and torch.isfinite(x).all()
    xs, _ = oracle.pcg(O, b, rtol=1e-13)
    x, r = A.solve(t(b), x=t(xs.copy()), rtol=1e-8, nonzero_guess=True)
    assert r["status"] == B.OK and r["iterations"] == 0
    x, r = A.solve(t(b), x=t(0.5 * xs), rtol=1e-10, nonzero_guess=True)
    assert r["status"] == B.OK
    assert np.linalg.norm(b - oracle.spmv(O, x.cpu().numpy())) <= 1.05e-10 * np.linalg.norm(b)
    bad = b.copy()
    bad[n // 2] = np.nan
    assert A.solve(t(bad))[1]["status"] == B.ERR_NAN
    assert A.solve(t(b))[1]["status"] == B.OK
    A.close()
    w = v.copy()
    w[(i == n - 1) & (j == n - 1)] = 0.0
    A, _ = make(n, i, j, w)
    assert A.solve(t(b))[1]["status"] == B.ERR_NOT_SPD
    A.close()
    w = np.where(i == j, v, 40.0 * v)                     # not positive definite
    A, _ = make(n, i, j, w)
    assert A.solve(t(b))[1]["status"] == B.ERR_BREAKDOWN
    A.close()


def test_two_streams_at_once():
    """Two handles' grid teams on two streams: each fills the GPU, so one waits for the other."""
    handles = [make(*grid((150 + k, 140), 31 + k)) for k in range(2)]
    bs = [np.random.default_rng(k).standard_normal(h[0].nrows) for k, h in enumerate(handles)]
    alone = [h[0].solve(t(b), rtol=1e-10)[0] for h, b in zip(handles, bs)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    tb = [t(b) for b in bs]
    xs = [torch.empty_like(b) for b in tb]
    torch.cuda.synchronize()
    for _ in range(4):
        for (A, _), s, b, x in zip(handles, streams, tb, xs):
            A.solve(b, x=x, rtol=1e-10, stream=s, want_result=False)
    torch.cuda.synchronize()
    for x, y in zip(xs, alone):
        assert torch.equal(x, y)
    for A, _ in handles:
        A.close()


def batch_of(shapes, seed):
    rng = np.random.default_rng(seed)
    I, J, V, rows, ncoo = [], [], [], [], []
    for s in shapes:
        n = int(np.prod(s))
        if n:
            ea, eb = W.grid_edges(s)
            i, j, v = W.edge_coo(ea, eb, 10.0 ** rng.uniform(-1, 1, ea.shape[0]))
        else:
            i, j, v = np.zeros(0, np.int32), np.zeros(0, np.int32), np.zeros(0)
        I.append(i), J.append(j), V.append(v), rows.append(n), ncoo.append(i.size)
    b = rng.standard_normal(sum(rows))
    A = B.Mat.from_coo_batched(rows, ncoo, t(np.concatenate(I)), t(np.concatenate(J)))
    A.set_values(t(np.concatenate(V)))
    off = np.concatenate([[0], np.cumsum(rows)])
    gi = np.concatenate([np.where(i >= 0, i + o, -1) for i, o in zip(I, off)]).astype(np.int32)
    gj = np.concatenate([np.where(j >= 0, j + o, -1) for j, o in zip(J, off)]).astype(np.int32)
    O = oracle.coo_symbolic(int(off[-1]), int(off[-1]), gi, gj)
    oracle.coo_numeric(O, np.concatenate(V))
    return A, O, off, b


BATCHES = {
    # clusters of 16 (each other size below), systems of every kind of smallness
    "2 systems": [(40, 40), (9, 10, 11)],
    "9 systems, tiny and empty": [(32, 3), (8, 8), (0, 5), (33, 1), (64, 2), (12, 8), (20, 20),
                                  (6, 6, 6), (31, 31)],
    "12 systems": [(30 + k, 40) for k in range(12)],
    "30 systems": [(20 + k, 23) for k in range(30)],
    "60 systems": [(10 + k, 20) for k in range(60)],
    "160 systems, one large": [(8 + k % 9, 16) for k in range(159)] + [(110, 100)],
    "3 systems, the rows' limit": [(160, 1000), (40, 60, 60), (50, 50)],
}


@pytest.mark.parametrize("name", list(BATCHES))
def test_batches(name):
    A, O, off, b = batch_of(BATCHES[name], len(name))
    c0 = B.launch_count()
    x, rs = A.solve_batched(t(b), rtol=1e-10)
    if A.plan()["kernel"] == B.SPMV_SELL:
        assert B.launch_count() - c0 == 2
    else:
        assert "tiny" in name
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
    A.close()


def test_batch_statuses():
    A, O, off, b = batch_of([(30, 30), (20, 40), (25, 25), (10, 10, 10), (18, 30)], 3)
    b[off[1]:off[2]] = 0.0
    b[off[2] + 5] = np.nan
    x, rs = A.solve_batched(t(b), x=torch.ones(b.size, dtype=torch.float64, device=DEV),
                            rtol=1e-9, nonzero_guess=True)
    assert [r["status"] for r in rs] == [B.OK, B.OK, B.ERR_NAN, B.OK, B.OK]
    assert rs[1]["iterations"] == 0 and torch.count_nonzero(x[off[1]:off[2]]) == 0
    xg = x.cpu().numpy()
    for s in (0, 3, 4):
        sl = slice(off[s], off[s + 1])
        r = b[sl] - oracle.spmv(O, np.where(np.isfinite(xg), xg, 0.0))[sl]
        assert np.linalg.norm(r) <= 1.05e-9 * np.linalg.norm(b[sl])
    b[off[2] + 5] = 1.0
    _, rs = A.solve_batched(t(b), maxit=3)
    assert [r["status"] for r in rs] == [B.ERR_MAXIT, B.OK] + [B.ERR_MAXIT] * 3
    _, rs = A.solve_batched(t(b), timeout_ns=1)
    assert [r["status"] for r in rs] == [B.ERR_TIMEOUT, B.OK] + [B.ERR_TIMEOUT] * 3
    assert all(r["iterations"] <= 1 for r in rs)
    A.close()


FULL = [(60, 60)] * 100 + [(59, 61)] * 54 + [(1023, 1), (1025, 1), (31, 33), (33, 1), (1, 1), (0, 5)]


@pytest.mark.parametrize("precision", ["fp64", "refined"])
@pytest.mark.parametrize("name, shapes, solver", [
    ("full", FULL, "CTA"),              # rows for more than half the SMs of the largest's size
    ("one large", [(10, 10)] * 159 + [(110, 100)], "PHASES"),
])
def test_batch_choice(name, shapes, solver, precision):
    """Automatic choice for batches of one to two systems an SM (the large one of the
    second batch: FP64 takes a cluster, reported as the phase kernels' choice)."""
    A, O, off, b = batch_of(shapes, 7)
    kw = dict(rtol=1e-10, precision=B.FP32_REFINED if precision == "refined" else B.FP64)
    x, rs = A.solve_batched(t(b), **kw)
    resid = b - oracle.spmv(O, x.cpu().numpy())
    for s, r in enumerate(rs):
        sl = slice(off[s], off[s + 1])
        assert r["status"] == B.OK and r["solver"] == getattr(B, "SOLVER_" + solver), (s, r)
        assert np.linalg.norm(resid[sl]) <= 1.05e-10 * np.linalg.norm(b[sl])
    x2, rs2 = A.solve_batched(t(b), **kw)
    assert torch.equal(x, x2) and rs == rs2
    A.set_solver(B.SOLVER_PHASES)
    _, rs = A.solve_batched(t(b), **kw)
    assert all(r["status"] == B.OK and r["solver"] == B.SOLVER_PHASES for r in rs)
    A.close()


@pytest.mark.parametrize("n, solver", [(64, "CTA"), (86, "CTA"), (110, "PHASES")])
def test_refined_choice(n, solver):
    g = grid((n, n), n)
    A, O = make(*g)
    b = np.random.default_rng(n).standard_normal(n * n)
    x, r = A.solve(t(b), rtol=1e-10, precision=B.FP32_REFINED)
    assert r["status"] == B.OK and r["solver"] == getattr(B, "SOLVER_" + solver)
    assert np.linalg.norm(b - oracle.spmv(O, x.cpu().numpy())) <= 1.05e-10 * np.linalg.norm(b)
    A.close()


@pytest.mark.parametrize("method", ["BICG", "TFQMR"])
def test_nonsymmetric_batch_sizes(method):
    """Per-CTA BiCG and TFQMR on systems around the size (96 slices) from which BiCG's
    products keep more pairs in flight, and on far smaller ones; the bar of the
    nonsymmetric solvers' tests (twice rtol)."""
    A, O, off, b = batch_of([(37, 83), (48, 64), (7, 439), (32, 97), (64, 70), (5, 8), (1, 1)], 5)
    A.set_solver(B.SOLVER_CTA)
    kw = dict(rtol=1e-9, method=getattr(B, "KSP_" + method))
    x, rs = A.solve_batched(t(b), **kw)
    resid = b - oracle.spmv(O, x.cpu().numpy())
    for s, r in enumerate(rs):
        sl = slice(off[s], off[s + 1])
        assert r["status"] == B.OK and r["solver"] == B.SOLVER_CTA, (s, r)
        assert np.linalg.norm(resid[sl]) <= 2e-9 * np.linalg.norm(b[sl]), s
    x2, rs2 = A.solve_batched(t(b), **kw)
    assert torch.equal(x, x2) and rs == rs2
    A.close()
