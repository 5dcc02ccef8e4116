"""Performance cases of the library: what its users have it do, from the smallest calls to the largest.

A case names a kind of call, a matrix (the mesh it comes from and its size) and the options the call takes:

  mult      y = A x on an assembled matrix (``Mat.mult``)
  values    new COO values into an existing pattern (``Mat.set_values``): the per-step half of assembly
  assemble  pattern and values from COO triples (``Mat.from_coo`` and ``Mat.set_values``)
  solve     one system from x0 = 0 (``Mat.solve``): FP64 CG or the FP32-refined solve
  gradient  a solve and its backward pass (``autograd.solve``), as one step of a training loop takes them
  batch     many independent systems in one call (``Mat.solve_batched``): CG, refined, TFQMR or BiCG

The meshes are the ones the repository's workloads and benchmark use -- Poisson stencils, Q1 hexahedral
elements, edge diffusion, upwind convection-diffusion -- and an unstructured graph with ragged rows, whose
matrix has no stencil pattern.  Symmetric solves run to a relative residual of 1e-12, as the repository's
gradient checks do, nonsymmetric ones to 1e-11.  All inputs are drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import torch

from paper_2406_08646_gb300 import autograd as AG
from paper_2406_08646_gb300 import binding as B

DEV = "cuda"
METHODS = {"cg": B.KSP_CG, "bicg": B.KSP_BICG, "tfqmr": B.KSP_TFQMR}


def listed():
    return [
        # one product on a system of a few thousand rows: launch and call overhead
        {"name": "mult_poisson2d_64", "kind": "mult", "mesh": "poisson2d", "size": 64},
        # the finite-element matrix of the benchmark: 27-point rows, 24 million nonzeros
        {"name": "mult_q1hex_96", "kind": "mult", "mesh": "q1hex", "size": 96},
        # an unstructured mesh: 4 to 40 entries a row, no common column pattern
        {"name": "mult_graph_300k", "kind": "mult", "mesh": "graph", "size": 300007},
        # refilling the finite-element matrix: every Newton or time step does this
        {"name": "values_q1hex_96", "kind": "values", "mesh": "q1hex", "size": 96},
        # a new 2D diffusion matrix from its edges: pattern and values
        {"name": "assemble_edge2d_1024", "kind": "assemble", "mesh": "edge2d", "size": 1024},
        # a new finite-element matrix: 57 million COO entries with duplicates
        {"name": "assemble_q1hex_96", "kind": "assemble", "mesh": "q1hex", "size": 96},
        # a small solve: a few thousand rows, a couple of hundred iterations
        {"name": "solve_poisson2d_64", "kind": "solve", "mesh": "poisson2d", "size": 64, "precision": "fp64", "rtol": 1e-12},
        # the finite-element system of the benchmark
        {"name": "solve_q1hex_96", "kind": "solve", "mesh": "q1hex", "size": 96, "precision": "fp64", "rtol": 1e-12},
        # the mixed-precision solve of a 7-million-row stencil: vectors larger than the cache
        {"name": "refined_poisson3d_192", "kind": "solve", "mesh": "poisson3d", "size": 192, "precision": "refined", "rtol": 1e-12},
        # one training step through a 2D diffusion solve: forward, adjoint, gradients of values and right-hand side
        {"name": "gradient_edge2d_1024", "kind": "gradient", "mesh": "edge2d", "size": 1024, "rtol": 1e-12},
        # hundreds of uneven symmetric systems at once
        {"name": "batch_cg_512", "kind": "batch", "mesh": "edge", "nsys": 512, "lo": 1000, "hi": 20000, "method": "cg", "precision": "fp64", "rtol": 1e-12},
        # nonsymmetric systems of a time integrator, the batched Krylov method of the paper
        {"name": "batch_tfqmr_256", "kind": "batch", "mesh": "convdiff", "nsys": 256, "lo": 1000, "hi": 20000, "method": "tfqmr", "precision": "fp64", "rtol": 1e-11},
    ]


def draw(rng):
    kind = rng.choice(["mult", "values", "assemble", "solve", "solve", "gradient", "batch"])
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    if kind == "batch":
        nonsym = rng.random() < 0.4
        lo = log(500, 4000)
        c = {"kind": kind, "mesh": "convdiff" if nonsym else "edge", "nsys": log(4, 400), "lo": lo, "hi": log(lo + 100, 20000),
             "method": rng.choice(["tfqmr", "bicg"]) if nonsym else "cg", "precision": "fp64", "rtol": 1e-11 if nonsym else 1e-12}
        if not nonsym and rng.random() < 0.3:
            c["precision"] = "refined"
        return c
    if kind == "gradient":
        mesh, size = rng.choice([("edge2d", log(24, 800)), ("edge3d", log(8, 96))])
        return {"kind": kind, "mesh": mesh, "size": size, "rtol": 1e-12}
    if kind == "solve":
        mesh, size = rng.choice([("poisson2d", log(24, 800)), ("poisson3d", log(8, 160)), ("q1hex", log(6, 90)),
                                 ("edge2d", log(24, 800)), ("edge3d", log(8, 128)), ("graph", log(700, 300000))])
        refined = rng.random() < 0.3
        return {"kind": kind, "mesh": mesh, "size": size, "precision": "refined" if refined else "fp64", "rtol": 1e-12}
    meshes = [("q1hex", log(6, 90)), ("edge2d", log(24, 1000)), ("edge3d", log(8, 110)), ("graph", log(700, 1000000))]
    if kind == "mult":
        meshes += [("poisson2d", log(24, 1500)), ("poisson3d", log(8, 160))]
    mesh, size = rng.choice(meshes)
    return {"kind": kind, "mesh": mesh, "size": size}


# ------------------------------------------------------------------ the matrices, as COO triples


def _log_uniform(n, gen):
    return 10.0 ** (2.0 * torch.rand(n, dtype=torch.float64, device=DEV, generator=gen) - 1.0)


def _coords(shape):
    g = torch.arange(math.prod(shape), dtype=torch.int64, device=DEV)
    out, rem = [], g
    for s in shape:
        out.append(rem % s)
        rem = rem // s
    return g, out


def _stencil(shape):
    """Rows of the (2d+1)-point Laplacian, a neighbour outside the grid written as column -1."""
    g, xs = _coords(shape)
    cols, stride = [g], 1
    for x, s in zip(xs, shape):
        for d in (-1, 1):
            cols.append(torch.where((x + d >= 0) & (x + d < s), g + d * stride, -1))
        stride *= s
    j = torch.stack(cols, 1).to(torch.int32)
    i = g.to(torch.int32)[:, None].expand_as(j)
    return i.reshape(-1).contiguous(), j.reshape(-1)


def _poisson(shape):
    i, j = _stencil(shape)
    k, h2 = 2 * len(shape) + 1, float(shape[0] + 1) ** 2
    v = torch.full((j.numel() // k, k), -h2, dtype=torch.float64, device=DEV)
    v[:, 0] = 2 * len(shape) * h2
    return math.prod(shape), i, j, v.reshape(-1)


def _convdiff(side, angle, speed):
    """First-order upwind convection-diffusion on a square grid: nonsymmetric."""
    n, i, j, v = _poisson((side, side))
    v, h = v.view(-1, 5), 1.0 / (side + 1)
    bx, by = speed * math.cos(angle), speed * math.sin(angle)
    v[:, 0] += (abs(bx) + abs(by)) / h
    v[:, 1 if bx > 0 else 2] -= abs(bx) / h
    v[:, 3 if by > 0 else 4] -= abs(by) / h
    return n, i, j, v.reshape(-1)


def _edges(shape, gen):
    """Variable-coefficient diffusion: four entries an edge, an entry at a ghost node ignored."""
    ea, eb = [], []
    for d in range(len(shape)):
        longer = list(shape)
        longer[d] += 1
        _, xs = _coords(longer)
        lo, hi, stride = torch.zeros_like(xs[0]), torch.zeros_like(xs[0]), 1
        for q, s in enumerate(shape):
            lo, hi, stride = lo + (xs[q] - int(q == d)) * stride, hi + xs[q] * stride, stride * s
        ea.append(torch.where(xs[d] >= 1, lo, -1))
        eb.append(torch.where(xs[d] < shape[d], hi, -1))
    ea, eb = torch.cat(ea).to(torch.int32), torch.cat(eb).to(torch.int32)
    ghost = (ea < 0) | (eb < 0)
    i, j = torch.stack([ea, eb, ea, eb], 1), torch.stack([ea, eb, eb, ea], 1)
    i[:, 2:][ghost] = -1
    j[:, 2:][ghost] = -1
    k = _log_uniform(ea.numel(), gen)
    return math.prod(shape), i.reshape(-1), j.reshape(-1), torch.stack([k, k, -k, -k], 1).reshape(-1)


def _q1hex(ne, gen):
    """Q1 hexahedra on the unit cube, 8 x 8 blocks in element order; boundary rows are identity rows."""
    nn = ne + 1
    _, (ex, ey, ez) = _coords((ne, ne, ne))
    corner = torch.arange(8, device=DEV)
    bits = [corner & 1, (corner >> 1) & 1, corner >> 2]
    xs = [e[:, None] + b[None, :] for e, b in zip((ex, ey, ez), bits)]
    node = (xs[0] + nn * (xs[1] + nn * xs[2])).to(torch.int32)
    on = [(x == 0) | (x == ne) for x in xs]
    bnd = on[0] | on[1] | on[2]
    share = torch.ones(node.shape, dtype=torch.float64, device=DEV)
    for f in on:
        share = torch.where(f, share, share * 0.5)
    del xs, on
    differ = corner[:, None] ^ corner[None, :]
    ones = (differ & 1) + ((differ >> 1) & 1) + (differ >> 2)
    K = torch.tensor([1 / 3, 0.0, -1 / 12, -1 / 12], dtype=torch.float64, device=DEV)[ones]
    v = (_log_uniform(ne ** 3, gen) / ne)[:, None, None] * K
    v.masked_fill_(bnd[:, :, None] | bnd[:, None, :], 0.0)
    v.diagonal(dim1=1, dim2=2).add_(torch.where(bnd, share, 0.0))
    i = node[:, :, None].expand(-1, 8, 8).reshape(-1)
    j = node[:, None, :].expand(-1, 8, 8).reshape(-1)
    return nn ** 3, i, j, v.reshape(-1)


def _graph(n, gen):
    """A weighted graph Laplacian plus a mass term: each node draws 1 to 20 neighbours near it in the numbering, so rows hold
    about 4 to 40 entries in no common pattern; both directions of an edge and both diagonal shares are written, duplicates too.
    The graph is the size's own, the weights are drawn."""
    own_gen = torch.Generator(device=DEV)
    own_gen.manual_seed(n)
    deg = (2.0 * _log_uniform(n, own_gen).sqrt() * math.sqrt(10.0)).long().clamp_(1, 20)
    a = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    reach = (torch.randn(a.numel(), dtype=torch.float64, device=DEV, generator=own_gen) * min(2000.0, n / 8)).round().long()
    b = (a + torch.where(reach == 0, 1, reach)) % n
    k = _log_uniform(a.numel(), gen)
    own, mass = torch.arange(n, device=DEV), torch.full((n,), 0.05, dtype=torch.float64, device=DEV)
    i = torch.cat([torch.stack([a, b, a, b], 1).reshape(-1), own]).to(torch.int32)
    j = torch.cat([torch.stack([a, b, b, a], 1).reshape(-1), own]).to(torch.int32)
    return n, i, j, torch.cat([torch.stack([k, k, -k, -k], 1).reshape(-1), mass])


def _one(case, gen):
    m, s = case["mesh"], case["size"]
    if m == "poisson2d":
        return _poisson((s, s))
    if m == "poisson3d":
        return _poisson((s, s, s))
    if m == "edge2d":
        return _edges((s, s), gen)
    if m == "edge3d":
        return _edges((s, s, s), gen)
    if m == "q1hex":
        return _q1hex(s, gen)
    return _graph(s, gen)


def _sides(case):
    """The systems of a batch: row counts spread evenly over the range, in a scattered order; every second edge system is 3D."""
    n, out = case["nsys"], []
    for q in range(n):
        rows = case["lo"] + (case["hi"] - case["lo"]) * (((q * 0.6180339887498949) % 1.0))
        dims = 3 if case["mesh"] == "edge" and q % 2 else 2
        out.append((dims, max(2, round(rows ** (1.0 / dims)))))
    return out


def _batch(case, gen):
    parts = []
    for q, (dims, side) in enumerate(_sides(case)):
        if case["mesh"] == "edge":
            parts.append(_edges((side,) * dims, gen))
        else:
            parts.append(_convdiff(side, 2.4 * q, 10.0 ** (2.0 * ((q * 0.7548776662466927) % 1.0))))
    rows, ncoo = [p[0] for p in parts], [p[1].numel() for p in parts]
    return rows, ncoo, torch.cat([p[1] for p in parts]), torch.cat([p[2] for p in parts]), torch.cat([p[3] for p in parts])


def _problem(case, seed):
    """(row counts, COO counts, i, j, v, vectors): one system's counts are lists of one."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    if case["kind"] == "batch":
        rows, ncoo, i, j, v = _batch(case, gen)
    else:
        n, i, j, v = _one(case, gen)
        rows, ncoo = [n], [i.numel()]
    vec = [torch.randn(sum(rows), dtype=torch.float64, device=DEV, generator=gen) for _ in range(2)]
    return rows, ncoo, i, j, v, vec


# ------------------------------------------------------------------ a pass


def prepare(case, seed):
    rows, ncoo, i, j, v, (b, target) = _problem(case, seed)
    s = {"case": case, "n": sum(rows), "v": v, "b": b}
    if case["kind"] == "assemble":
        return dict(s, i=i, j=j, A=None)
    if case["kind"] == "batch":
        A = B.Mat.from_coo_batched(rows, ncoo, i, j)
    else:
        A = B.Mat.from_coo(s["n"], s["n"], i, j)
    if case["kind"] == "gradient":
        return dict(s, A=A, v=v.requires_grad_(True), b=b.requires_grad_(True), target=target)
    A.set_values(v)
    if case["kind"] == "values":
        s["val"] = A.csr()[2]
        s["val"].owner = A  # a view of the handle's memory
    return dict(s, A=A)


def run(s):
    case, A = s["case"], s["A"]
    kind = case["kind"]
    if kind == "mult":
        return A.mult(s["b"])
    if kind == "values":
        A.set_values(s["v"])
        return s["val"]
    if kind == "assemble":
        if A is not None:
            A.close()
        s["A"] = A = B.Mat.from_coo(s["n"], s["n"], s["i"], s["j"])
        A.set_values(s["v"])
        csr = A.csr()
        for t in csr:
            t.owner = A  # a view of the handle's memory
        return csr
    if kind == "gradient":
        x = AG.solve(s["v"], s["b"], A, rtol=case["rtol"])
        loss = 0.5 * (x - s["target"]).square().sum()
        gv, gb = torch.autograd.grad(loss, (s["v"], s["b"]))
        return {"x": x, "dv": gv, "db": gb}
    opts = {"rtol": case["rtol"], "precision": B.FP32_REFINED if case["precision"] == "refined" else B.FP64}
    if kind == "solve":
        return A.solve(s["b"], **opts)[0]
    return A.solve_batched(s["b"], method=METHODS[case["method"]], **opts)[0]


# ------------------------------------------------------------------ the work a pass cannot do without


def _counts(case):
    """(rows, nonzeros, COO entries, iterations a CG of this accuracy takes: about 2.5 per grid line of the longest side)."""
    def of(mesh, s):
        if mesh in ("poisson2d", "edge2d", "convdiff"):
            n, z = s * s, 5 * s * s - 4 * s
            return n, z, (8 * s * (s + 1) if mesh == "edge2d" else 5 * n), 2.5 * s
        if mesh in ("poisson3d", "edge3d"):
            n, z = s ** 3, 7 * s ** 3 - 6 * s * s
            return n, z, (12 * s * s * (s + 1) if mesh == "edge3d" else 7 * n), 2.5 * s
        if mesh == "q1hex":
            return (s + 1) ** 3, (3 * s + 1) ** 3, 64 * s ** 3, 2.5 * s
        return s, 19 * s, 37 * s, 60.0
    if case["kind"] != "batch":
        return of(case["mesh"], case["size"])
    each = [of("convdiff" if case["mesh"] == "convdiff" else "edge%dd" % d, s) for d, s in _sides(case)]
    return sum(e[0] for e in each), sum(e[1] for e in each), sum(e[2] for e in each), sum(e[1] * e[3] for e in each) / max(1, sum(e[1] for e in each))


def work(case):
    n, z, k, its = _counts(case)
    kind = case["kind"]
    if kind == "mult":
        return {"bytes": 12 * z + 4 * n + 16 * n, "flops": 2 * z}
    if kind == "values":
        return {"bytes": 8 * k + 8 * z, "flops": max(0, k - z)}
    if kind == "assemble":
        return {"bytes": 16 * k + 12 * z + 4 * n, "flops": max(0, k - z)}
    iteration = 2 * z + 13 * n  # one product, two inner products, three vector updates, the diagonal
    if kind == "gradient":
        return {"bytes": 8 * k * 2 + 12 * z + 5 * 8 * n, "flops": 2 * its * iteration}
    return {"bytes": 12 * z + 4 * n + 16 * n, "flops": its * iteration * (2 if case.get("method") in ("tfqmr", "bicg") else 1)}


# ------------------------------------------------------------------ the same in plain torch, 64 bits


def _assembled(case, seed):
    rows, ncoo, i, j, v, vec = _problem(case, seed)
    n = sum(rows)
    if len(rows) > 1:
        first = torch.tensor([0] + rows[:-1], device=DEV).cumsum(0)
        shift = torch.repeat_interleave(first, torch.tensor(ncoo, device=DEV))
        i, j = torch.where(i >= 0, i + shift, -1), torch.where(j >= 0, j + shift, -1)
    kept = (i >= 0) & (j >= 0)
    key, back = torch.unique(i[kept].long() * n + j[kept].long(), return_inverse=True)
    val = torch.zeros(key.numel(), dtype=torch.float64, device=DEV).index_add_(0, back, v[kept])
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    col = key % n
    diag = torch.zeros(n, dtype=torch.float64, device=DEV)
    on = key // n == col
    diag[col[on]] = val[on]
    return torch.sparse_csr_tensor(ptr, col, val, size=(n, n)), diag, (i, j, kept), vec


def _cg(A, diag, b, rtol):
    x, r = torch.zeros_like(b), b.clone()
    z = r / diag
    p, rho, stop = z.clone(), r @ z, rtol * b.norm()
    for k in range(40000):
        q = A @ p
        alpha = rho / (p @ q)
        x.add_(alpha * p)
        r.sub_(alpha * q)
        if k % 16 == 15 and not r.norm() > stop:
            break
        z = r / diag
        new = r @ z
        p = z + (new / rho) * p
        rho = new
    return x


def _bicgstab(A, diag, b, rtol):
    x, r = torch.zeros_like(b), b.clone()
    rt, p, v = r.clone(), torch.zeros_like(b), torch.zeros_like(b)
    rho = alpha = omega = torch.ones((), dtype=torch.float64, device=DEV)
    stop = rtol * b.norm()
    for k in range(20000):
        new = rt @ r
        p = r + (new / rho) * (alpha / omega) * (p - omega * v)
        rho, y = new, p / diag
        v = A @ y
        alpha = rho / (rt @ v)
        s = r - alpha * v
        z = s / diag
        t = A @ z
        omega = (t @ s) / (t @ t)
        x.add_(alpha * y + omega * z)
        r = s - omega * t
        if k % 8 == 7 and not r.norm() > stop:
            break
    return x


def _solved(A, diag, b, symmetric=True):
    x = torch.zeros_like(b)
    for _ in range(3):
        x = x + (_cg if symmetric else _bicgstab)(A, diag, b - A @ x, 1e-9)
    return x


def exact(case, seed):
    A, diag, (i, j, kept), (b, target) = _assembled(case, seed)
    kind = case["kind"]
    if kind == "mult":
        return A @ b
    if kind == "values":
        return A.values()
    if kind == "assemble":
        return None, None, A.values()
    if kind == "gradient":
        x = _solved(A, diag, b)
        lam = _solved(A, diag, x - target)
        gv = torch.zeros(i.numel(), dtype=torch.float64, device=DEV)
        gv[kept] = -lam[i[kept].long()] * x[j[kept].long()]
        return {"x": x, "dv": gv, "db": lam}
    return _solved(A, diag, b, symmetric=case["mesh"] != "convdiff")
