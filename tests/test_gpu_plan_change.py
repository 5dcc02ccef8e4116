"""GPU solves after the plan moves a handle to another row-product kernel: what the new plan
reads is made when it is first needed, with the bits of a handle that had the plan from the start.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_08646_gb300 import binding as B  # noqa: E402

DEV = "cuda"


def ragged(n, seed):
    """A graph Laplacian plus a mass term with rows of 1 to 82 entries: CSR row products."""
    rng = np.random.default_rng(seed)
    deg = rng.integers(0, 9, n) ** 2 // 2
    a = np.repeat(np.arange(n), deg)
    b = (a + 1 + rng.integers(0, n - 1, a.size)) % n
    k, own = rng.uniform(0.1, 1.0, a.size), np.arange(n)
    i = np.concatenate([a, b, a, b, own]).astype(np.int32)
    j = np.concatenate([a, b, b, a, own]).astype(np.int32)
    return [torch.from_numpy(x).to(DEV)
            for x in (i, j, np.concatenate([k, k, -k, -k, np.full(n, 0.3)]))]


@pytest.mark.parametrize("first, second", [(B.SPMV_AUTO, B.SPMV_SELL), (4, B.SPMV_SELL),
                                           (B.SPMV_SELL, 4), (4, 32), (32, 8)])
def test_refined_after_plan_change(first, second):
    n = 3001
    i, j, v = ragged(n, 7)
    b = torch.from_numpy(np.random.default_rng(1).standard_normal(n)).to(DEV)
    got = []
    for plans in ((first, second), (second,)):
        A = B.Mat.from_coo(n, n, i, j)
        A.set_values(v)
        assert A.plan()["kernel"] != B.SPMV_SELL
        for kernel in plans:
            A.set_plan(kernel=kernel)
            x, r = A.solve(b, rtol=1e-10, precision=B.FP32_REFINED)
            assert r["status"] == B.OK and r["true_rel_residual"] <= 1.05e-10
        got.append((x, r))
        A.close()
    assert torch.equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
