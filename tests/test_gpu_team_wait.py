"""GPU: a grid team whose partner never comes.  csrc/team.cu's kernel for batches on a shared grid
is launched with one CTA fewer than the last system's team counts on (nothing else waits for
it), and with short limits: its waits run out, the kernel returns, that system is reported as
GBS_ERR_TIMEOUT and the other one, on a team that is complete, is solved; the handle solves
again.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2406_08646_gb300 import _build
from paper_2406_08646_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2406_08646_gb300 import binding as B  # noqa: E402

DEV = "cuda"
SOURCE = r"""
#include "team.cu"
using namespace gbs;

static int launch(gbs_mat A, const double *b, double *x, unsigned polls, long long ns) {
  cudaStream_t s = nullptr;
  ksp_opts o;
  ksp_opts_default(&o);
  o.maxit = 1000;
  o.rtol = 1e-10;
  GBS_TRY(ensure_solver_workspace(A, false, s));
  PcgArgs a = make_args(A, true, false);
  a.order = A->cta_order;
  a.cta_n = A->nsys;
  A->last_count = A->nsys;
  A->last_solver = GBS_SOLVER_PHASES;
  A->trips_counted = true;
  TeamParts parts = {};
  parts.first[1] = 1;   // the first system on CTA 0; the second counts on CTAs 1 and 2
  parts.first[2] = 3;
  unsigned *ctr = reinterpret_cast<unsigned *>(A->part + 4 * sm_count(A));
  GBS_TRY_CUDA(cudaMemsetAsync(ctr, 0, sizeof(unsigned) * TEAM_CTR_STRIDE * 2, s));
  GBS_TRY_CUDA(cudaMemsetAsync(A->ctl, 0, sizeof(DevCtl), s));
  GBS_TRY(put_call(A->call, call_args(b, x, o), s, A->ctl));
  GBS_TRY_CUDA(cudaFuncSetAttribute(k_team_parts<512>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)TEAM_SMEM));
  k_team_parts<512><<<2, 512, TEAM_SMEM, s>>>(a, parts, A->col_span, (int32_t)TEAM_SMEM, 0, ctr,
                                              A->part, polls, ns);
  GBS_TRY_CUDA(cudaGetLastError());
  return GBS_OK;
}

extern "C" int solve_with_a_missing_cta(gbs_mat A, const double *b, double *x, unsigned polls,
                                        long long ns, ksp_result *res) {
  const int st = launch(A, b, x, polls, ns);
  if (st != GBS_OK) return -st;
  return read_results(A, res, 2, nullptr);
}
"""


@pytest.fixture(scope="module")
def native(tmp_path_factory):
    d = tmp_path_factory.mktemp("team")
    (d / "wait.cu").write_text(SOURCE)
    B.lib()
    subprocess.run([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-Xlinker", "-Bsymbolic", "-I", _build.INCLUDE,
                    "-I", _build.CSRC, "-shared", "-o", str(d / "wait.so"), str(d / "wait.cu"),
                    _build.LIB, "-Xlinker", f"-rpath={os.path.dirname(_build.LIB)}"], check=True)
    f = ctypes.CDLL(str(d / "wait.so")).solve_with_a_missing_cta
    P = ctypes.c_void_p
    f.argtypes, f.restype = [P, P, P, ctypes.c_uint, ctypes.c_longlong, P], ctypes.c_int
    return f


def t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def test_wait_runs_out(native):
    rng = np.random.default_rng(5)
    parts, rows = [], [1200, 600]                       # (the larger one comes first)
    for shape in ((40, 30), (20, 30)):
        ea, eb = W.grid_edges(shape)
        parts.append(W.edge_coo(ea, eb, 10.0 ** rng.uniform(-1, 1, ea.shape[0])))
    i, j, v = (np.concatenate([p[k] for p in parts]) for k in range(3))
    A = B.Mat.from_coo_batched(rows, [p[0].size for p in parts], t(i), t(j))
    A.set_values(t(v))
    b = t(rng.standard_normal(1800))
    x = torch.zeros_like(b)
    torch.cuda.synchronize()
    for polls, ns in ((1023, 1000000), (1 << 14, 1000)):
        res = (B.KspResult * 2)()
        st = native(A.h, b.data_ptr(), x.data_ptr(), polls, ns, ctypes.cast(res, ctypes.c_void_p))
        assert st == B.ERR_TIMEOUT
        assert [r.status for r in res] == [B.OK, B.ERR_TIMEOUT]
    O = oracle.coo_symbolic(1200, 1200, *parts[0][:2])
    oracle.coo_numeric(O, parts[0][2])
    bh = b.cpu().numpy()

    def residual(x):
        return np.linalg.norm(bh[:1200] - oracle.spmv(O, x.cpu().numpy()[:1200]))
    assert residual(x) <= 1.05e-10 * np.linalg.norm(bh[:1200])
    x, rs = A.solve_batched(b, rtol=1e-10)
    assert [r["status"] for r in rs] == [B.OK, B.OK]
    assert residual(x) <= 1.05e-10 * np.linalg.norm(bh[:1200])
    A.close()
