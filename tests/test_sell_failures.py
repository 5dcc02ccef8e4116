"""Building the sliced copy when a step fails, without a GPU: csrc/sell.cu's host code against
a stand-in CUDA runtime (kernels that do nothing, host memory) in which the k-th allocation, or
the k-th launch or copy, fails.  The call reports it and leaves no half-built copy behind: the next
call on the handle builds what a fresh handle gets, and no memory is lost.
"""
import ctypes
import os
import subprocess

import pytest

from paper_2406_08646_gb300 import _build

SOURCE = r"""
#include <cstdlib>
#include <cstring>
#include <set>

#include "internal.cuh"

static std::set<void *> live;
static int calls, fail_at;          // steps so far; the one that fails (-1: none)
static int launches;
static bool fails() { return calls++ == fail_at; }

extern "C" {
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *,
                            dim3 *, dim3 *, int *) {}
char __cudaInitModule(void **) { return 0; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *) { *k = nullptr; return cudaSuccess; }
static cudaError_t last;
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) {
  ++launches;
  last = fails() ? cudaErrorLaunchFailure : cudaSuccess;
  return last;
}
cudaError_t cudaGetLastError() { return last; }
const char *cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
  if (fails()) return cudaErrorUnknown;
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (fails()) return cudaErrorUnknown;
  memcpy(d, s, n);
  return cudaSuccess;
}
}  // extern "C"

namespace gbs {
void set_error(const char *, ...) {}
void count_launches(int64_t) {}
void drop_graphs(gbs_mat) {}
int sm_count(gbs_mat) { return 152; }
int dev_alloc_bytes(void **p, size_t n, cudaStream_t) {
  *p = nullptr;
  if (fails()) return GBS_ERR_ALLOC;
  *p = calloc(n + 16, 1);
  live.insert(*p);
  return GBS_OK;
}
void dev_free(void *p, cudaStream_t) {
  if (p && !live.erase(p)) abort();
  free(p);
}
int64_t scan_tmp_words(int64_t) { return 1; }
int exclusive_scan(const uint32_t *, uint32_t *, int64_t, uint32_t *, uint32_t *, cudaStream_t) {
  return fails() ? GBS_ERR_CUDA : GBS_OK;
}
}  // namespace gbs

// Status of a build whose step `fail` fails; what the build after it made goes to out: its
// launches, its allocations alive, which arrays it has.  fail < 0: the first build alone.
extern "C" int build(int nsys, int rows, int patterns, int fail, int *out) {
  gbs_mat_s A;
  A.nsys = nsys;
  A.row_off_h.clear();
  for (int q = 0; q <= nsys; ++q) A.row_off_h.push_back((int64_t)q * rows);
  A.nrows = A.ncols = (int64_t)nsys * rows;
  A.sell_patterns = patterns;
  A.values_set = true;
  live.clear();
  calls = 0;
  fail_at = fail;
  launches = 0;
  int st = gbs::sell_build(&A, nullptr);
  out[0] = calls;
  if (fail >= 0) {
    fail_at = -1;
    last = cudaSuccess;
    launches = 0;
    if (gbs::sell_build(&A, nullptr) != GBS_OK) return -1;
  }
  out[1] = launches;
  out[2] = (int)live.size();
  out[3] = (A.sell_row0 != nullptr) + 2 * (A.sell_ptr != nullptr) + 4 * (A.sell_pat != nullptr) +
           8 * (A.sell_pool != nullptr) + 16 * (A.sell_mask != nullptr) +
           32 * (A.sell_val != nullptr) + 64 * (A.sell_off16 != nullptr) +
           128 * (A.sell_col != nullptr) + 256 * (int)A.nslices;
  gbs::free_sell(&A);
  out[4] = (int)live.size();
  return st;
}
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    d = tmp_path_factory.mktemp("sell")
    (d / "fake.cpp").write_text(SOURCE)
    try:
        nvcc = _build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    subprocess.run([nvcc, *_build.ARCH, "-std=c++17", "-O0", "-Xcompiler", "-fPIC", "-cudart",
                    "none", "--expt-relaxed-constexpr", "-Xlinker", "-Bsymbolic", "-I",
                    _build.INCLUDE, "-I", _build.CSRC, "-shared", "-o", str(d / "fake.so"),
                    os.path.join(_build.CSRC, "sell.cu"), str(d / "fake.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "fake.so"))

    def build(nsys, rows, patterns, fail):
        out = (ctypes.c_int * 5)()
        return lib.build(nsys, rows, patterns, fail, out), list(out)
    return build


@pytest.mark.parametrize("nsys, rows, patterns", [(1, 100, 1), (1, 100, 0), (3, 40, 1), (1, 0, 1)])
def test_failed_step_leaves_nothing(fake, nsys, rows, patterns):
    st, fresh = fake(nsys, rows, patterns, -1)
    assert st == 0 and fresh[4] == 0
    for k in range(fresh[0]):
        st, again = fake(nsys, rows, patterns, k)
        assert st > 0, k
        assert again[1:] == fresh[1:], k
