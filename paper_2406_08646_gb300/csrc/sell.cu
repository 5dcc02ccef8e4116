// Sliced-ELL copy of the assembled CSR matrix for the row products of the
// solves and of MatMult (Sec. 6.1).  The CSR arrays stay the assembled matrix
// (Sec. 5); this copy only changes how a warp reads it.
//
// Rows are cut into slices of 32 consecutive rows (aligned to each system's
// first row, so no slice straddles two systems).  Slice s has width w_s (its
// longest row) and holds 32 x w_s entries from b = sell_ptr[s] on, padding
// with column -1 and value 0.  Entries 2m and 2m + 1 of the slice's row i sit
// side by side at b + 64 m + 2 i (+1) for m < w_s / 2; an odd last entry sits
// at b + 64 (w_s / 2) + i.  A warp reads one slice with lane i on row i: each
// load instruction fetches a contiguous 256-byte (columns, FP32 values) or
// 512-byte (FP64 values) run holding two entries per lane, the x gathers of a
// stencil-like pattern are contiguous too, each row is summed in CSR order
// with one FMA per stored nonzero, and no cross-lane adds are needed.  b is a
// multiple of 32 entries, so the paired loads are aligned.
//
// Column patterns.  When the rows of every slice draw their offsets col -
// row from a common set of at most 32 (a stencil matrix's slices), each slice
// stores that set once (its pattern, ascending) and one 32-bit mask per row
// (bit k: the row holds pattern entry k); entry k of row i is then the value
// at the pattern's k-th offset, 0 where the row lacks it, and the slice's
// width is the pattern's size U.  The row products then read no column
// index: the columns follow from the row, the pattern (one broadcast load a
// pair) and the mask, which also skips the absent entries, so each row still
// takes one FMA per nonzero in CSR order (the same sums, bit for bit, as with
// column indices).  The copy takes patterns when every slice has U <= 32 and
// the U add up to at most 1.25 times the slices' longest rows (which bounds
// the zeros they add; slices across a layer seam of a stencil have U above
// their longest row); else it keeps column indices.  8 bytes per FP64 entry
// plus 4 per row instead of 10 or 12.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "device_util.cuh"
#include "internal.cuh"

namespace gbs {

static unsigned grid_of(int64_t n, int tpb) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + tpb - 1) / tpb, 1 << 20));
}

// The union of the offsets col - row of a slice's rows (lane i holds row r,
// its entries [j, je)), smallest first, by repeated warp minima over the
// rows' next offsets (a row's offsets ascend).  Returns its size, or 33 once
// it passes 32.  With pool set, lane 0 writes the offsets there and *mk gets
// each lane's mask.
__device__ int slice_union(const int32_t *__restrict__ col, int32_t r, int32_t j, int32_t je,
                           int lane, int32_t *__restrict__ pool, uint32_t *mk) {
  uint32_t m = 0;
  int n = 0;
  for (;;) {
    const int32_t c = j < je ? col[j] - r : INT32_MAX;
    const int32_t lo = __reduce_min_sync(0xffffffffu, c);
    if (lo == INT32_MAX) break;
    if (n == 32) return 33;
    if (c == lo) {
      m |= 1u << n;
      ++j;
    }
    if (pool && lane == 0) pool[n] = lo;
    ++n;
  }
  if (mk) *mk = m;
  return n;
}

// Sums over all slices, read back once: they decide patterns and sizes.
struct ShapeSums {
  unsigned long long w, u;  // longest rows; offset unions (33 at most each)
  int32_t over;             // a slice's union has more than 32 offsets
  int32_t nnz, coo;         // largest nonzeros and COO entries of a slice
  int32_t run;              // largest nonzeros of a run of slices (one system, cut into nruns)
  int32_t uneven, pad;      // run_uneven (a batch)
};

// One warp per slice: its first row (a batch's slices start at their system's
// first row: sys holds nsys + 1 first rows, then nsys + 1 first slices), w[s] =
// its longest row, u[s] = the size of its rows' offset union (33: more than
// 32, or patterns not built); their sums over all slices.  Block 0 also cuts one
// system's slices into nruns equal runs, as team.cu does; a batch's systems of 16
// slices and more are cut into 16.
constexpr int SHAPE_TPB = 256;
__global__ void __launch_bounds__(SHAPE_TPB)
    k_slice_shape(int64_t nslices, int64_t nrows, int32_t nsys, const int32_t *__restrict__ sys,
                  const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                  const int32_t *__restrict__ jmap, int32_t patterns, int32_t nruns,
                  int32_t *__restrict__ srow0, uint32_t *__restrict__ w,
                  uint32_t *__restrict__ u, ShapeSums *sums) {
  __shared__ unsigned long long sw[SHAPE_TPB / 32], su[SHAPE_TPB / 32];
  __shared__ int32_t sn[SHAPE_TPB / 32], se[SHAPE_TPB / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  unsigned long long tw = 0, tu = 0;
  int32_t nz = 0, ne = 0;
  bool over = false;
  if (!sys && blockIdx.x == 0) {
    int32_t run = 0;
    for (int k = threadIdx.x; k < nruns; k += SHAPE_TPB) {
      const int64_t f = 32 * (nslices * k / nruns), e = 32 * (nslices * (k + 1) / nruns);
      run = max(run, row_ptr[e < nrows ? e : nrows] - row_ptr[f < nrows ? f : nrows]);
    }
    run = __reduce_max_sync(0xffffffffu, run);
    if (lane == 0) atomicMax(&sums->run, run);
  }
  if (sys && nsys <= RUN_SYSTEMS) {
    const int k = (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 4, c = threadIdx.x & 15;
    if (k < nsys) {
      const int64_t f = sys[k], e = sys[k + 1], n = sys[nsys + 2 + k] - sys[nsys + 1 + k];
      const int64_t a = f + 32 * (n * c / 16), b = f + 32 * (n * (c + 1) / 16);
      const int64_t nn = row_ptr[e] - row_ptr[f];
      if (n >= 16 && nn > 0) {
        const int64_t x = 16 * RUN_EVEN * (int64_t)(row_ptr[b < e ? b : e] - row_ptr[a]) / nn;
        if (4 * x > 5 * RUN_EVEN) atomicMax(&sums->uneven, (int32_t)x);
      }
    }
  }
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslices; s += nw) {
    int64_t r0 = 32 * s, r1 = nrows;
    if (sys) {
      int lo = 0, hi = nsys;  // the last system whose first slice is <= s
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(sys + nsys + 1 + mid) <= s) lo = mid;
        else hi = mid;
      }
      r0 = __ldg(sys + lo) + 32 * (s - __ldg(sys + nsys + 1 + lo));
      r1 = __ldg(sys + lo + 1);
    }
    const int64_t r = r0 + lane;
    const bool live = r < r1;
    const int32_t rs = live ? row_ptr[r] : 0, re = live ? row_ptr[r + 1] : 0;
    const int32_t m = __reduce_max_sync(0xffffffffu, re - rs);
    const int n = patterns ? slice_union(col, (int32_t)r, rs, re, lane, nullptr, nullptr) : 33;
    if (lane == 0) {
      srow0[s] = (int32_t)r0;
      if (s == nslices - 1) srow0[nslices] = (int32_t)nrows;
      w[s] = (uint32_t)m;
      u[s] = (uint32_t)n;
    }
    const int64_t rl = r0 + 32 < r1 ? r0 + 32 : r1;
    const int32_t a = row_ptr[r0], b = row_ptr[rl];
    nz = max(nz, b - a);
    ne = max(ne, jmap[b] - jmap[a]);
    tw += (unsigned long long)m;
    tu += (unsigned long long)n;
    over = over || n > 32;
  }
  if (lane == 0) {
    sw[warp] = tw;
    su[warp] = tu;
    sn[warp] = nz;
    se[warp] = ne;
    if (over) sums->over = 1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < SHAPE_TPB / 32; ++k) {
      tw += sw[k];
      tu += su[k];
      nz = max(nz, sn[k]);
      ne = max(ne, se[k]);
    }
    atomicAdd(&sums->w, tw);
    atomicAdd(&sums->u, tu);
    if (nz > *(volatile int32_t *)&sums->nnz) atomicMax(&sums->nnz, nz);
    if (ne > *(volatile int32_t *)&sums->coo) atomicMax(&sums->coo, ne);
  }
}

// Entries (size[s]) and, with patterns, pool words (even) of each slice, for
// the scans that turn them into starts; one word beyond the last is 0.
__global__ void k_slice_sizes(int64_t nslices, const uint32_t *__restrict__ width,
                              uint32_t *__restrict__ size, uint32_t *__restrict__ pool) {
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s <= nslices;
       s += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t k = s < nslices ? width[s] : 0u;
    size[s] = 32u * k;
    if (pool) pool[s] = (k + 1u) & ~1u;
  }
}

// Position of entry k of a lane's row in slice storage from b on (pair
// layout; np = width / 2).
__device__ __forceinline__ int64_t sell_slot(int64_t b, int32_t k, int32_t np, int lane) {
  return k < 2 * np ? b + 64 * (k >> 1) + 2 * lane + (k & 1) : b + 64 * np + lane;
}

// Columns (SYM: with pat set each slice's pattern and row masks, else 32-bit
// columns or 16-bit offsets col - row, padding -1 / -32768) or values (0 in
// padding and in pattern entries a row lacks) of the sliced copy: one warp
// per slice, lane i on row i of the slice.
template <typename T, bool SYM>
__global__ void k_sell_fill(int64_t nslices, const int32_t *__restrict__ sptr,
                            const int32_t *__restrict__ srow0, const int32_t *__restrict__ row_ptr,
                            const int32_t *__restrict__ col, const T *__restrict__ val,
                            const int32_t *__restrict__ pat, int32_t *__restrict__ pool,
                            uint32_t *__restrict__ mask, int32_t *__restrict__ scol,
                            int16_t *__restrict__ soff, T *__restrict__ sval) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslices; s += nw) {
    const int32_t r = srow0[s] + lane;
    const bool live = r < srow0[s + 1];
    const int32_t rs = live ? row_ptr[r] : 0, len = live ? row_ptr[r + 1] - rs : 0;
    const int64_t b = sptr[s];
    const int32_t w = (int32_t)((sptr[s + 1] - b) >> 5), np = w >> 1;
    if (pat) {
      if constexpr (SYM) {
        uint32_t mk = 0;
        slice_union(col, r, rs, rs + len, lane, pool + pat[s], &mk);
        mask[32 * s + lane] = mk;
      } else {
        const uint32_t mk = mask[32 * s + lane];
        int32_t j = rs;
        for (int32_t k = 0; k < w; ++k) {
          const bool has = (mk >> k) & 1u;
          sval[sell_slot(b, k, np, lane)] = has ? val[j] : T(0);
          j += has ? 1 : 0;
        }
      }
      continue;
    }
    for (int32_t k = 0; k < w; ++k) {
      const bool ok = k < len;
      const int64_t q = sell_slot(b, k, np, lane);
      if constexpr (SYM) {
        if (scol) scol[q] = ok ? col[rs + k] : -1;
        if (soff) soff[q] = ok ? (int16_t)(col[rs + k] - r) : (int16_t)-32768;
      } else {
        sval[q] = ok ? val[rs + k] : T(0);
      }
    }
  }
}

// FP32 values of the sliced copy, RN(FP64 values), padding stays 0.
__global__ void k_sell_to_fp32(int64_t n, const double *__restrict__ v, float *__restrict__ v32) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x)
    v32[p] = __double2float_rn(v[p]);
}

void free_sell(gbs_mat A) {
  for (void *p : {(void *)A->sell_ptr, (void *)A->sell_row0, (void *)A->sell_col,
                  (void *)A->sell_off16, (void *)A->sell_val, (void *)A->sell_val32,
                  (void *)A->sell_pat, (void *)A->sell_pool, (void *)A->sell_mask})
    dev_free(p, nullptr);
  A->sell_pat = nullptr;
  A->sell_pool = nullptr;
  A->sell_mask = nullptr;
  A->sell_npat = 0;
  A->sell_nnz_rows = 0;
  A->sell_ptr = nullptr;
  A->sell_row0 = nullptr;
  A->sell_col = nullptr;
  A->sell_off16 = nullptr;
  A->sell_val = nullptr;
  A->sell_val32 = nullptr;
  A->nslices = A->sell_nnz = 0;
}

// ... after a failed step, once the steps before it are done with the arrays.
static void drop_copy(gbs_mat A, cudaStream_t s) {
  cudaStreamSynchronize(s);
  free_sell(A);
}

// The slice table, the column patterns chosen and the padded size.
static int shape_copy(gbs_mat A, cudaStream_t st) {
  A->sell_slice0_h.assign(A->nsys + 1, 0);
  for (int32_t q = 0; q < A->nsys; ++q)
    A->sell_slice0_h[q + 1] =
        A->sell_slice0_h[q] + (int32_t)((A->row_off_h[q + 1] - A->row_off_h[q] + 31) / 32);
  const int64_t ns = A->sell_slice0_h[A->nsys];
  ShapeSums h;
  memset(&h, 0, sizeof(h));
  // w, u (ns + 1 words each, 16-byte aligned), the sums, a batch's first rows and slices
  const int64_t pad = (ns + 4) & ~(int64_t)3, nsy = A->nsys > 1 ? 2 * (A->nsys + 1) : 0;
  uint32_t *d = nullptr;
  GBS_TRY(dev_alloc(&A->sell_row0, ns + 1, st));
  int32_t *const row0 = A->sell_row0;
  if (ns == 0) {
    const int32_t end = (int32_t)A->nrows;
    GBS_TRY_CUDA(cudaMemcpyAsync(row0, &end, sizeof(end), cudaMemcpyHostToDevice, st));
  }
  struct Scratch {  // returned to the pool on every exit path
    uint32_t *p = nullptr;
    cudaStream_t s;
    ~Scratch() { dev_free(p, s); }
  } scratch{nullptr, st};
  GBS_TRY(dev_alloc(&scratch.p, 2 * pad + (int64_t)sizeof(ShapeSums) / 4 + nsy, st));
  d = scratch.p;
  uint32_t *w = d, *u = d + pad;
  ShapeSums *sums = reinterpret_cast<ShapeSums *>(d + 2 * pad);
  int32_t *sys = nsy ? reinterpret_cast<int32_t *>(sums + 1) : nullptr;
  if (ns > 0) {
    GBS_TRY_CUDA(cudaMemsetAsync(sums, 0, sizeof(ShapeSums), st));
    if (sys) {
      std::vector<int32_t> t(nsy);
      for (int32_t q = 0; q <= A->nsys; ++q) {
        t[q] = (int32_t)A->row_off_h[q];
        t[A->nsys + 1 + q] = A->sell_slice0_h[q];
      }
      GBS_TRY_CUDA(cudaMemcpyAsync(sys, t.data(), sizeof(int32_t) * nsy, cudaMemcpyHostToDevice,
                                   st));
    }
    k_slice_shape<<<grid_of(ns * 32, SHAPE_TPB), SHAPE_TPB, 0, st>>>(
        ns, A->nrows, A->nsys, sys, A->row_ptr, A->col, A->jmap, A->sell_patterns ? 1 : 0,
        sm_count(A), row0, w, u, sums);
    GBS_LAUNCHED(1);
    GBS_TRY_CUDA(cudaMemcpyAsync(&h, sums, sizeof(h), cudaMemcpyDeviceToHost, st));
    GBS_TRY_CUDA(cudaStreamSynchronize(st));
  }
  // patterns when every slice has at most 32 offsets and they add at most a
  // quarter to the entries; pattern starts are even (pair loads)
  const bool fit = A->sell_patterns && ns > 0 && !h.over && 4 * h.u <= 5 * h.w;
  const int64_t total = 32 * (int64_t)(fit ? h.u : h.w);
  A->sell_nnz_rows = 32 * (int64_t)h.w;
  A->slice_max_nnz = h.nnz;
  A->slice_max_coo = h.coo;
  A->run_max_nnz = h.run;
  A->run_uneven = h.uneven;
  A->nslices = ns;
  A->sell_nnz = total;
  if (total > 2147483647LL) return GBS_OK;  // too large for 32-bit offsets: no copy
  GBS_TRY(dev_alloc(&A->sell_ptr, ns + 1, st));
  if (ns > 0) {
    uint32_t *tmp = nullptr;
    GBS_TRY(dev_alloc(&tmp, scan_tmp_words(ns + 1), st));
    struct Scratch tmp_free {tmp, st};
    if (fit) {
      GBS_TRY(dev_alloc(&A->sell_pat, ns + 1, st));
      GBS_TRY(dev_alloc(&A->sell_pool, h.u + ns + 2, st));  // (each start rounded up to even)
      GBS_TRY(dev_alloc(&A->sell_mask, 32 * ns, st));
    }
    uint32_t *ptr = reinterpret_cast<uint32_t *>(A->sell_ptr);
    uint32_t *pat = reinterpret_cast<uint32_t *>(A->sell_pat);
    k_slice_sizes<<<grid_of(ns + 1, 256), 256, 0, st>>>(ns, fit ? u : w, ptr, pat);
    GBS_LAUNCHED(1);
    GBS_TRY(exclusive_scan(ptr, ptr, ns + 1, tmp, nullptr, st));
    if (fit) GBS_TRY(exclusive_scan(pat, pat, ns + 1, tmp, nullptr, st));
  } else {
    GBS_TRY_CUDA(cudaMemsetAsync(A->sell_ptr, 0, sizeof(int32_t), st));
  }
  A->sell_npat = fit ? ns : 0;
  return GBS_OK;
}

// Slice table, column patterns chosen and padded size (no entries yet); when
// the padded size reaches 2^31 only the size is recorded.  Idempotent.
// Synchronises s once: the sums over the slices decide the sizes (the tables
// themselves stay on the device).  sell_row0 and sell_val say that the shape
// and the copy exist: where a step fails, what the others made goes back, so
// that the next call starts over instead of using half a copy.
int sell_shape(gbs_mat A, cudaStream_t st) {
  if (A->sell_row0) return GBS_OK;
  const int status = shape_copy(A, st);
  if (status != GBS_OK) drop_copy(A, st);
  return status;
}

// The copy's arrays beyond its shape: column patterns' masks and offsets or
// column indices, and the values if they are set.
static int fill_copy(gbs_mat A, cudaStream_t s) {
  const size_t m = (size_t)std::max<int64_t>(A->sell_nnz, 1);
  GBS_TRY(dev_alloc(&A->sell_val, m, s));
  if (A->sell_npat == 0) {
    if (A->col_span <= 32767) GBS_TRY(dev_alloc(&A->sell_off16, m, s));
    else GBS_TRY(dev_alloc(&A->sell_col, m, s));
  }
  if (A->nslices > 0) {
    k_sell_fill<double, true><<<grid_of(A->nslices * 32, 256), 256, 0, s>>>(
        A->nslices, A->sell_ptr, A->sell_row0, A->row_ptr, A->col, (const double *)nullptr,
        A->sell_npat ? A->sell_pat : nullptr, A->sell_pool, A->sell_mask, A->sell_col,
        A->sell_off16, (double *)nullptr);
    GBS_LAUNCHED(1);
  }
  return A->values_set ? sell_values(A, s) : GBS_OK;
}

// Column patterns or column indices and, if the values are set, FP64 values
// of the sliced copy.  Column indices are stored as 16-bit offsets col - row
// when every column lies within 2^15 - 1 of its row (the symbolic stage
// measured the span), else as 32-bit columns.
int sell_build(gbs_mat A, cudaStream_t s) {
  GBS_TRY(sell_shape(A, s));
  if (!A->sell_ptr) {
    set_error("the sliced-ELL copy would hold %lld entries (limit 2^31 - 1)",
              (long long)A->sell_nnz);
    return GBS_ERR_ARG;
  }
  if (A->sell_val) return GBS_OK;
  const int status = fill_copy(A, s);
  if (status != GBS_OK) drop_copy(A, s);
  return status;
}

// FP64 values of the sliced copy from the CSR values (after every numeric
// stage); the FP32 copy is refreshed by sell_values32 when a refined solve
// needs it.
int sell_values(gbs_mat A, cudaStream_t s) {
  if (!A->sell_val || A->nslices == 0) return GBS_OK;
  k_sell_fill<double, false><<<grid_of(A->nslices * 32, 256), 256, 0, s>>>(
      A->nslices, A->sell_ptr, A->sell_row0, A->row_ptr, A->col, A->val,
      A->sell_npat ? A->sell_pat : nullptr, A->sell_pool, A->sell_mask, (int32_t *)nullptr,
      (int16_t *)nullptr, A->sell_val);
  GBS_LAUNCHED(1);
  return GBS_OK;
}

int sell_values32(gbs_mat A, cudaStream_t s) {
  if (!A->sell_val) return GBS_OK;
  if (!A->sell_val32) GBS_TRY(dev_alloc(&A->sell_val32, std::max<int64_t>(A->sell_nnz, 1), s));
  if (A->sell_nnz > 0) {
    k_sell_to_fp32<<<grid_of(A->sell_nnz, 256), 256, 0, s>>>(A->sell_nnz, A->sell_val,
                                                             A->sell_val32);
    GBS_LAUNCHED(1);
  }
  return GBS_OK;
}

SellView sell_view(gbs_mat A) {
  SellView v;
  v.ptr = A->sell_ptr;
  v.row0 = A->sell_row0;
  v.col = A->sell_off16 ? nullptr : A->sell_col;
  v.off = A->sell_off16;
  v.pat = A->sell_npat ? A->sell_pat : nullptr;
  v.pool = A->sell_pool;
  v.mask = A->sell_mask;
  return v;
}

// Rebuilds a sliced copy that exists (and its transpose's) with or without
// column patterns; the cached graphs hold the old arrays and are dropped.
int set_slice_patterns(gbs_mat A, bool on, cudaStream_t s) {
  if (A->At && A->At->sell_patterns != on) {
    GBS_TRY(set_slice_patterns(A->At, on, s));
    drop_graphs(A);  // A's BiCG graphs hold the transpose's arrays
  }
  if (A->sell_patterns == on) return GBS_OK;
  A->sell_patterns = on;
  if (!A->sell_row0) return GBS_OK;
  const bool built = A->sell_val != nullptr, fp32 = A->sell_val32 != nullptr;
  GBS_TRY_CUDA(cudaStreamSynchronize(s));  // the old copy may be in use
  drop_graphs(A);
  free_sell(A);
  GBS_TRY(sell_shape(A, s));
  if (built) GBS_TRY(sell_build(A, s));
  if (fp32) GBS_TRY(sell_values32(A, s));
  return GBS_OK;
}

}  // namespace gbs
