// MatMult (Sec. 6.1): y = A x on the assembled CSR, FP64, and the launch plan
// (block tables, lanes per row, grid caps) shared with the solves.
#include <cuda_runtime.h>

#include <algorithm>

#include "device_util.cuh"
#include "internal.cuh"
#include "phases.cuh"

namespace gbs {

constexpr int SPMV_ROWS = PHASE_TPB;  // rows per CTA pass of the CSR-vector SpMV (32 per warp)

// y = A x with the CSR-vector row product of the solves (csr_rows), over
// chunks of 32 rows per warp.
template <int L>
__global__ void __launch_bounds__(PHASE_TPB) k_spmv(const int32_t *__restrict__ row_ptr,
                                                    const int32_t *__restrict__ col,
                                                    const double *__restrict__ val,
                                                    const double *__restrict__ x,
                                                    double *__restrict__ y, int32_t n,
                                                      const int32_t *__restrict__ order) {
  auto f = [&](int r, double s) { y[r] = s; };
  for (int64_t r0 = (int64_t)blockIdx.x * SPMV_ROWS; r0 < n;
       r0 += (int64_t)gridDim.x * SPMV_ROWS) {
    const int r1 = (int)(r0 + SPMV_ROWS < n ? r0 + SPMV_ROWS : n);
    csr_rows<double, L, false>(row_ptr, col, val, x, (int)r0, r1, order, f);
  }
}

// order[r0 .. r1): the rows of [r0, r1) by decreasing length (ties by index),
// in windows of at most W rows from r0 on -- one CTA a window, a bitonic sort in
// shared memory.  Windows start at the blocks' first rows (row0, nblocks + 1)
// or, without blocks, every W rows.
constexpr int ORDER_W = 1024;
__global__ void __launch_bounds__(ORDER_W)
    k_row_order(int32_t nblocks, const int32_t *__restrict__ row0, int32_t n, int32_t W,
                const int32_t *__restrict__ row_ptr, int32_t *__restrict__ order) {
  __shared__ uint32_t key[ORDER_W];
  const int t = (int)threadIdx.x;
  for (int b = blockIdx.x; b < nblocks; b += gridDim.x) {
    const int64_t f = row0 ? row0[b] : (int64_t)b * W;
    const int64_t e = row0 ? row0[b + 1] : (f + W < n ? f + W : n);
    for (int64_t w = f; w < e; w += W) {
      const int m = e - w < W ? (int)(e - w) : W;
      uint32_t k = ~0u;
      if (t < m) {
        const int len = row_ptr[w + t + 1] - row_ptr[w + t];
        k = ((uint32_t)(0x1fffff - min(len, 0x1fffff)) << 10) | (uint32_t)t;
      }
      key[t] = k;
      __syncthreads();
      for (int s = 2; s <= ORDER_W; s <<= 1)
        for (int j = s >> 1; j > 0; j >>= 1) {
          const int q = t ^ j;
          if (q > t) {
            const uint32_t u = key[t], v = key[q];
            if ((u > v) == ((t & s) == 0)) {
              key[t] = v;
              key[q] = u;
            }
          }
          __syncthreads();
        }
      if (t < m) order[w + t] = (int32_t)(w + (int)(key[t] & 1023u));
      __syncthreads();
    }
  }
}

// The row orders of a CSR-vector plan (after table A).
static int build_row_orders(gbs_mat A, cudaStream_t st) {
  const int64_t n = A->nrows;
  if (n == 0) return GBS_OK;
  if (!A->order_s) {
    int32_t *order = nullptr;
    GBS_TRY(dev_alloc(&order, 2 * (size_t)n, st));
    const int32_t nb = (int32_t)((n + SPMV_ROWS - 1) / SPMV_ROWS);
    k_row_order<<<(unsigned)std::min(nb, 1 << 16), ORDER_W, 0, st>>>(
        nb, nullptr, (int32_t)n, SPMV_ROWS, A->row_ptr, order);
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) dev_free(order, st);
    GBS_TRY_CUDA(e);
    A->order_s = order;
  }
  k_row_order<<<(unsigned)std::min(std::max(A->ta.nblocks, 1), 1 << 16), ORDER_W, 0, st>>>(
      A->ta.nblocks, A->ta.row0, (int32_t)n, ORDER_W, A->row_ptr, A->order_s + n);
  GBS_LAUNCHED(1);
  A->order_a = A->order_s + n;
  return GBS_OK;
}

// y = A x with the sliced-ELL row product (sell_rows), 16 slices per CTA pass.
__global__ void __launch_bounds__(PHASE_TPB, SELL_MIN_CTAS)
    k_spmv_sell(const SellView S, const double *__restrict__ sval,
                const double *__restrict__ x, double *__restrict__ y, int32_t nslices,
                int32_t stream_matrix) {
  auto f = [&](int r, double s) { y[r] = s; };
  const int per = PHASE_TPB / 32;
  for (int64_t s0 = (int64_t)blockIdx.x * per; s0 < nslices; s0 += (int64_t)gridDim.x * per) {
    const int s1 = (int)(s0 + per < nslices ? s0 + per : nslices);
    if (stream_matrix)
      sell_rows<double, true, GATHER_NC>(S, sval, x, (int)s0, s1, f);
    else sell_rows<double, false, GATHER_NC>(S, sval, x, (int)s0, s1, f);
  }
}

// The same with 64 registers a thread on a grid of two CTAs an SM, one wave,
// each with its run of slices: sell_rows_deep, which has four pairs a thread and
// the next slice's tables in flight.  The FP64 pipe bounds wide slices in both
// (Q1 96^3: 40 us of FMAs), HBM and the gathers' latency narrow ones.
// k_spmv_sell's many small CTAs balance themselves and, four of them an SM, hide
// more latency where slices are narrow, so this form is taken where it was
// measured to be the faster one (deep_form).  Measured, us a product,
// k_spmv_sell / this (waves of slices in brackets):
//   27-point 60^3 (1.4) 14.5 / 15.9   64^3 (1.8) 19.1 / 16.6   72^3 (2.5) 25.0 / 23.3
//            80^3 (3.4) 29.3 / 30.5   96^3 (5.9) 48.0 / 45.9   90^3 (4.8) 38.9 / 37.5
//            102^3 (7.0) 52.1 / 55.3  120^3 (11.4) 85.7 / 87.2
//            (mean of 18 sizes between 1.5 and 7 waves: 3% faster; 0.95 to 1.15)
//   19-point 60^3 9.7 / 10.1   120^3 59.7 / 62.2   13-point 700^2 15.5 / 17.9   9-point 1000^2 20.1 / 24.1
//   7-point  70^3 6.7 / 7.3    140^3 (208 MB) 40.2 / 41.2
//            150^3 (256 MB) 52.8 / 50.3   170^3 83.3 / 76.4   192^3 118.5 / 112.5
//   9-point 2000^2 (368 MB, near neighbours) 78.8 / 84.4
//   27-point 65^3 followed by three times as many diagonal rows 19.1 / 44.3, by
//            7-point 90^3 25.4 / 41.5
// (The slices dealt to the CTAs in turns: the same mean, 0.97 to 1.12, 96^3 1% slower,
// 7-point 150^3 54.0; the uneven ones 21.9 and 26.8, slower than k_spmv_sell still.)
constexpr int DEEP_CTAS = 2;
__global__ void __launch_bounds__(PHASE_TPB, DEEP_CTAS)
    k_spmv_sell_deep(const SellView S, const double *__restrict__ sval,
                     const double *__restrict__ x, double *__restrict__ y, int32_t nslices,
                     int32_t ncols, int32_t stream_matrix) {
  auto f = [&](int r, double s) { y[r] = s; };
  const int s0 = (int)((int64_t)nslices * blockIdx.x / gridDim.x);
  const int s1 = (int)((int64_t)nslices * (blockIdx.x + 1) / gridDim.x);
  if (stream_matrix)
    sell_rows<double, true, GATHER_NC, false, 4>(S, sval, x, s0, s1, f, ncols - 1);
  else sell_rows<double, false, GATHER_NC, false, 4>(S, sval, x, s0, s1, f, ncols - 1);
}

// Whether MatMult takes k_spmv_sell_deep.  Slices have to be alike (the largest
// at most an eighth over the mean), or the CTAs' runs are not; then wide ones (24
// entries a row and more) from 1.5 up to 7 waves, and narrow ones (6 to 12) of matrices
// that stream from HBM (from 7/4 of the L2's size on) and gather from afar (8192
// rows and more away).
constexpr double DEEP_WIDTH = 6.0, DEEP_NARROW = 12.0, DEEP_WIDE = 24.0;
constexpr int32_t DEEP_SPAN = 8192;
static bool deep_form(gbs_mat A) {
  const int64_t ns = A->nslices;
  const double width = (double)A->sell_nnz / (32.0 * (double)ns);
  if (A->sell_npat == 0 || width < DEEP_WIDTH ||
      8.0 * (double)A->slice_max_nnz * (double)ns > 9.0 * (double)A->nnz)
    return false;
  const int64_t wave = (int64_t)DEEP_CTAS * sm_count(A) * (PHASE_TPB / 32);  // slices of a wave
  if (width >= DEEP_WIDE) return 2 * ns >= 3 * wave && ns < 7 * wave;
  if (width > DEEP_NARROW || A->col_span < DEEP_SPAN) return false;
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, A->device);
  return 4 * (8 * A->sell_nnz + 20 * A->nrows) >= 7 * (int64_t)l2;
}

int launch_spmv(gbs_mat A, const double *x, double *y, cudaStream_t s) {
  if (A->nrows == 0) return GBS_OK;
  const int32_t n = (int32_t)A->nrows;
  if (A->lanes == GBS_SPMV_SELL) {
    GBS_TRY(sell_build(A, s));  // a no-op once built
    const int64_t ns = A->nslices, per = PHASE_TPB / 32;
    const int64_t ctas = (ns + per - 1) / per;
    if (deep_form(A))
      k_spmv_sell_deep<<<(unsigned)(DEEP_CTAS * sm_count(A)), PHASE_TPB, 0, s>>>(
          sell_view(A), A->sell_val, x, y, (int32_t)ns, (int32_t)A->ncols, stream_matrix(A, 12));
    else
      k_spmv_sell<<<(unsigned)std::min<int64_t>(ctas, 1 << 20), PHASE_TPB, 0, s>>>(
          sell_view(A), A->sell_val, x, y, (int32_t)ns, stream_matrix(A, 12));
    GBS_LAUNCHED(1);
    return GBS_OK;
  }
  const int64_t chunks = (A->nrows + SPMV_ROWS - 1) / SPMV_ROWS;
  const unsigned grid = (unsigned)std::min<int64_t>(chunks, 1 << 20);
  const int32_t *const order = A->order_a ? A->order_s : nullptr;
  switch (A->lanes) {
    case 1: k_spmv<1><<<grid, PHASE_TPB, 0, s>>>(A->row_ptr, A->col, A->val, x, y, n, order); break;
    case 2: k_spmv<2><<<grid, PHASE_TPB, 0, s>>>(A->row_ptr, A->col, A->val, x, y, n, order); break;
    case 8: k_spmv<8><<<grid, PHASE_TPB, 0, s>>>(A->row_ptr, A->col, A->val, x, y, n, order); break;
    case 32: k_spmv<32><<<grid, PHASE_TPB, 0, s>>>(A->row_ptr, A->col, A->val, x, y, n, order); break;
    default: k_spmv<4><<<grid, PHASE_TPB, 0, s>>>(A->row_ptr, A->col, A->val, x, y, n, order); break;
  }
  GBS_LAUNCHED(1);
  return GBS_OK;
}

// 1 when the sliced copy (bytes_per_entry per padded entry) is larger than
// half of L2: its loads then carry the evict-first hint.
int32_t stream_matrix(gbs_mat A, int bytes_per_entry) {
  int l2 = 0;
  if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, A->device) != cudaSuccess) l2 = 0;
  return (double)A->sell_nnz * bytes_per_entry > 0.5 * (double)l2 ? 1 : 0;
}

// Lanes per row from the mean row length: enough lanes that a warp's loads
// cover whole 32-byte sectors of the value stream, few enough that masked
// slots and the cross-lane adds stay a small part of the FP64 work.
int auto_lanes(int64_t nnz, int64_t nrows) {
  const double m = nrows > 0 ? (double)nnz / (double)nrows : 0.0;
  if (m < 3.0) return 1;
  if (m < 12.0) return 2;
  if (m < 48.0) return 4;
  if (m < 160.0) return 8;
  return 32;
}

void free_table(TableDev &t) {
  dev_free(t.row0, nullptr);  // one buffer holds all five arrays (build_table)
  t.row0 = t.sys = t.sys_blk0 = t.sys_slot0 = t.slice0 = t.row1 = t.slice1 = nullptr;
  t.nblocks = 0;
  t.grid = 0;
  t.nslots = 0;
  t.sys_blk0_h.clear();
}

// Each system's rows cut into ceil(n_s / R) blocks of R rows (the last one
// ragged); blocks never straddle systems.  R is a multiple of 32, so a block
// is a whole number of the 32-row slices of the sliced-ELL layout (slice0).
// The kernels walking the table run min(blocks, cap_per_sm x SMs) CTAs;
// system s owns min(blocks_s, grid) reduction slots.
// min_rows > 0: only the systems of at least min_rows rows get blocks (the
// size split's table; the others have none and are never visited).
static int build_table(gbs_mat A, int32_t R, int32_t cap_per_sm, TableDev &t, cudaStream_t st,
                       int64_t min_rows = 0) {
  std::vector<int32_t> row0, sys, sb0(A->nsys + 1, 0), sl0, row1, sl1;
  int32_t slices = 0;
  for (int32_t q = 0; q < A->nsys; ++q) {
    const int64_t a = A->row_off_h[q], e = A->row_off_h[q + 1];
    for (int64_t r = a; r < e && e - a >= min_rows; r += R) {
      const int64_t re = std::min<int64_t>(r + R, e);
      row0.push_back((int32_t)r);
      sys.push_back(q);
      sl0.push_back(slices + (int32_t)((r - a) / 32));
      row1.push_back((int32_t)re);
      sl1.push_back(slices + (int32_t)((re - a + 31) / 32));
    }
    slices += (int32_t)((e - a + 31) / 32);
    sb0[q + 1] = (int32_t)row0.size();
  }
  row0.push_back((int32_t)A->nrows);
  sl0.push_back(slices);
  const int32_t nb = (int32_t)sys.size();
  int nsm = 0;
  GBS_TRY_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, A->device));
  int64_t grid = std::min<int64_t>(nb, (int64_t)std::max(cap_per_sm, 1) * nsm);
  grid = std::max<int64_t>(grid, 1);
  std::vector<int32_t> so(A->nsys + 1, 0);
  for (int32_t q = 0; q < A->nsys; ++q)
    so[q + 1] = so[q] + (int32_t)std::min<int64_t>(sb0[q + 1] - sb0[q], grid);
  free_table(t);
  // one buffer: row0 (nb + 1), slice0 (nb + 1), sys (nb), sys_blk0, sys_slot0 (nsys + 1
  // each), and with gaps (min_rows > 0) row1, slice1 (nb each)
  const bool ends = min_rows > 0;
  const size_t tot = 3 * (size_t)nb + 2 + 2 * ((size_t)A->nsys + 1) + (ends ? 2 * (size_t)nb : 0);
  std::vector<int32_t> h;
  h.reserve(tot);
  h.insert(h.end(), row0.begin(), row0.end());
  h.insert(h.end(), sl0.begin(), sl0.end());
  h.insert(h.end(), sys.begin(), sys.end());
  h.insert(h.end(), sb0.begin(), sb0.end());
  h.insert(h.end(), so.begin(), so.end());
  if (ends) {
    h.insert(h.end(), row1.begin(), row1.end());
    h.insert(h.end(), sl1.begin(), sl1.end());
  }
  int32_t *d = nullptr;
  GBS_TRY(dev_alloc(&d, tot, st));
  GBS_TRY_CUDA(cudaMemcpyAsync(d, h.data(), sizeof(int32_t) * tot, cudaMemcpyHostToDevice, st));
  t.row0 = d;
  t.slice0 = d + nb + 1;
  t.sys = d + 2 * (size_t)nb + 2;
  t.sys_blk0 = t.sys + nb;
  t.sys_slot0 = t.sys_blk0 + A->nsys + 1;
  t.row1 = ends ? t.sys_slot0 + A->nsys + 1 : nullptr;
  t.slice1 = ends ? t.row1 + nb : nullptr;
  t.sys_blk0_h = sb0;
  t.nblocks = nb;
  t.grid = (int32_t)grid;
  t.nslots = std::max<int64_t>(so[A->nsys], 1);
  return GBS_OK;
}

// The one-kernel CG's wait window over table A (blocks of R rows per
// system, grid G, CTA c taking blocks c, c + G, ...): block b's row products
// read rows within col_span of its own, i.e. blocks b - lo_b .. b + hi_b;
// with lo and hi the largest lo_b and hi_b, CTA c's blocks need only CTAs
// c - lo .. c + hi (mod G).  halo_lo = lo, halo_n = lo + hi + 1, or the
// whole grid (halo_lo = 0, halo_n = G) when that window would wrap onto
// itself.
static void halo_window(gbs_mat A, int32_t R, const TableDev &t) {
  std::vector<int64_t> row0;
  for (int32_t q = 0; q < A->nsys; ++q)
    for (int64_t r = A->row_off_h[q]; r < A->row_off_h[q + 1]; r += R) row0.push_back(r);
  const int64_t nb = (int64_t)row0.size();
  row0.push_back(A->nrows);
  const int64_t span = A->col_span;
  auto blk = [&](int64_t r) {  // the block holding row r, 0 <= r < nrows
    return (int64_t)(std::upper_bound(row0.begin(), row0.end() - 1, r) - row0.begin()) - 1;
  };
  int64_t lo = 0, hi = 0;
  for (int64_t b = 0; b < nb; ++b) {
    const int64_t a = std::max<int64_t>(0, row0[b] - span);
    const int64_t e = std::min<int64_t>(A->nrows - 1, row0[b + 1] - 1 + span);
    lo = std::max(lo, b - blk(a));
    hi = std::max(hi, blk(e) - b);
  }
  const int64_t G = std::max<int32_t>(t.grid, 1);
  if (nb == 0) {
    A->halo_lo = A->halo_n = 0;
  } else if (lo + hi + 1 >= G) {
    A->halo_lo = 0;
    A->halo_n = (int32_t)G;
  } else {
    A->halo_lo = (int32_t)lo;
    A->halo_n = (int32_t)(lo + hi + 1);
  }
}

// The size split's tables: the systems of at least split_rows rows, cut into
// blocks sized for them alone (about one block per CTA of a one-wave grid, as
// the plan's automatic sizes are for the whole batch), at the plan's
// occupancy.  Rebuilt when the split or the plan changes.
int build_split_tables(gbs_mat A, cudaStream_t st) {
  if (A->split_built == A->split_rows && A->sa.row0) return GBS_OK;
  int occ_rows = 1, occ_upd = 1, nsm = 1;
  GBS_TRY(phase_occupancy(A->lanes, &occ_rows, &occ_upd));
  GBS_TRY_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, A->device));
  const int cap_a = A->ctas_per_sm ? A->ctas_per_sm : occ_rows;
  const int cap_e = A->ctas_per_sm ? A->ctas_per_sm : occ_upd;
  int64_t rows = 0;
  for (int32_t q = 0; q < A->nsys; ++q) {
    const int64_t n = A->row_off_h[q + 1] - A->row_off_h[q];
    if (n >= A->split_rows) rows += n;
  }
  auto auto_rows = [&](int cap) {
    const int64_t per = (rows + (int64_t)cap * nsm - 1) / ((int64_t)cap * nsm);
    return (int32_t)std::min<int64_t>(65536, std::max<int64_t>(PHASE_TPB, (per + 31) / 32 * 32));
  };
  GBS_TRY(build_table(A, auto_rows(cap_a), cap_a, A->sa, st, A->split_rows));
  GBS_TRY(build_table(A, auto_rows(cap_e), cap_e, A->se, st, A->split_rows));
  A->split_built = A->split_rows;
  return GBS_OK;
}

// nnz_off[q] = row_ptr[first row of system q] (q = 0 .. nsys).
__global__ void k_system_nnz(int32_t nsys, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ row0,
                             const int32_t *__restrict__ sys_blk0, int32_t *__restrict__ nnz_off) {
  const int32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q <= nsys) nnz_off[q] = row_ptr[row0[sys_blk0[q]]];
}

// Systems in decreasing row count (ties by index): the per-CTA solver hands
// them to CTAs in this order, so the longest solves start first.  Also the
// largest system's rows and nonzeros (the solver choice uses them; a batch's
// per-system counts are read back, which synchronises st).
static int build_cta_order(gbs_mat A, cudaStream_t st) {
  std::vector<int32_t> ord(A->nsys), noff(A->nsys + 1, 0);
  if (A->nsys == 1) {
    noff[1] = (int32_t)A->nnz;
  } else {
    int32_t *d = nullptr;
    GBS_TRY(dev_alloc(&d, A->nsys + 1, st));
    k_system_nnz<<<(A->nsys + 256) / 256, 256, 0, st>>>(A->nsys, A->row_ptr, A->ta.row0,
                                                        A->ta.sys_blk0, d);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(noff.data(), d, sizeof(int32_t) * (A->nsys + 1), cudaMemcpyDeviceToHost,
                          st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    dev_free(d, st);
    count_launches(1);
    GBS_TRY_CUDA(e);
  }
  A->max_sys_rows = A->max_sys_nnz = 0;
  for (int32_t q = 0; q < A->nsys; ++q) {
    ord[q] = q;
    A->max_sys_rows = std::max(A->max_sys_rows, A->row_off_h[q + 1] - A->row_off_h[q]);
    A->max_sys_nnz = std::max<int64_t>(A->max_sys_nnz, noff[q + 1] - noff[q]);
  }
  std::stable_sort(ord.begin(), ord.end(), [&](int32_t u, int32_t v) {
    return A->row_off_h[u + 1] - A->row_off_h[u] > A->row_off_h[v + 1] - A->row_off_h[v];
  });
  A->cta_order_h = ord;
  A->sys_nnz_h.resize(A->nsys);
  for (int32_t k = 0; k < A->nsys; ++k) A->sys_nnz_h[k] = noff[ord[k] + 1] - noff[ord[k]];
  A->batch_engine[0] = A->batch_engine[1] = -1;
  if (!A->cta_order) GBS_TRY(dev_alloc(&A->cta_order, A->nsys, st));
  if (A->nsys == 1) {
    GBS_TRY_CUDA(cudaMemsetAsync(A->cta_order, 0, sizeof(int32_t), st));
    return GBS_OK;
  }
  GBS_TRY_CUDA(cudaMemcpyAsync(A->cta_order, ord.data(), sizeof(int32_t) * A->nsys,
                               cudaMemcpyHostToDevice, st));
  GBS_TRY_CUDA(cudaStreamSynchronize(st));  // ord is a local vector
  return GBS_OK;
}

// Plan: SpMV-phase blocks of Ra rows, update-phase blocks of Re rows (both
// multiples of 32), the row-product kernel (GBS_SPMV_AUTO, GBS_SPMV_SELL or
// CSR-vector lanes per row) and a cap of CTAs per SM on the grids (0: as many
// as fit on an SM at once, so each phase kernel runs in one wave).  Cached graphs are dropped: they bake in the tables and grids.
// Work is ordered on stream st; the host copies of the tables are synchronous.
int build_plan(gbs_mat A, int32_t Ra, int32_t Re, int32_t kernel, int32_t ctas_per_sm,
               cudaStream_t st) {
  const bool bad_ra = Ra != 0 && (Ra < 32 || Ra > 65536 || (Ra % 32) != 0);
  const bool bad_re = Re != 0 && (Re < 32 || Re > 65536 || (Re % 32) != 0);
  if (bad_ra || bad_re ||
      !(kernel == GBS_SPMV_AUTO || kernel == GBS_SPMV_SELL || kernel == 1 || kernel == 2 ||
        kernel == 4 || kernel == 8 || kernel == 32) ||
      ctas_per_sm < 0 || ctas_per_sm > 64) {
    set_error("plan: spmv_rows %d and update_rows %d must be 0 (auto) or multiples of 32 in "
              "[32, 65536], "
              "kernel %d one of -1 (auto), 0 (sliced ELL), 1, 2, 4, 8, 32 (CSR lanes), "
              "ctas_per_sm %d in [0, 64]",
              Ra, Re, kernel, ctas_per_sm);
    return GBS_ERR_ARG;
  }
  const bool all_auto = Ra == 0 && Re == 0 && kernel == GBS_SPMV_AUTO && ctas_per_sm == 0;
  drop_graphs(A);
  free_table(A->sa);  // the size split's tables follow the plan
  free_table(A->se);
  A->split_built = 0;
  A->order_a = nullptr;  // (it orders the rows of table A's blocks, which change below)
  if (kernel == GBS_SPMV_AUTO) {
    GBS_TRY(sell_shape(A, st));
    kernel = (A->sell_ptr && (double)A->sell_nnz_rows <= 1.2 * (double)A->nnz)
                 ? GBS_SPMV_SELL
                 : auto_lanes(A->nnz, A->nrows);
  }
  if (kernel == GBS_SPMV_SELL) GBS_TRY(sell_build(A, st));
  // grids: one wave of the phase kernels unless capped explicitly; automatic
  // block sizes give about one block per CTA of that wave (at least one row
  // per thread, so every warp of a CTA has rows)
  int occ_rows = 1, occ_upd = 1, nsm = 1;
  GBS_TRY(phase_occupancy(kernel, &occ_rows, &occ_upd));
  GBS_TRY_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, A->device));
  const int cap_a = ctas_per_sm ? ctas_per_sm : occ_rows;
  const int cap_e = ctas_per_sm ? ctas_per_sm : occ_upd;
  auto auto_rows = [&](int cap) {
    const int64_t per = (A->nrows + (int64_t)cap * nsm - 1) / ((int64_t)cap * nsm);
    return (int32_t)std::min<int64_t>(65536, std::max<int64_t>(PHASE_TPB, (per + 31) / 32 * 32));
  };
  if (Ra == 0) Ra = auto_rows(cap_a);
  if (Re == 0) Re = auto_rows(cap_e);
  GBS_TRY(build_table(A, Ra, cap_a, A->ta, st));
  // Rows in length order: for four and eight lanes a row on rows too uneven for the
  // sliced copy.  Shorter rows (fewer lanes) waste little, and even ones lose the
  // neighbours they share columns with: us a CG iteration in row order / so, rows
  // drawn from 2 to 16 entries (two lanes) 100k 23.0 / 23.4, 1M 80.0 / 79.9, from 2 to 120
  // (four) 100k 43.8 / 33.8, 300k 103 / 75, 2 to 40 1M 111 / 93; 3D 7-point 1M with one
  // lane 61 / 68, two 62 / 69, four 67 / 70.
  if ((kernel == 4 || kernel == 8) && (double)A->sell_nnz_rows > 1.2 * (double)A->nnz)
    GBS_TRY(build_row_orders(A, st));
  halo_window(A, Ra, A->ta);
  GBS_TRY(build_table(A, Re, cap_e, A->te, st));
  GBS_TRY(build_cta_order(A, st));
  A->Ra = Ra;
  A->Re = Re;
  A->lanes = kernel;
  A->ctas_per_sm = ctas_per_sm;
  A->plan_auto = all_auto;
  A->team_tuned = false;
  return GBS_OK;
}

}  // namespace gbs
