// COO -> CSR assembly on the device (Sec. 5: MatSetPreallocationCOO /
// MatSetValuesCOO), the Jacobi diagonal (Sec. 7), the FP32 copy used by the
// refined solve (Sec. 2, A7) and the adjoint scatter over the pattern.
//
// Symbolic stage, all on the GPU:
//   (patterns with a row of more than 4096 entries; the others: the row-bucketed
//   stage below)
//   1. keep flags (negative index -> ignored; out of range -> error) and an
//      exclusive scan, compaction into 64-bit keys i*ncols + j with the
//      original COO index as payload;
//   2. stable LSD radix sort of the keys (8-bit digits, as many passes as the
//      largest key needs): per-tile digit histograms, one scan of the
//      digit-major count table, then a stable scatter that ranks equal digits
//      with warp match/ballot in input order;
//   3. segment heads of the sorted keys and a scan -> nnz, jmap (segment
//      offsets), the unique keys, then col, the diagonal positions and
//      row_ptr (lower bound of r*ncols in the unique keys).
// The sorted payload is perm (sorted position -> original COO index): equal
// keys keep increasing COO index, which is what makes the numeric stage's
// in-order sum well defined.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "device_util.cuh"
#include "internal.cuh"

namespace gbs {

// ------------------------------------------------------------------ scan

constexpr int SCAN_T = 256, SCAN_IPT = 16, SCAN_TILE = SCAN_T * SCAN_IPT;

__device__ __forceinline__ uint32_t block_excl_scan_u32(uint32_t v, uint32_t *warp_tot,
                                                        uint32_t *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    uint32_t y = __shfl_up_sync(FULL_MASK, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) warp_tot[warp] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int w = 0; w < nw; ++w) {
      uint32_t t = warp_tot[w];
      warp_tot[w] = run;
      run += t;
    }
    *total = run;
  }
  __syncthreads();
  const uint32_t r = warp_tot[warp] + x - v;
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(SCAN_T) k_scan_reduce(const uint32_t *in, int64_t n,
                                                        uint32_t *tile_sums) {
  __shared__ uint32_t red[32];
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  uint32_t s = 0;
  for (int k = threadIdx.x; k < SCAN_TILE; k += SCAN_T) {
    const int64_t idx = base + k;
    if (idx < n) s += in[idx];
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(FULL_MASK, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < SCAN_T / 32; ++w) t += red[w];
    tile_sums[blockIdx.x] = t;
  }
}

// One CTA: exclusive scan of tile_sums in place; grand total to *total.
__global__ void __launch_bounds__(1024) k_scan_tiles(uint32_t *tile_sums, int64_t ntiles,
                                                     uint32_t *total) {
  __shared__ uint32_t warp_tot[32];
  __shared__ uint32_t chunk_tot;
  uint32_t carry = 0;
  for (int64_t c0 = 0; c0 < ntiles; c0 += blockDim.x) {
    const int64_t idx = c0 + threadIdx.x;
    const uint32_t v = idx < ntiles ? tile_sums[idx] : 0u;
    const uint32_t ex = block_excl_scan_u32(v, warp_tot, &chunk_tot);
    if (idx < ntiles) tile_sums[idx] = carry + ex;
    carry += chunk_tot;
    __syncthreads();
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

__device__ __forceinline__ int pad_idx(int k) { return k + (k >> 5); }

__global__ void __launch_bounds__(SCAN_T) k_scan_down(const uint32_t *in, int64_t n,
                                                      const uint32_t *tile_offs,
                                                      uint32_t *out) {
  __shared__ uint32_t tile[SCAN_TILE + SCAN_TILE / 32];
  __shared__ uint32_t warp_tot[32];
  __shared__ uint32_t tot;
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  for (int k = threadIdx.x; k < SCAN_TILE; k += SCAN_T) {
    const int64_t idx = base + k;
    tile[pad_idx(k)] = idx < n ? in[idx] : 0u;
  }
  __syncthreads();
  uint32_t loc[SCAN_IPT];
  uint32_t s = 0;
#pragma unroll
  for (int q = 0; q < SCAN_IPT; ++q) {
    loc[q] = s;
    s += tile[pad_idx(threadIdx.x * SCAN_IPT + q)];
  }
  const uint32_t ex = block_excl_scan_u32(s, warp_tot, &tot) + tile_offs[blockIdx.x];
#pragma unroll
  for (int q = 0; q < SCAN_IPT; ++q) tile[pad_idx(threadIdx.x * SCAN_IPT + q)] = ex + loc[q];
  __syncthreads();
  for (int k = threadIdx.x; k < SCAN_TILE; k += SCAN_T) {
    const int64_t idx = base + k;
    if (idx < n) out[idx] = tile[pad_idx(k)];
  }
}

// Exclusive scan of n uint32 (in may equal out), reduce-then-scan; the tile
// sums are scanned by one CTA when they fit one tile, else recursively.
// tmp: scan_tmp_words(n) words.  Grand total written to *total (device) when
// non-null.
int exclusive_scan(const uint32_t *in, uint32_t *out, int64_t n, uint32_t *tmp,
                          uint32_t *total, cudaStream_t s) {
  const int64_t ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
  if (ntiles == 0) {
    if (total) GBS_TRY_CUDA(cudaMemsetAsync(total, 0, sizeof(uint32_t), s));
    return GBS_OK;
  }
  k_scan_reduce<<<(unsigned)ntiles, SCAN_T, 0, s>>>(in, n, tmp);
  GBS_LAUNCHED(1);
  if (ntiles <= SCAN_TILE) {
    k_scan_tiles<<<1, 1024, 0, s>>>(tmp, ntiles, total);
    GBS_LAUNCHED(1);
  } else {
    GBS_TRY(exclusive_scan(tmp, tmp, ntiles, tmp + ntiles + 1, total, s));
  }
  k_scan_down<<<(unsigned)ntiles, SCAN_T, 0, s>>>(in, n, tmp, out);
  GBS_LAUNCHED(1);
  return GBS_OK;
}

int64_t scan_tmp_words(int64_t n) {
  int64_t w = 1, t = (n + SCAN_TILE - 1) / SCAN_TILE;
  for (;;) {
    w += t + 1;
    if (t <= SCAN_TILE) break;
    t = (t + SCAN_TILE - 1) / SCAN_TILE;
  }
  return w;
}

// ------------------------------------------------------------------ keep + compact

// Batched handles pass per-system COO offsets (coo_off, nsys+1) and row offsets
// (row_off, nsys+1): local indices are shifted to the block-diagonal numbering.
struct KeepArgs {
  const int32_t *i, *j;
  int64_t ncoo, nrows, ncols;
  const int64_t *coo_off, *row_off;  // null for a single system
  int32_t nsys;
};

__device__ __forceinline__ bool keep_entry(const KeepArgs &a, int64_t k, int32_t li, int32_t lj,
                                           int64_t &gi, int64_t &gj, bool &bad) {
  bad = false;
  if (li < 0 || lj < 0) return false;
  if (a.coo_off) {
    int lo = 0, hi = a.nsys;  // find s with coo_off[s] <= k < coo_off[s+1]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(a.coo_off + mid) <= k) lo = mid; else hi = mid;
    }
    const int64_t r0 = __ldg(a.row_off + lo), n = __ldg(a.row_off + lo + 1) - r0;
    if (li >= n || lj >= n) {
      bad = true;
      return false;
    }
    gi = r0 + li;
    gj = r0 + lj;
  } else {
    if (li >= a.nrows || lj >= a.ncols) {
      bad = true;
      return false;
    }
    gi = li;
    gj = lj;
  }
  return true;
}

__device__ __forceinline__ bool keep_entry(const KeepArgs &a, int64_t k, int64_t &gi,
                                           int64_t &gj, bool &bad) {
  return keep_entry(a, k, a.i[k], a.j[k], gi, gj, bad);
}

__global__ void k_keep_flags(KeepArgs a, uint32_t *flags, int32_t *err) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.ncoo;
       k += (int64_t)gridDim.x * blockDim.x) {
    int64_t gi, gj;
    bool bad;
    const bool keep = keep_entry(a, k, gi, gj, bad);
    if (bad) atomicExch(err, GBS_ERR_INDEX);
    flags[k] = keep ? 1u : 0u;
  }
}

__global__ void k_compact(KeepArgs a, const uint32_t *pos, uint64_t *keys, uint32_t *vals) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.ncoo;
       k += (int64_t)gridDim.x * blockDim.x) {
    int64_t gi, gj;
    bool bad;
    if (keep_entry(a, k, gi, gj, bad)) {
      const uint32_t d = pos[k];
      keys[d] = (uint64_t)gi * (uint64_t)a.ncols + (uint64_t)gj;
      vals[d] = (uint32_t)k;
    }
  }
}

// ------------------------------------------------------------------ radix sort

constexpr int RS_T = 256, RS_WARPS = RS_T / 32, RS_SLOTS = 16, RS_TILE = RS_T * RS_SLOTS;

__global__ void __launch_bounds__(RS_T) k_radix_hist(const uint64_t *keys, int64_t n,
                                                     int shift, uint32_t *counts,
                                                     int64_t ntiles) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * RS_TILE;
  const int lane = threadIdx.x & 31;
  for (int k = threadIdx.x; k < RS_TILE; k += RS_T) {
    const int64_t idx = base + k;
    const uint32_t d = idx < n ? (uint32_t)((keys[idx] >> shift) & 255u) : 256u;
    const unsigned peers = __match_any_sync(FULL_MASK, d);
    if (d < 256u && lane == __ffs(peers) - 1) atomicAdd(&h[d], (uint32_t)__popc(peers));
  }
  __syncthreads();
  counts[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter of one tile.  Warp w owns the contiguous items
// [base + w*SLOTS*32, base + (w+1)*SLOTS*32); it walks them slot by slot, lane
// order within a slot, which is the input order, so ranks of equal digits
// follow input order.  The tile is first reordered by digit in shared memory
// (stable), then written out by consecutive threads to consecutive addresses
// of each digit's run, so the stores coalesce instead of scattering single
// items over 256 runs.  vals_in == null means payload = item index.
struct RadixShared {
  uint64_t key[RS_TILE];
  uint32_t val[RS_TILE];
  uint32_t whist[RS_WARPS][256];  // per-warp digit counts, then per-warp offsets in the tile
  uint32_t toff[256];             // the tile's global offset of each digit
  uint32_t dbase[256];            // first position of each digit in the reordered tile
};

__global__ void __launch_bounds__(RS_T) k_radix_scatter(const uint64_t *keys_in,
                                                        const uint32_t *vals_in, int64_t n,
                                                        int shift, const uint32_t *offsets,
                                                        int64_t ntiles, uint64_t *keys_out,
                                                        uint32_t *vals_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  RadixShared &S = *reinterpret_cast<RadixShared *>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int w = 0; w < RS_WARPS; ++w) S.whist[w][threadIdx.x] = 0;
  S.toff[threadIdx.x] = offsets[(int64_t)threadIdx.x * ntiles + blockIdx.x];
  __syncthreads();
  const int64_t tile0 = (int64_t)blockIdx.x * RS_TILE;
  const int64_t base = tile0 + (int64_t)warp * RS_SLOTS * 32;
  const unsigned lt_mask = (1u << lane) - 1u;
  uint64_t key[RS_SLOTS];
  uint32_t val[RS_SLOTS], rank[RS_SLOTS];
#pragma unroll
  for (int sl = 0; sl < RS_SLOTS; ++sl) {
    const int64_t idx = base + sl * 32 + lane;
    const bool ok = idx < n;
    key[sl] = ok ? keys_in[idx] : 0ull;
    val[sl] = ok ? (vals_in ? vals_in[idx] : (uint32_t)idx) : 0u;
  }
#pragma unroll
  for (int sl = 0; sl < RS_SLOTS; ++sl) {
    const int64_t idx = base + sl * 32 + lane;
    const uint32_t d = idx < n ? (uint32_t)((key[sl] >> shift) & 255u) : 256u;
    const unsigned peers = __match_any_sync(FULL_MASK, d);
    const uint32_t before = d < 256u ? S.whist[warp][d] : 0u;
    rank[sl] = before + (uint32_t)__popc(peers & lt_mask);
    __syncwarp();
    if (d < 256u && lane == __ffs(peers) - 1) S.whist[warp][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {  // per digit: exclusive prefix over warps; the digit's total
    const int d = threadIdx.x;
    uint32_t run = 0;
    for (int w = 0; w < RS_WARPS; ++w) {
      const uint32_t c = S.whist[w][d];
      S.whist[w][d] = run;
      run += c;
    }
    S.dbase[d] = run;
  }
  __syncthreads();
  if (warp == 0) {  // exclusive scan of the 256 digit totals (8 per lane)
    uint32_t t[8], sum = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      t[k] = S.dbase[lane * 8 + k];
      sum += t[k];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(FULL_MASK, incl, off);
      if (lane >= off) incl += y;
    }
    uint32_t run = incl - sum;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      S.dbase[lane * 8 + k] = run;
      run += t[k];
    }
  }
  __syncthreads();
#pragma unroll
  for (int sl = 0; sl < RS_SLOTS; ++sl) {  // reorder the tile by digit (stable)
    const int64_t idx = base + sl * 32 + lane;
    if (idx < n) {
      const uint32_t d = (uint32_t)((key[sl] >> shift) & 255u);
      const uint32_t lp = S.dbase[d] + S.whist[warp][d] + rank[sl];
      S.key[lp] = key[sl];
      S.val[lp] = val[sl];
    }
  }
  __syncthreads();
  const int cnt = (int)(n - tile0 < RS_TILE ? n - tile0 : RS_TILE);
  for (int i = threadIdx.x; i < cnt; i += RS_T) {  // runs of a digit go to consecutive addresses
    const uint64_t k = S.key[i];
    const uint32_t d = (uint32_t)((k >> shift) & 255u);
    const uint32_t dst = S.toff[d] + (uint32_t)i - S.dbase[d];
    keys_out[dst] = k;
    vals_out[dst] = S.val[i];
  }
}

// The CTA's largest value to *out: one atomic a CTA, and none where it would
// not raise the maximum (an atomic per warp on one address, a million of them,
// took 0.6 ms).
__device__ __forceinline__ void block_atomic_max(int32_t m, int32_t *out) {
  __shared__ int32_t wm[32];
  m = (int32_t)__reduce_max_sync(FULL_MASK, (unsigned)m);
  if ((threadIdx.x & 31) == 0) wm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, wm[w]);
    if (m > *(volatile int32_t *)out) atomicMax(out, m);
  }
}

// The longest row.
__global__ void k_max_row(const int32_t *row_ptr, int64_t nrows, int32_t *out) {
  int32_t m = 0;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows;
       r += (int64_t)gridDim.x * blockDim.x)
    m = max(m, row_ptr[r + 1] - row_ptr[r]);
  block_atomic_max(m, out);
}

// ------------------------------------------------------------------ segments

__global__ void k_seg_flags(const uint64_t *keys, int64_t n, uint32_t *flags) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    flags[t] = (t == 0 || keys[t] != keys[t - 1]) ? 1u : 0u;
}

__global__ void k_seg_write(const uint64_t *keys, int64_t n, const uint32_t *flags,
                            const uint32_t *seg, uint64_t *ukey, int32_t *jmap) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    if (flags[t]) {
      const uint32_t s = seg[t];
      ukey[s] = keys[t];
      jmap[s] = (int32_t)t;
    }
  }
}

// Columns, diagonal positions and the largest |col - row| (capped at 2^30,
// into *span): the sliced copy stores 16-bit column offsets when it is
// below 2^15.
__global__ void k_csr_cols(const uint64_t *ukey, int64_t nnz, int64_t ncols, int32_t *col,
                           int32_t *diag_pos, int32_t *span) {
  int32_t m = 0;
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < nnz;
       s += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = ukey[s];
    const int64_t r = (int64_t)(k / (uint64_t)ncols), c = (int64_t)(k % (uint64_t)ncols);
    col[s] = (int32_t)c;
    if (r == c) diag_pos[r] = (int32_t)s;
    const int64_t d = c - r, ad = d < 0 ? -d : d;
    m = max(m, (int32_t)(ad > (1 << 30) ? (1 << 30) : ad));
  }
  block_atomic_max(m, span);
}

// row_ptr[r] = first unique key >= r * ncols, for r in [0, nrows].
__global__ void k_row_ptr(const uint64_t *ukey, int64_t nnz, int64_t ncols, int64_t nrows,
                          int32_t *row_ptr) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= nrows;
       r += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t target = (uint64_t)r * (uint64_t)ncols;
    int64_t lo = 0, hi = nnz;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (ukey[mid] < target) lo = mid + 1; else hi = mid;
    }
    row_ptr[r] = (int32_t)lo;
  }
}

static unsigned grid_for(int64_t n, int tpb) {
  int64_t g = (n + tpb - 1) / tpb;
  if (g < 1) g = 1;
  if (g > 1048576) g = 1048576;
  return (unsigned)g;
}

// A grid that keeps every SM of A's device busy and no more: for kernels that
// end in one atomic a CTA.
static unsigned wave_for(gbs_mat A, int64_t n, int tpb) {
  return std::min(grid_for(n, tpb), 8u * (unsigned)sm_count(A));
}

// Error exits of the symbolic stages: set status and jump to cleanup.
#define SYM_CUDA(call)                                                            \
  do {                                                                            \
    cudaError_t e_ = (call);                                                      \
    if (e_ != cudaSuccess) {                                                      \
      set_error("%s:%d %s: %s", __FILE__, __LINE__, #call, cudaGetErrorString(e_)); \
      status = (e_ == cudaErrorMemoryAllocation) ? GBS_ERR_ALLOC : GBS_ERR_CUDA;  \
      goto cleanup;                                                               \
    }                                                                             \
  } while (0)
#define SYM_TRY(call)                                                             \
  do {                                                                            \
    status = (call);                                                              \
    if (status != GBS_OK) goto cleanup;                                           \
  } while (0)

// ------------------------------------------------------------------ row-bucketed symbolic stage
//
// The symbolic stage for patterns whose rows hold at most ROW_SORT_CTA COO
// entries (finite-element, stencil and graph matrices): no global sort.
//   1. per-row counts of the kept entries (one atomic per run of equal rows on
//      a warp's lanes); the old count plus the lane's place in its run is the
//      entry's slot in its row, kept as 16 bits;
//   2. their exclusive scan -> each row's range of the kept entries;
//   3. every kept entry placed at its slot of its row's range as the 64-bit key
//      (j << 32) | k (the slots depend on the atomics' timing);
//   4. each row sorted by that key (register bitonic networks, four rows a
//      warp, up to ROW_SORT_WARP entries; a CTA's shared-memory one up to
//      ROW_SORT_CTA): the keys are distinct, so the result is the same on every run, and it
//      is the order of the radix path -- rows ascending, columns ascending,
//      equal (i, j) by increasing COO index; written out as perm and the
//      column with a head bit (first entry of its column), with each row's
//      count of distinct columns and the place of its diagonal among them;
//   5. the scan of those counts is row_ptr (and nnz); a pass over the sorted
//      entries writes col and jmap, one over the rows the diagonal positions.
// Traffic: about 40 bytes per kept entry, against about 140 for the 5-pass
// radix sort of 40-bit keys.  A longer row sends the pattern to the radix
// path.  Measured on the Q1 96^3 pattern (56.6M entries, 62 a row) and the
// 2D 1024^2 edges (8.4M, 8 a row), us, against one warp to a row, an atomic a
// warp for the largest |col - row| and match-aggregated atomics with one entry
// a thread in flight:
//   counts 240 / 79 -> 139 / 24, placement 314 / 80 -> 169 / 30, sorts 589 /
//   669 -> 410 / 80, emission 628 / 675 -> 144 / 28.
// The long rows' sort is held by the ALU (64-bit compares), the short rows' by
// the latency of its loads, the others by HBM and the stores' scatter.
constexpr int ROW_SORT_WARP = 64, ROW_SORT_CTA = 4096, ROW_SORT_TPB = 512;

// Counts the kept entries per row (and flags out-of-range indices); slot[k]
// is entry k's place in its row (rows of up to ROW_SORT_CTA entries need 13
// bits; a longer row leaves the pattern to the radix path).
// A warp takes 32 BUCKET_U consecutive entries at a time, all their loads in
// flight before the first use (one entry a thread kept 8 bytes a thread in
// flight: 1.6 TB/s).
constexpr int BUCKET_U = 4;
__global__ void k_row_count(KeepArgs a, uint32_t *cnt, uint16_t *__restrict__ slot, int32_t *err) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t base = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32 * BUCKET_U;
       base < a.ncoo; base += nw * 32 * BUCKET_U) {
    int32_t li[BUCKET_U], lj[BUCKET_U];
    uint32_t old[BUCKET_U];
    int first[BUCKET_U];
#pragma unroll
    for (int u = 0; u < BUCKET_U; ++u) {
      const int64_t k = base + 32 * u + lane;
      li[u] = k < a.ncoo ? __ldg(a.i + k) : -1;
      lj[u] = k < a.ncoo ? __ldg(a.j + k) : -1;
    }
#pragma unroll
    for (int u = 0; u < BUCKET_U; ++u) {
      int64_t gi = 0, gj = 0;
      bool bad = false;
      const bool keep = keep_entry(a, base + 32 * u + lane, li[u], lj[u], gi, gj, bad);
      if (bad) atomicExch(err, GBS_ERR_INDEX);
      const int32_t row = keep ? (int32_t)gi : -1;
      const int32_t before = __shfl_up_sync(FULL_MASK, row, 1);
      const bool head = keep && (lane == 0 || before != row);
      const unsigned heads = __ballot_sync(FULL_MASK, head), kept = __ballot_sync(FULL_MASK, keep);
      // the head of my run: the last one up to my lane
      first[u] = keep ? 31 - __clz(heads & (0xffffffffu >> (31 - lane))) : lane;
      old[u] = 0;
      if (head) {
        const unsigned ends = lane == 31 ? 0u : (heads | ~kept) >> (lane + 1);
        old[u] = atomicAdd(cnt + row, (uint32_t)(ends ? __ffs(ends) : 32 - lane));
      }
      li[u] = row;
    }
#pragma unroll
    for (int u = 0; u < BUCKET_U; ++u) {
      const uint32_t o = __shfl_sync(FULL_MASK, old[u], first[u]);
      if (li[u] >= 0) slot[base + 32 * u + lane] = (uint16_t)(o + (uint32_t)(lane - first[u]));
    }
  }
}

// Places every kept entry at its slot of its row as (j << 32) | k.
__global__ void k_row_place(KeepArgs a, const uint32_t *__restrict__ rstart,
                            const uint16_t *__restrict__ slot, uint64_t *__restrict__ keys) {
  const int64_t T = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k0 < a.ncoo;
       k0 += BUCKET_U * T) {
    int32_t li[BUCKET_U], lj[BUCKET_U];
    uint32_t at[BUCKET_U];
#pragma unroll
    for (int u = 0; u < BUCKET_U; ++u) {
      const int64_t k = k0 + u * T;
      li[u] = k < a.ncoo ? __ldg(a.i + k) : -1;
      lj[u] = k < a.ncoo ? __ldg(a.j + k) : -1;
      at[u] = k < a.ncoo ? __ldg(slot + k) : 0u;
    }
    uint64_t key[BUCKET_U];
    bool keep[BUCKET_U];
#pragma unroll
    for (int u = 0; u < BUCKET_U; ++u) {
      const int64_t k = k0 + u * T;
      int64_t gi = 0, gj = 0;
      bool bad;
      keep[u] = keep_entry(a, k, li[u], lj[u], gi, gj, bad);
      key[u] = ((uint64_t)(uint32_t)gj << 32) | (uint32_t)k;
      if (keep[u]) at[u] += __ldg(rstart + gi);
    }
#pragma unroll
    for (int u = 0; u < BUCKET_U; ++u)
      if (keep[u]) keys[at[u]] = key[u];
  }
}

// What a sorted row leaves: its distinct columns, the place of its diagonal
// among them (-1: none) and the largest |col - row|.
struct RowOut {
  int32_t *perm;
  uint32_t *jh;        // the sorted columns, bit 31: first entry of its column
  uint32_t *ucnt;      // distinct columns
  int32_t *dloc;       // the diagonal's place among them
  int32_t *span;
  int32_t *long_rows;  // rows for k_row_sort_cta, their count
  uint32_t *nlong;
};
constexpr uint32_t HEAD_BIT = 0x80000000u;

// |j - r| capped at 2^30.
__device__ __forceinline__ int32_t col_dist(uint32_t j, int64_t r) {
  const int64_t d = (int64_t)j - r, ad = d < 0 ? -d : d;
  return (int32_t)(ad > (1 << 30) ? (1 << 30) : ad);
}

constexpr int SORT_TPB = 256;

// Rows r .. r + 3, of at most 8 KPL entries each, on a warp: eight lanes a row,
// KPL keys a lane, a bitonic network whose elements are blocked (element KPL g
// + i is lane g's key i).  Keys of one lane compare in registers; with KPL = 8
// six of the network's 21 stages need shuffles, where two keys a lane on 32
// lanes shuffle in 15.  The sorted keys go through shared memory (x: 36 KPL
// words a warp, one word of padding in nine against bank conflicts), so that
// every lane writes out consecutive entries.
template <int KPL>
__device__ __forceinline__ int32_t sort_rows4(int64_t r, int64_t nrows,
                                              const uint32_t *__restrict__ rstart,
                                              const uint64_t *__restrict__ keys, uint64_t *x,
                                              const RowOut &o) {
  constexpr int N = 8 * KPL;
  const int lane = threadIdx.x & 31, g = lane & 7, l0 = lane & 24;
  const int64_t row = r + (lane >> 3);
  const uint32_t s0 = row < nrows ? __ldg(rstart + row) : 0u;
  const int len = row < nrows ? (int)(__ldg(rstart + row + 1) - s0) : 0;
  uint64_t a[KPL];
#pragma unroll
  for (int i = 0; i < KPL; ++i) a[i] = 8 * i + g < len ? __ldg(keys + s0 + 8 * i + g) : ~0ull;
#pragma unroll
  for (int k = 2; k <= N; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= KPL) {
        const bool asc = ((g * KPL) & k) == 0, low = (g & (j / KPL)) == 0;
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
          const uint64_t other = __shfl_xor_sync(FULL_MASK, a[i], j / KPL);
          a[i] = ((a[i] < other) == (low == asc)) ? a[i] : other;
        }
      } else {
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
          if ((i & j) == 0) {
            const bool asc = k < KPL ? (i & k) == 0 : ((g * KPL) & k) == 0;
            const uint64_t u = a[i], v = a[i | j];
            const bool swap = (u > v) == asc;
            a[i] = swap ? v : u;
            a[i | j] = swap ? u : v;
          }
        }
      }
    }
  }
  uint64_t *xr = x + (lane >> 3) * 9 * KPL;
  __syncwarp();
#pragma unroll
  for (int i = 0; i < KPL; ++i) {
    const int e = g * KPL + i;
    xr[e + (e >> 3)] = a[i];
  }
  __syncwarp();
  int u = 0, diag = -1;
  int32_t m = 0;
#pragma unroll
  for (int i = 0; i < KPL; ++i) {
    const int e = 8 * i + g;
    const uint64_t key = xr[e + i];
    const uint32_t j = (uint32_t)(key >> 32);
    const uint32_t before = e > 0 ? (uint32_t)(xr[e - 1 + ((e - 1) >> 3)] >> 32) : 0u;
    const bool in = e < len, head = in && (e == 0 || j != before);
    const unsigned hb = (__ballot_sync(FULL_MASK, head) >> l0) & 255u;
    const unsigned db = (__ballot_sync(FULL_MASK, head && (int64_t)j == row) >> l0) & 255u;
    if (db) diag = u + __popc(hb & (db - 1u));
    u += __popc(hb);
    if (in) {
      o.perm[s0 + e] = (int32_t)(uint32_t)key;
      o.jh[s0 + e] = j | (head ? HEAD_BIT : 0u);
      m = max(m, col_dist(j, row));
    }
  }
  if (g == 0 && row < nrows) {
    o.ucnt[row] = (uint32_t)u;
    o.dloc[row] = diag;
  }
  return m;
}

// Sorts the rows, four consecutive ones a warp at a time with the smallest
// network that holds the longest of them; MAXK (keys a lane: 1, 2, 4 or 8) is
// what the pattern's longest row needs, so that patterns of short rows run a
// kernel of few registers.  Rows of more than ROW_SORT_WARP entries (MAXK = 8)
// go to long_rows for k_row_sort_cta.
template <int MAXK>
__global__ void __launch_bounds__(SORT_TPB)
    k_row_sort(int64_t nrows, const uint32_t *__restrict__ rstart,
               const uint64_t *__restrict__ keys, RowOut o) {
  __shared__ uint64_t sx[SORT_TPB / 32][36 * MAXK];
  const int lane = threadIdx.x & 31;
  uint64_t *x = sx[threadIdx.x >> 5];
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int32_t m = 0;
  for (int64_t r = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4; r < nrows;
       r += 4 * nw) {
    if constexpr (MAXK == 1) {
      m = max(m, sort_rows4<1>(r, nrows, rstart, keys, x, o));
    } else {
      const uint32_t st = lane <= 4 && r + lane <= nrows ? __ldg(rstart + r + lane) : 0u;
      const uint32_t nxt = __shfl_down_sync(FULL_MASK, st, 1);
      const unsigned len = lane < 4 && r + lane < nrows ? nxt - st : 0u;
      int longest = (int)__reduce_max_sync(FULL_MASK, len);
      if (longest <= 8) {
        m = max(m, sort_rows4<1>(r, nrows, rstart, keys, x, o));
      } else if (longest <= 16) {
        m = max(m, sort_rows4<2>(r, nrows, rstart, keys, x, o));
      } else if constexpr (MAXK >= 4) {
        if (longest <= 32) {
          m = max(m, sort_rows4<4>(r, nrows, rstart, keys, x, o));
        } else if constexpr (MAXK >= 8) {
          if (longest <= ROW_SORT_WARP) {
            m = max(m, sort_rows4<8>(r, nrows, rstart, keys, x, o));
          } else {  // the rows that fit one at a time, the others later
            for (int q = 0; q < 4 && r + q < nrows; ++q) {
              const int l = (int)__shfl_sync(FULL_MASK, len, q);
              if (l <= ROW_SORT_WARP)
                m = max(m, sort_rows4<8>(r + q, r + q + 1, rstart, keys, x, o));
              else if (lane == 0)
                o.long_rows[atomicAdd(o.nlong, 1u)] = (int32_t)(r + q);
            }
          }
        }
      }
    }
  }
  block_atomic_max(m, o.span);
}

// The long rows (ROW_SORT_WARP < len <= ROW_SORT_CTA), one CTA each: a
// bitonic sort in shared memory, then as k_row_sort.
__global__ void __launch_bounds__(ROW_SORT_TPB)
    k_row_sort_cta(const uint32_t *__restrict__ rstart, const uint64_t *__restrict__ keys,
                   RowOut o) {
  __shared__ uint64_t sk[ROW_SORT_CTA];
  __shared__ int cnt_w[2][ROW_SORT_TPB / 32];
  __shared__ int diag;
  const uint32_t nl = *o.nlong;
  int32_t m = 0;
  for (uint32_t li = blockIdx.x; li < nl; li += gridDim.x) {
    const int32_t r = o.long_rows[li];
    const uint32_t s0 = rstart[r];
    const int len = (int)(rstart[r + 1] - s0);
    int n2 = 1;
    while (n2 < len) n2 <<= 1;
    if (threadIdx.x == 0) diag = -1;
    for (int q = threadIdx.x; q < n2; q += blockDim.x) sk[q] = q < len ? keys[s0 + q] : ~0ull;
    __syncthreads();
    for (int k = 2; k <= n2; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int q = threadIdx.x; q < n2; q += blockDim.x) {
          const int pq = q ^ j;
          if (pq > q) {
            const uint64_t x = sk[q], y = sk[pq];
            const bool asc = (q & k) == 0;
            if ((x > y) == asc) {
              sk[q] = y;
              sk[pq] = x;
            }
          }
        }
        __syncthreads();
      }
    auto is_head = [&](int q) { return q == 0 || (sk[q] >> 32) != (sk[q - 1] >> 32); };
    int u = 0;
    for (int q = threadIdx.x; q < len; q += blockDim.x) {
      const uint64_t x = sk[q];
      const uint32_t j = (uint32_t)(x >> 32);
      const bool head = is_head(q);
      o.perm[s0 + q] = (int32_t)(uint32_t)x;
      o.jh[s0 + q] = j | (head ? HEAD_BIT : 0u);
      if (head && (int64_t)j == r) diag = q;  // (one entry at most)
      u += head ? 1 : 0;
      m = max(m, col_dist(j, r));
    }
    __syncthreads();
    int before = 0;  // heads before the diagonal's
    const int dq = diag;
    for (int q = threadIdx.x; q < dq; q += blockDim.x) before += is_head(q) ? 1 : 0;
    u = (int)__reduce_add_sync(FULL_MASK, (unsigned)u);
    before = (int)__reduce_add_sync(FULL_MASK, (unsigned)before);
    if ((threadIdx.x & 31) == 0) {
      cnt_w[0][threadIdx.x >> 5] = u;
      cnt_w[1][threadIdx.x >> 5] = before;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int t = 0, d = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        t += cnt_w[0][w];
        d += cnt_w[1][w];
      }
      o.ucnt[r] = (uint32_t)t;
      o.dloc[r] = dq >= 0 ? d : -1;
    }
    __syncthreads();
  }
  block_atomic_max(m, o.span);
}

// col and jmap from the sorted entries: entry q that heads its column is the
// pattern's nonzero number (heads before q).  A CTA takes EMIT_TILE entries:
// the row of the first one (a binary search over rstart) gives the number of
// heads before that row, row_ptr; counting those between the row's start and
// the tile gives the tile's first number, a scan of the tile's flags the rest.
constexpr int EMIT_T = 256, EMIT_IPT = 8, EMIT_TILE = EMIT_T * EMIT_IPT;
__global__ void __launch_bounds__(EMIT_T)
    k_row_emit(int64_t nkept, int64_t nrows, const uint32_t *__restrict__ rstart,
               const uint32_t *__restrict__ jh, const int32_t *__restrict__ row_ptr,
               int32_t *__restrict__ jmap, int32_t *__restrict__ col) {
  __shared__ int s_row, s_extra;
  __shared__ uint32_t warp_tot[EMIT_T / 32];
  const int64_t t0 = (int64_t)blockIdx.x * EMIT_TILE;
  if (threadIdx.x < 32) {  // the last row with rstart[row] <= t0, 32 probes a step
    int64_t lo = 0, hi = nrows;  // rstart[lo] <= t0 < rstart[hi]
    while (hi - lo > 1) {
      const int64_t step = (hi - lo + 31) / 32;
      const int64_t at = min(lo + step * (int)(threadIdx.x + 1), hi);
      const unsigned le = __ballot_sync(FULL_MASK, at < hi && (int64_t)rstart[at] <= t0);
      const int k = __popc(le);  // (monotone: the first k probes)
      const int64_t nlo = lo + step * k;
      hi = min(nlo + step, hi);
      lo = nlo;
    }
    if (threadIdx.x == 0) {
      s_row = (int)lo;
      s_extra = 0;
    }
  }
  __syncthreads();
  int extra = 0;
  for (int64_t q = rstart[s_row] + threadIdx.x; q < t0; q += EMIT_T) extra += (int)(jh[q] >> 31);
  extra = (int)__reduce_add_sync(FULL_MASK, (unsigned)extra);
  if ((threadIdx.x & 31) == 0 && extra) atomicAdd(&s_extra, extra);
  __syncthreads();
  uint32_t base = (uint32_t)(row_ptr[s_row] + s_extra);
  // EMIT_IPT rounds of one entry a thread: coalesced, and in order
  uint32_t j[EMIT_IPT];
#pragma unroll
  for (int i = 0; i < EMIT_IPT; ++i) {
    const int64_t q = t0 + i * EMIT_T + threadIdx.x;
    j[i] = q < nkept ? __ldg(jh + q) : 0u;
  }
#pragma unroll
  for (int i = 0; i < EMIT_IPT; ++i) {
    const int64_t q = t0 + i * EMIT_T + threadIdx.x;
    const unsigned hb = __ballot_sync(FULL_MASK, (j[i] & HEAD_BIT) != 0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_tot[warp] = (uint32_t)__popc(hb);
    __syncthreads();
    uint32_t below = 0, all = 0;
#pragma unroll
    for (int w = 0; w < EMIT_T / 32; ++w) {
      const uint32_t c = warp_tot[w];
      below += w < warp ? c : 0u;
      all += c;
    }
    if (j[i] & HEAD_BIT) {
      const uint32_t u = base + below + (uint32_t)__popc(hb & ((1u << lane) - 1u));
      jmap[u] = (int32_t)q;
      col[u] = (int32_t)(j[i] & ~HEAD_BIT);
    }
    base += all;
    __syncthreads();
  }
}

// diag_pos[r] from the diagonal's place in its row.
__global__ void k_row_diag(int64_t nrows, const int32_t *__restrict__ row_ptr,
                           const int32_t *__restrict__ dloc, int32_t *__restrict__ diag_pos) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t d = dloc[r];
    diag_pos[r] = d < 0 ? -1 : row_ptr[r] + d;
  }
}

// Symbolic stage, enqueued on s: its buffers are ready on s (the caller
// synchronises before other streams may use them).  coo_off_h (host, nsys+1)
// is non-null for batched handles;
// A->row_off_h, nrows, ncols, ncoo, nsys are set by the caller.  The
// row-bucketed path runs unless a row holds more than ROW_SORT_CTA entries.
static int symbolic_radix(gbs_mat A, const int32_t *i, const int32_t *j,
                          const int64_t *coo_off_h, cudaStream_t s);
static int symbolic_rows(gbs_mat A, const int32_t *i, const int32_t *j,
                         const int64_t *coo_off_h, cudaStream_t s, bool *done);

int symbolic(gbs_mat A, const int32_t *i, const int32_t *j, const int64_t *coo_off_h,
             cudaStream_t s) {
  // more entries than the rows could hold at ROW_SORT_CTA each: unless many are
  // ignored some row is longer, and counting so few rows would only serialise
  // on their counters (1M entries of 10 rows: 420 us with the counts, 203 without)
  if (A->ncoo > (int64_t)ROW_SORT_CTA * A->nrows) return symbolic_radix(A, i, j, coo_off_h, s);
  bool done = false;
  const int st = symbolic_rows(A, i, j, coo_off_h, s, &done);
  if (st != GBS_OK || done) return st;
  return symbolic_radix(A, i, j, coo_off_h, s);
}

static int symbolic_rows(gbs_mat A, const int32_t *i, const int32_t *j,
                         const int64_t *coo_off_h, cudaStream_t s, bool *done) {
  *done = false;
  const int64_t ncoo = A->ncoo, n = A->nrows;
  KeepArgs ka{i, j, ncoo, A->nrows, A->ncols, nullptr, nullptr, A->nsys};
  int64_t *d_off = nullptr;
  uint32_t *cnt = nullptr, *rstart = nullptr, *scan_tmp = nullptr, *jh = nullptr;
  uint64_t *keys = nullptr;
  uint16_t *slot = nullptr;
  int32_t *perm = nullptr, *long_rows = nullptr, *dloc = nullptr;
  int status = GBS_OK;
  struct Ctl {
    uint32_t nkept, nnz;
    int32_t err, maxcnt, span;
    uint32_t nlong;
  } hc{};
  Ctl *dctl = nullptr;
  const int64_t n1 = std::max<int64_t>(n, 1);

  {
    SYM_TRY(dev_alloc(&dctl, 1, s));
    SYM_CUDA(cudaMemsetAsync(dctl, 0, sizeof(Ctl), s));
    if (coo_off_h) {
      SYM_TRY(dev_alloc(&d_off, 2 * (A->nsys + 1), s));
      SYM_CUDA(cudaMemcpyAsync(d_off, coo_off_h, sizeof(int64_t) * (A->nsys + 1),
                               cudaMemcpyHostToDevice, s));
      SYM_CUDA(cudaMemcpyAsync(d_off + A->nsys + 1, A->row_off_h.data(),
                               sizeof(int64_t) * (A->nsys + 1), cudaMemcpyHostToDevice, s));
      ka.coo_off = d_off;
      ka.row_off = d_off + A->nsys + 1;
    }
    // 1-2. counts per row and slots, the counts' scan (total: nkept), the
    // largest count
    SYM_TRY(dev_alloc(&cnt, n1 + 1, s));
    SYM_TRY(dev_alloc(&rstart, n1 + 1, s));
    SYM_TRY(dev_alloc(&slot, std::max<int64_t>(ncoo, 1), s));
    SYM_TRY(dev_alloc(&scan_tmp, scan_tmp_words(n1 + 1), s));
    SYM_CUDA(cudaMemsetAsync(cnt, 0, sizeof(uint32_t) * (n1 + 1), s));
    if (ncoo > 0) {
      k_row_count<<<grid_for(ncoo, 256 * BUCKET_U), 256, 0, s>>>(ka, cnt, slot, &dctl->err);
      GBS_LAUNCHED(1);
    }
    SYM_TRY(exclusive_scan(cnt, rstart, n + 1, scan_tmp, &dctl->nkept, s));
    if (n > 0) {
      k_max_row<<<wave_for(A, n, 256), 256, 0, s>>>(reinterpret_cast<const int32_t *>(rstart), n,
                                                 &dctl->maxcnt);
      GBS_LAUNCHED(1);
    }
    SYM_CUDA(cudaMemcpyAsync(&hc, dctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    SYM_CUDA(cudaStreamSynchronize(s));
    if (hc.err != 0) {
      set_error("mat_create_coo: a kept COO index is out of range");
      status = GBS_ERR_INDEX;
      goto cleanup;
    }
    if (hc.maxcnt > ROW_SORT_CTA) goto cleanup;  // the radix path takes it
    const int64_t nkept = hc.nkept;
    const int64_t nk = std::max<int64_t>(nkept, 1);
    // 3. placement
    SYM_TRY(dev_alloc(&keys, nk, s));
    SYM_TRY(dev_alloc(&perm, nk, s));
    SYM_TRY(dev_alloc(&jh, nk, s));
    SYM_TRY(dev_alloc(&dloc, n1, s));
    if (hc.maxcnt > ROW_SORT_WARP) SYM_TRY(dev_alloc(&long_rows, n1, s));
    if (nkept > 0) {
      k_row_place<<<grid_for(ncoo, 256 * BUCKET_U), 256, 0, s>>>(ka, rstart, slot, keys);
      GBS_LAUNCHED(1);
    }
    // 4. per-row sorts, distinct columns (over cnt, whose last word the scan needs 0)
    SYM_CUDA(cudaMemsetAsync(cnt + n, 0, sizeof(uint32_t), s));
    if (n > 0) {
      const RowOut o{perm, jh, cnt, dloc, &dctl->span, long_rows, &dctl->nlong};
      const auto sort = hc.maxcnt <= 8    ? k_row_sort<1>
                        : hc.maxcnt <= 16 ? k_row_sort<2>
                        : hc.maxcnt <= 32 ? k_row_sort<4>
                                          : k_row_sort<8>;
      sort<<<grid_for((n + 3) / 4 * 32, SORT_TPB), SORT_TPB, 0, s>>>(n, rstart, keys, o);
      GBS_LAUNCHED(1);
      if (hc.maxcnt > ROW_SORT_WARP) {
        k_row_sort_cta<<<1024, ROW_SORT_TPB, 0, s>>>(rstart, keys, o);
        GBS_LAUNCHED(1);
      }
    }
    // 5. row_ptr, nnz; then col, jmap, diagonal positions
    SYM_TRY(dev_alloc(&A->row_ptr, n + 1, s));
    SYM_TRY(exclusive_scan(cnt, reinterpret_cast<uint32_t *>(A->row_ptr), n + 1, scan_tmp,
                           &dctl->nnz, s));
    SYM_CUDA(cudaMemcpyAsync(&hc, dctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    SYM_CUDA(cudaStreamSynchronize(s));
    const int64_t nnz = hc.nnz;
    A->nkept = nkept;
    A->nnz = nnz;
    A->col_span = hc.span;
    const int64_t nz1 = std::max<int64_t>(nnz, 1);
    SYM_TRY(dev_alloc(&A->jmap, nnz + 1, s));
    SYM_TRY(dev_alloc(&A->col, nz1, s));
    SYM_TRY(dev_alloc(&A->val, nz1, s));
    SYM_TRY(dev_alloc(&A->diag_pos, n1, s));
    SYM_TRY(dev_alloc(&A->dinv, n1, s));
    SYM_CUDA(cudaMemsetAsync(A->val, 0, sizeof(double) * nz1, s));
    SYM_CUDA(cudaMemsetAsync(A->dinv, 0, sizeof(double) * n1, s));
    // (nkept, the last offset of jmap, is in the control words)
    SYM_CUDA(cudaMemcpyAsync(A->jmap + nnz, &dctl->nkept, sizeof(int32_t),
                             cudaMemcpyDeviceToDevice, s));
    if (nkept > 0) {
      k_row_emit<<<(unsigned)((nkept + EMIT_TILE - 1) / EMIT_TILE), EMIT_T, 0, s>>>(
          nkept, n, rstart, jh, A->row_ptr, A->jmap, A->col);
      GBS_LAUNCHED(1);
    }
    if (n > 0) {
      k_row_diag<<<grid_for(n, 256), 256, 0, s>>>(n, A->row_ptr, dloc, A->diag_pos);
      GBS_LAUNCHED(1);
    }
    A->perm = perm;
    perm = nullptr;
    *done = true;
  }

cleanup:
  for (void *p : {(void *)dctl, (void *)d_off, (void *)cnt, (void *)rstart, (void *)scan_tmp,
                  (void *)slot, (void *)jh, (void *)dloc, (void *)keys, (void *)perm,
                  (void *)long_rows})
    dev_free(p, s);
  if (status != GBS_OK) cudaStreamSynchronize(s);
  return status;
}

// The radix path: keep flags and compaction, a stable LSD radix sort of the
// 64-bit keys i * ncols + j, segment heads.
static int symbolic_radix(gbs_mat A, const int32_t *i, const int32_t *j,
                          const int64_t *coo_off_h, cudaStream_t s) {
  const int64_t ncoo = A->ncoo;
  KeepArgs ka{i, j, ncoo, A->nrows, A->ncols, nullptr, nullptr, A->nsys};
  int64_t *d_off = nullptr;
  uint32_t *flags = nullptr, *scan_tmp = nullptr, *dsc = nullptr;
  uint64_t *kA = nullptr, *kB = nullptr, *ukey = nullptr;
  uint32_t *vA = nullptr, *vB = nullptr, *counts = nullptr;
  int status = GBS_OK;
  // host mirrors read back after each synchronisation
  struct Ctl {
    uint32_t nkept, nnz;
    int32_t err, span;
  } hc{};
  Ctl *dctl = nullptr;


  {
    SYM_TRY(dev_alloc(&dctl, 1, s));
    SYM_CUDA(cudaMemsetAsync(dctl, 0, sizeof(Ctl), s));
    if (coo_off_h) {
      SYM_TRY(dev_alloc(&d_off, 2 * (A->nsys + 1), s));
      SYM_CUDA(cudaMemcpyAsync(d_off, coo_off_h, sizeof(int64_t) * (A->nsys + 1),
                               cudaMemcpyHostToDevice, s));
      SYM_CUDA(cudaMemcpyAsync(d_off + A->nsys + 1, A->row_off_h.data(),
                               sizeof(int64_t) * (A->nsys + 1), cudaMemcpyHostToDevice, s));
      ka.coo_off = d_off;
      ka.row_off = d_off + A->nsys + 1;
    }
    const int64_t nflag = std::max<int64_t>(ncoo, 1);
    SYM_TRY(dev_alloc(&flags, nflag, s));
    SYM_TRY(dev_alloc(&dsc, nflag, s));
    SYM_TRY(dev_alloc(&scan_tmp, scan_tmp_words(nflag), s));

    // 1. keep flags, positions, nkept
    if (ncoo > 0) {
      k_keep_flags<<<grid_for(ncoo, 256), 256, 0, s>>>(ka, flags, &dctl->err);
      GBS_LAUNCHED(1);
    }
    SYM_TRY(exclusive_scan(flags, dsc, ncoo, scan_tmp, &dctl->nkept, s));
    SYM_CUDA(cudaMemcpyAsync(&hc, dctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    SYM_CUDA(cudaStreamSynchronize(s));
    if (hc.err != 0) {
      set_error("mat_create_coo: a kept COO index is out of range");
      status = GBS_ERR_INDEX;
      goto cleanup;
    }
    const int64_t nkept = hc.nkept;
    A->nkept = nkept;
    const int64_t nk = std::max<int64_t>(nkept, 1);
    SYM_TRY(dev_alloc(&kA, nk, s));
    SYM_TRY(dev_alloc(&kB, nk, s));
    SYM_TRY(dev_alloc(&vA, nk, s));
    SYM_TRY(dev_alloc(&vB, nk, s));  // becomes perm
    if (ncoo > 0) {
      k_compact<<<grid_for(ncoo, 256), 256, 0, s>>>(ka, dsc, kA, vA);
      GBS_LAUNCHED(1);
    }

    // 2. stable LSD radix sort (the scatter stages a tile in ~58 KB of shared memory)
    {
      static bool smem_opt_in = false;
      if (!smem_opt_in) {
        SYM_CUDA(cudaFuncSetAttribute(k_radix_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(RadixShared)));
        smem_opt_in = true;
      }
    }
    const uint64_t maxkey = (uint64_t)A->nrows * (uint64_t)A->ncols;
    int bits = 0;
    while (bits < 64 && (maxkey > 1) && ((maxkey - 1) >> bits) != 0) ++bits;
    const int passes = (bits + 7) / 8;
    const int64_t ntiles = (nkept + RS_TILE - 1) / RS_TILE;
    if (ntiles > 0 && passes > 0) {
      const int64_t ncount = 256 * ntiles;
      SYM_TRY(dev_alloc(&counts, ncount, s));
      uint32_t *ctmp = nullptr;
      SYM_TRY(dev_alloc(&ctmp, scan_tmp_words(ncount), s));
      uint64_t *kin = kA, *kout = kB;
      uint32_t *vin = vA, *vout = vB;
      for (int pass = 0; pass < passes; ++pass) {
        const int shift = 8 * pass;
        k_radix_hist<<<(unsigned)ntiles, RS_T, 0, s>>>(kin, nkept, shift, counts, ntiles);
        GBS_LAUNCHED(1);
        status = exclusive_scan(counts, counts, ncount, ctmp, nullptr, s);
        if (status != GBS_OK) {
          dev_free(ctmp, s);
          goto cleanup;
        }
        k_radix_scatter<<<(unsigned)ntiles, RS_T, sizeof(RadixShared), s>>>(
            kin, vin, nkept, shift, counts, ntiles, kout, vout);
        GBS_LAUNCHED(1);
        std::swap(kin, kout);
        std::swap(vin, vout);
      }
      dev_free(ctmp, s);
      // sorted data is in kin / vin; make kA / vB hold it
      if (kin != kA) std::swap(kA, kB);
      if (vin != vB) {
        // vin == vA: copy into vB (the buffer that becomes perm)
        SYM_CUDA(cudaMemcpyAsync(vB, vA, sizeof(uint32_t) * nkept, cudaMemcpyDeviceToDevice, s));
      }
    } else if (nkept > 0) {
      SYM_CUDA(cudaMemcpyAsync(vB, vA, sizeof(uint32_t) * nkept, cudaMemcpyDeviceToDevice, s));
    }

    // 3. segments
    if (nkept > 0) {
      k_seg_flags<<<grid_for(nkept, 256), 256, 0, s>>>(kA, nkept, flags);
      GBS_LAUNCHED(1);
    }
    SYM_TRY(exclusive_scan(flags, dsc, nkept, scan_tmp, &dctl->nnz, s));
    SYM_CUDA(cudaMemcpyAsync(&hc, dctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    SYM_CUDA(cudaStreamSynchronize(s));
    const int64_t nnz = hc.nnz;
    A->nnz = nnz;
    const int64_t nz1 = std::max<int64_t>(nnz, 1);
    SYM_TRY(dev_alloc(&A->jmap, nnz + 1, s));
    SYM_TRY(dev_alloc(&A->col, nz1, s));
    SYM_TRY(dev_alloc(&A->val, nz1, s));
    SYM_TRY(dev_alloc(&A->row_ptr, A->nrows + 1, s));
    SYM_TRY(dev_alloc(&A->diag_pos, std::max<int64_t>(A->nrows, 1), s));
    SYM_TRY(dev_alloc(&A->dinv, std::max<int64_t>(A->nrows, 1), s));
    SYM_CUDA(cudaMemsetAsync(A->val, 0, sizeof(double) * nz1, s));
    SYM_CUDA(cudaMemsetAsync(A->diag_pos, 0xff, sizeof(int32_t) * std::max<int64_t>(A->nrows, 1), s));
    SYM_CUDA(cudaMemsetAsync(A->dinv, 0, sizeof(double) * std::max<int64_t>(A->nrows, 1), s));
    SYM_TRY(dev_alloc(&ukey, nz1, s));
    A->perm = (int32_t *)vB;
    vB = nullptr;
    {
      const int32_t nk32 = (int32_t)nkept;
      SYM_CUDA(cudaMemcpyAsync(A->jmap + nnz, &nk32, sizeof(int32_t), cudaMemcpyHostToDevice, s));
    }
    if (nkept > 0) {
      k_seg_write<<<grid_for(nkept, 256), 256, 0, s>>>(kA, nkept, flags, dsc, ukey, A->jmap);
      GBS_LAUNCHED(1);
    }
    if (nnz > 0) {
      k_csr_cols<<<wave_for(A, nnz, 256), 256, 0, s>>>(ukey, nnz, A->ncols, A->col, A->diag_pos,
                                                    &dctl->span);
      GBS_LAUNCHED(1);
    }
    k_row_ptr<<<grid_for(A->nrows + 1, 256), 256, 0, s>>>(ukey, nnz, A->ncols, A->nrows,
                                                          A->row_ptr);
    GBS_LAUNCHED(1);
    SYM_CUDA(cudaMemcpyAsync(&hc, dctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    SYM_CUDA(cudaStreamSynchronize(s));
    A->col_span = hc.span;
  }

cleanup:
  for (void *p : {(void *)dctl, (void *)d_off, (void *)flags, (void *)dsc, (void *)scan_tmp,
                  (void *)kA, (void *)kB, (void *)vA, (void *)counts, (void *)ukey, (void *)vB})
    dev_free(p, s);
  cudaStreamSynchronize(s);
  return status;
}

// ------------------------------------------------------------------ numeric

// a_p = v[perm[jmap[p]]] + v[perm[jmap[p]+1]] + ... in increasing COO index
// order (Sec. 5: each nonzero is accumulated by one thread, no atomics).
//
// A CTA takes a tile of consecutive nonzeros in three steps.
//   1. Their COO values, contiguous in sorted order, into shared memory: perm
//      read coalesced, v gathered, every load independent of the others.  (One
//      thread per nonzero walking its own segment had two dependent loads a
//      term and at most eight of them in flight.)
//   2. The sums, from shared memory, in order of segment length: a warp issues
//      each FP64 add for all its lanes, and with consecutive nonzeros on
//      consecutive lanes nearly every warp of the Q1 matrix (segments of 1, 2, 4
//      and 8 terms) would run 7 add steps for 1.3 on average -- the FP64 pipe
//      held the kernel; a counting sort over NUM_CLASSES length classes puts
//      segments of about one length on a warp.
//   3. The results in nonzero order, coalesced.
// The lane a nonzero lands on depends on its class's ballots; its sum does not.
//
// SLICES: the tile is a few whole slices of the sliced copy, whose values and
// the rows' D^-1 are written from the same shared sums -- otherwise two more
// kernels, the fill reading every value again.
// What is left: shared-memory wavefronts (L1 data pipe 70% busy, half of the
// loads' wavefronts bank conflicts of the segment sums), 61% of the issue
// slots, HBM at 41%.  Measured, us, values + fill + D^-1 in three kernels ->
// here: Q1 96^3 346 + 94 + 22 -> 311, 2D 1024^2 edges 63 + 15 + 14 -> 72;
// k_coo_numeric on a graph of 300k rows 119 -> 74.
constexpr int NUM_TPB = 256, NUM_CLASSES = 5, NUM_BATCH = 4;
constexpr int NUM_NZ = 1024;   // nonzeros of a tile, at most
constexpr int NUM_E = 3072;    // COO entries of a tile that shared memory holds
constexpr int NUM_TILE = 512;  // nonzeros of a tile that is not cut by slices, at most
constexpr int NUM_SLICES = 8;  // slices of a tile, at most
constexpr int NUM_CTAS = 6;    // CTAs an SM (40 registers a thread)

__device__ __forceinline__ int length_class(int32_t len) {
  return len <= 1 ? 0 : (len == 2 ? 1 : (len <= 4 ? 2 : (len <= 8 ? 3 : 4)));
}

struct NumShared {  // in dynamic shared memory: as large as the launch's tiles
  double *v;       // COO values in sorted order
  double *sum;     // the nonzeros' sums
  uint16_t *j;     // segment starts in v
  int16_t *order;  // nonzeros by length class
};
__host__ __device__ constexpr size_t num_shared(int e, int nz) {  // bytes for e entries, nz nonzeros
  return 8 * (size_t)e + 8 * (size_t)nz + 2 * (((size_t)nz + 4) & ~(size_t)3) + 2 * (size_t)nz;
}
__device__ __forceinline__ NumShared num_carve(unsigned char *m, int e, int nz) {
  NumShared sh;
  sh.v = reinterpret_cast<double *>(m);
  sh.sum = sh.v + e;
  sh.j = reinterpret_cast<uint16_t *>(sh.sum + nz);
  sh.order = reinterpret_cast<int16_t *>(sh.j + ((nz + 4) & ~3));
  return sh;
}

// The sums of nonzeros [t0, t0 + nt) into sh.sum (ADD: with the old values).
// e_cap: the COO entries that sh.v holds.
__device__ __forceinline__ void numeric_tile(const NumShared &sh, int e_cap, int64_t t0, int nt,
                                             const int32_t *__restrict__ jmap,
                                             const int32_t *__restrict__ perm,
                                             const double *__restrict__ v, int mode,
                                             const double *val) {
  const int tid = (int)threadIdx.x;
  const int32_t e0 = __ldg(jmap + t0);
  const int ne = __ldg(jmap + t0 + nt) - e0;
  if (ne > e_cap) {  // long segments: one thread a nonzero, straight from memory
    for (int i = tid; i < nt; i += NUM_TPB) {
      int32_t t = __ldg(jmap + t0 + i);
      const int32_t e = __ldg(jmap + t0 + i + 1);
      double x = __ldg(v + __ldg(perm + t));
      ++t;
      while (t < e) {
        double y[NUM_BATCH];
#pragma unroll
        for (int u = 0; u < NUM_BATCH; ++u) y[u] = t + u < e ? __ldg(v + __ldg(perm + t + u)) : 0.0;
#pragma unroll
        for (int u = 0; u < NUM_BATCH; ++u)
          if (t + u < e) x = __dadd_rn(x, y[u]);
        t += NUM_BATCH;
      }
      sh.sum[i] = mode == GBS_ADD ? __dadd_rn(val[t0 + i], x) : x;
    }
    return;
  }
  __shared__ int32_t s_cnt[NUM_CLASSES][NUM_NZ / 32];  // per class and 32 nonzeros
  __shared__ int32_t s_base[NUM_CLASSES];
  for (int i = tid; i <= nt; i += NUM_TPB) sh.j[i] = (uint16_t)(__ldg(jmap + t0 + i) - e0);
  // the gathers run on while the classes are counted
  const uint32_t vs = (uint32_t)__cvta_generic_to_shared(sh.v);
  for (int e = tid; e < ne; e += 4 * NUM_TPB) {
    int32_t k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) k[u] = e + u * NUM_TPB < ne ? __ldg(perm + e0 + e + u * NUM_TPB) : 0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (e + u * NUM_TPB < ne)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(vs + 8u * (e + u * NUM_TPB)),
                     "l"(v + k[u])
                     : "memory");
  }
  __syncthreads();  // segment starts
  // places by length class: warp counts, their prefix sums, ranks by ballot
  const int lane = tid & 31, groups = (nt + 31) >> 5;
  for (int g = tid >> 5; g < groups; g += NUM_TPB / 32) {
    const int i = 32 * g + lane;
    const int c = i < nt ? length_class((int)sh.j[i + 1] - (int)sh.j[i]) : -1;
#pragma unroll
    for (int q = 0; q < NUM_CLASSES; ++q) {
      const unsigned m = __ballot_sync(FULL_MASK, c == q);
      if (lane == q) s_cnt[q][g] = __popc(m);
    }
  }
  __syncthreads();
  if (tid < 32 * NUM_CLASSES) {  // warp q: exclusive sums of class q's counts
    const int q = tid >> 5;
    const int n = lane < groups ? s_cnt[q][lane] : 0;
    int incl = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(FULL_MASK, incl, d);
      if (lane >= d) incl += y;
    }
    if (lane < groups) s_cnt[q][lane] = incl - n;
    if (lane == 31) s_base[q] = incl;
  }
  __syncthreads();
  for (int g = tid >> 5; g < groups; g += NUM_TPB / 32) {
    const int i = 32 * g + lane;
    const int c = i < nt ? length_class((int)sh.j[i + 1] - (int)sh.j[i]) : -1;
    unsigned mine = 0;
    int base = 0;
#pragma unroll
    for (int q = 0; q < NUM_CLASSES; ++q) {
      const unsigned m = __ballot_sync(FULL_MASK, c == q);
      if (c == q) mine = m;
      if (q < c) base += s_base[q];
    }
    if (c >= 0) sh.order[base + s_cnt[c][g] + __popc(mine & ((1u << lane) - 1u))] = (int16_t)i;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  for (int p = tid; p < nt; p += NUM_TPB) {
    const int i = sh.order[p];
    const int e = sh.j[i + 1];
    int t = sh.j[i];
    double x = sh.v[t];
    for (++t; t < e; ++t) x = __dadd_rn(x, sh.v[t]);  // in increasing COO index: plain adds
    sh.sum[i] = mode == GBS_ADD ? __dadd_rn(val[t0 + i], x) : x;
  }
}

// Tiles of `tile` nonzeros; the values only.
__global__ void __launch_bounds__(NUM_TPB, NUM_CTAS)
    k_coo_numeric(int64_t nnz, int32_t tile, const int32_t *__restrict__ jmap,
                  const int32_t *__restrict__ perm, const double *__restrict__ v, int mode,
                  double *__restrict__ val) {
  extern __shared__ __align__(16) unsigned char num_smem[];
  const NumShared sh = num_carve(num_smem, NUM_E, NUM_TILE);
  for (int64_t t0 = (int64_t)blockIdx.x * tile; t0 < nnz; t0 += (int64_t)gridDim.x * tile) {
    const int nt = nnz - t0 < tile ? (int)(nnz - t0) : tile;
    numeric_tile(sh, NUM_E, t0, nt, jmap, perm, v, mode, val);
    __syncthreads();
    for (int i = threadIdx.x; i < nt; i += NUM_TPB) val[t0 + i] = sh.sum[i];
    __syncthreads();  // the shared arrays are reused by the next tile
  }
}

// Tiles of per slices (at most NUM_NZ nonzeros): the CSR values, the sliced
// copy's values (k_sell_fill's) and D^-1 (k_jacobi's).
__global__ void __launch_bounds__(NUM_TPB, NUM_CTAS)
    k_numeric_slices(int64_t nslices, int32_t per, int32_t e_cap, int32_t nz_cap,
                     const int32_t *__restrict__ srow0,
                     const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ jmap,
                     const int32_t *__restrict__ perm, const double *__restrict__ v, int mode,
                     double *__restrict__ val, const int32_t *__restrict__ diag_pos,
                     double *__restrict__ dinv, const int32_t *__restrict__ sptr,
                     const uint32_t *__restrict__ mask, double *__restrict__ sval) {
  extern __shared__ __align__(16) unsigned char num_smem[];
  const NumShared sh = num_carve(num_smem, e_cap, nz_cap);
  __shared__ int32_t s_rs[32 * NUM_SLICES + 1];  // the rows' first nonzeros, from t0
  __shared__ uint32_t s_mk[32 * NUM_SLICES];     // patterns: the rows' masks
  const int tid = (int)threadIdx.x;
  const int64_t s0 = (int64_t)blockIdx.x * per;
  const int ns = nslices - s0 < per ? (int)(nslices - s0) : per;
  const int32_t r0 = __ldg(srow0 + s0), nr = __ldg(srow0 + s0 + ns) - r0;
  const int32_t t0 = __ldg(row_ptr + r0);
  const int nt = __ldg(row_ptr + r0 + nr) - t0;
  for (int i = tid; i <= nr; i += NUM_TPB) s_rs[i] = __ldg(row_ptr + r0 + i) - t0;
  if (mask)
    for (int i = tid; i < 32 * ns; i += NUM_TPB) s_mk[i] = __ldg(mask + 32 * s0 + i);
  if (nt > 0) numeric_tile(sh, e_cap, t0, nt, jmap, perm, v, mode, val);
  __syncthreads();
  for (int i = tid; i < nt; i += NUM_TPB) val[t0 + i] = sh.sum[i];
  for (int i = tid; i < nr; i += NUM_TPB) {
    const int32_t q = __ldg(diag_pos + r0 + i);
    const double x = q >= 0 ? sh.sum[q - t0] : 0.0;
    dinv[r0 + i] = (x > 0.0) ? 1.0 / x : 0.0;
  }
  for (int s = 0; s < ns; ++s) {
    const int32_t b = __ldg(sptr + s0 + s), w = (__ldg(sptr + s0 + s + 1) - b) >> 5, np = w >> 1;
    const int32_t f = __ldg(srow0 + s0 + s) - r0;  // the slice's first row, from r0
    const int32_t rows = __ldg(srow0 + s0 + s + 1) - r0 - f;
    for (int p = tid; p < 32 * w; p += NUM_TPB) {  // pair layout (sell.cu)
      const int i = p < 64 * np ? (p & 63) >> 1 : p - 64 * np;
      const int k = p < 64 * np ? 2 * (p >> 6) + (p & 1) : w - 1;
      double x = 0.0;
      if (i < rows) {
        if (mask) {
          const uint32_t mk = s_mk[32 * s + i];
          if ((mk >> k) & 1u) x = sh.sum[s_rs[f + i] + __popc(mk & ((1u << k) - 1u))];
        } else if (k < s_rs[f + i + 1] - s_rs[f + i]) {
          x = sh.sum[s_rs[f + i] + k];
        }
      }
      sval[b + p] = x;
    }
  }
}

// Jacobi: dinv_r = 1 / a_rr; a missing or non-positive diagonal stores 0,
// which the solves report as GBS_ERR_NOT_SPD for the system holding that row.
__global__ void k_jacobi(int64_t nrows, const int32_t *__restrict__ diag_pos,
                         const double *__restrict__ val, double *__restrict__ dinv) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t q = diag_pos[r];
    const double d = q >= 0 ? val[q] : 0.0;
    dinv[r] = (d > 0.0) ? 1.0 / d : 0.0;
  }
}

// The values of A, without its sliced copy, in tiles of 512 nonzeros.  Where a
// tile's entries would not fit shared memory its nonzeros go a thread each (which
// long segments want anyway: neighbours in the pattern are often neighbours in v),
// and few nonzeros are then dealt out to two CTAs an SM, a warp of them or more
// each, but no tile so small that it would fit again.  ms, tiles of 512 -> this: 1000
// sums of 3000 entries 1.22 -> 0.43, 10,000 of 300 0.141 -> 0.057, 300 of 3333 1.17 -> 0.47.
// (Tiles that fit, for every mean length: 912,673 sums of 8 entries 0.039 -> 0.048.)
static int numeric_values(gbs_mat A, const double *v, int mode, cudaStream_t s) {
  int64_t tile = NUM_TILE;
  if (NUM_TILE * A->nkept > NUM_E * A->nnz) {
    const int64_t least = NUM_E * A->nnz / A->nkept + 1, share = A->nnz / (2 * sm_count(A));
    tile = std::min<int64_t>(NUM_TILE, (std::max(least, share) + 31) / 32 * 32);
  }
  k_coo_numeric<<<grid_for(A->nnz, (int)tile), NUM_TPB, num_shared(NUM_E, NUM_TILE), s>>>(
      A->nnz, (int32_t)tile, A->jmap, A->perm, v, mode, A->val);
  GBS_LAUNCHED(1);
  return GBS_OK;
}

int launch_set_values(gbs_mat A, const double *v, int mode, cudaStream_t s) {
  // slices a tile holds, where every tile of so many fits (their largest
  // counts are the shape's)
  const int32_t per =
      A->sell_val && A->slice_max_nnz > 0
          ? (int32_t)std::min<int64_t>(NUM_SLICES, std::min<int64_t>(NUM_NZ / A->slice_max_nnz,
                                                                     NUM_E / A->slice_max_coo))
          : 0;
  if (per >= 1) {
    const int e_cap = per * A->slice_max_coo, nz_cap = per * A->slice_max_nnz;
    k_numeric_slices<<<(unsigned)((A->nslices + per - 1) / per), NUM_TPB,
                       num_shared(e_cap, nz_cap), s>>>(
        A->nslices, per, e_cap, nz_cap, A->sell_row0, A->row_ptr, A->jmap, A->perm, v, mode, A->val,
        A->diag_pos, A->dinv, A->sell_ptr, A->sell_npat ? A->sell_mask : nullptr, A->sell_val);
    GBS_LAUNCHED(1);
  } else {
    if (A->nnz > 0) GBS_TRY(numeric_values(A, v, mode, s));
    if (A->nrows > 0) {
      k_jacobi<<<grid_for(A->nrows, 256), 256, 0, s>>>(A->nrows, A->diag_pos, A->val, A->dinv);
      GBS_LAUNCHED(1);
    }
    GBS_TRY(sell_values(A, s));
  }
  A->values_set = true;
  A->val32_valid = false;
  A->values_version += 1;
  return GBS_OK;
}

// FP32 copies for the refined solve: val32 = RN(val), dinv32 = RN(dinv).
__global__ void k_to_fp32(int64_t nnz, const double *__restrict__ val, float *__restrict__ val32,
                          int64_t nrows, const double *__restrict__ dinv,
                          float *__restrict__ dinv32) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nnz; p += stride)
    val32[p] = __double2float_rn(val[p]);
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += stride)
    dinv32[r] = __double2float_rn(dinv[r]);
}

int launch_to_fp32(gbs_mat A, cudaStream_t s) {
  if (!A->val32) {
    GBS_TRY(dev_alloc(&A->val32, std::max<int64_t>(A->nnz, 1), s));
    GBS_TRY(dev_alloc(&A->dinv32, std::max<int64_t>(A->nrows, 1), s));
  }
  k_to_fp32<<<grid_for(std::max(A->nnz, A->nrows), 256), 256, 0, s>>>(
      A->nnz, A->val, A->val32, A->nrows, A->dinv, A->dinv32);
  GBS_LAUNCHED(1);
  GBS_TRY(sell_values32(A, s));
  A->val32_valid = true;
  return GBS_OK;
}

// ------------------------------------------------------------------ vectors

// y[r] = a_{p(r)} (INSERT) or y[r] + a_{p(r)} (ADD) for every index r that
// has an entry (its row of the n x 1 pattern is non-empty); other y[r] keep.
__global__ void k_vec_scatter(int64_t n, const int32_t *__restrict__ row_ptr,
                              const double *__restrict__ val, int mode, double *__restrict__ y) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t p = row_ptr[r];
    if (row_ptr[r + 1] > p) y[r] = (mode == GBS_ADD) ? y[r] + val[p] : val[p];
  }
}

// Vector numeric stage: the in-order sums of the n x 1 pattern (the matrix
// numeric kernel, INSERT into val), then the scatter into y.
int launch_vec_set_values(gbs_mat A, const double *v, int mode, double *y, cudaStream_t s) {
  if (A->nnz > 0) GBS_TRY(numeric_values(A, v, GBS_INSERT, s));
  if (A->nrows > 0) {
    k_vec_scatter<<<grid_for(A->nrows, 256), 256, 0, s>>>(A->nrows, A->row_ptr, A->val, mode, y);
    GBS_LAUNCHED(1);
  }
  return GBS_OK;
}

// ------------------------------------------------------------------ adjoint scatter

// dLda[p] = -lambda[row p] * x[col p]; dLdv[perm[t]] = dLda[p] for t in the
// segment of p.  One thread per nonzero, so the reads of col, jmap and perm
// and the writes of dLda are coalesced.  A warp takes 32 consecutive
// nonzeros: lane 0 finds the row of the first by binary search over row_ptr
// (the last r with row_ptr[r] <= p0, which skips empty rows), and each lane
// walks forward from there to its own row -- at most the number of rows the
// warp's nonzeros span.  Ignored COO entries are zeroed by the caller's
// memset.
__global__ void k_adjoint_scatter(int64_t nnz, int64_t nrows, const int32_t *__restrict__ row_ptr,
                                  const int32_t *__restrict__ col,
                                  const int32_t *__restrict__ jmap,
                                  const int32_t *__restrict__ perm,
                                  const double *__restrict__ lambda,
                                  const double *__restrict__ x, double *__restrict__ dLda,
                                  double *__restrict__ dLdv) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c * 32 < nnz; c += nw) {
    const int64_t p0 = c * 32, p = p0 + lane;
    int64_t r0 = 0;
    if (lane == 0) {
      int64_t lo = 0, hi = nrows;  // row_ptr[0] = 0 <= p0 < nnz = row_ptr[nrows]
      while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (row_ptr[mid] <= p0) lo = mid;
        else hi = mid - 1;
      }
      r0 = lo;
    }
    r0 = __shfl_sync(FULL_MASK, r0, 0);
    if (p < nnz) {
      int64_t r = r0;
      while (row_ptr[r + 1] <= p) ++r;
      const double g = -(lambda[r] * x[col[p]]);
      if (dLda) dLda[p] = g;
      if (dLdv)
        for (int32_t t = jmap[p]; t < jmap[p + 1]; ++t) dLdv[perm[t]] = g;
    }
  }
}

int launch_adjoint_scatter(gbs_mat A, const double *lambda, const double *x, double *dLda,
                           double *dLdv, cudaStream_t s) {
  if (dLdv && A->ncoo > 0 && A->nkept < A->ncoo)
    GBS_TRY_CUDA(cudaMemsetAsync(dLdv, 0, sizeof(double) * A->ncoo, s));
  if ((dLda || dLdv) && A->nnz > 0) {
    k_adjoint_scatter<<<grid_for((A->nnz + 31) / 32 * 32, 256), 256, 0, s>>>(
        A->nnz, A->nrows, A->row_ptr, A->col, A->jmap, A->perm, lambda, x, dLda, dLdv);
    GBS_LAUNCHED(1);
  }
  return GBS_OK;
}

}  // namespace gbs
