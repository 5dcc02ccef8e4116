// Jacobi-PCG with a team of CTAs per system, every iteration inside one
// launch (Sec. 6.1 CG with device-resident scalars and no host round trip).
//
// The phase kernels (phases.cuh) pay three kernel boundaries an iteration:
// each drains the grid, launches the next one, refills it and finishes its
// reduction in one last CTA -- 14 to 17 us an iteration however small the
// system.  Measured, us an iteration, phases -> here: 2D 64^2 15.7 -> 5.9,
// 256^2 15.9 -> 9.5, 512^2 21.5 -> 13.8, 1024^2 42.1 -> 35.9; Q1 32^3 21.1 ->
// 12.5, 64^3 37.0 -> 28.4, 96^3 76.0 -> 68.0; 3D 7-point 100^3 45.1 -> 39.7.
// What bounds them: the meetings and the FP64 latency of the sums on small
// systems (a dependent FP64 add takes 60 clocks and more), the FP64 pipe (two
// FMAs a clock an SM, nonzeros + 8 a row of them: 40 us of Q1 96^3's 68) and
// the gathers' latency on large ones.
//
// Here the CTAs stay: each owns a run of the system's 32-row slices
// for the whole solve, keeps its part of the vectors (and of the matrix, where
// it fits) in shared memory, and the team meets three times an iteration:
//
//   q = A p, p.q         -- sum over the team -> alpha
//   x, r, z, r.z, r.r    -- sum over the team -> tests, beta
//   p = z + beta p       -- barrier: p is what the other CTAs gather next
//
// Two kinds of team:
//   - a thread-block cluster (up to 16 CTAs) meets at the hardware cluster
//     barrier and exchanges its partial sums through distributed shared
//     memory: 0.2-0.3 us a barrier, 0.7-0.9 us a sum;
//   - the whole grid, one CTA per SM, launched cooperatively, meets at a
//     counter in global memory: 1.2 us a barrier, 1.9 us a sum (152 CTAs).
// Every wait of the grid team is bounded (over a second and 2^22 polls), after
// which the solve ends with GBS_ERR_TIMEOUT.  (A wait lasts as long as the other
// CTAs' longest run of rows takes: at most about a second for 2^31 entries on one SM.)
//
// Every CTA adds the team's partial sums itself, in rank order, and its thread
// 0 runs the scalar recurrences on the same totals, so all CTAs take the same
// decisions without a broadcast and results are the same on every run.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "cta.cuh"
#include "device_util.cuh"
#include "internal.cuh"
#include "phases.cuh"

namespace gbs {

constexpr int TEAM_MAX_CLUSTER = 16;
constexpr int64_t TEAM_WAIT_NS = 1000000000;   // bounded waits: over a second and
constexpr unsigned TEAM_WAIT_POLLS = 1u << 22;  // 2^22 polls

// How a launch lays out its dynamic shared memory: the block sums' scratch,
// the p window and (clusters) the halo of z, then nvec vectors of rows_cap
// rows, then mat_cap bytes for the CTA's part of the sliced copy.
struct TeamCfg {
  int32_t window;  // 1: windows of p in shared memory (halo rows beyond the CTA's own)
  int32_t halo, win_cap, zh_cap;
  int32_t nvec, rows_cap, mat_cap;
  unsigned *ctr;   // grid team: arrivals, zero at launch
  // ... and how long one of its waits may last: both so many polls and so many ns
  // (a process that the GPU sets aside for a while polls no more)
  unsigned wait_polls;
  int64_t wait_ns;
  double *slots;   // grid team: 2 parities x 2 values x CTAs
};

// The part of a system one CTA owns: slices [s0, s1), rows [r0, r1).
struct TeamPart {
  int s, s0, s1, r0, r1;
  int w0, w1;    // window of p: its own rows and those its row products read
  int dlo, dhi;  // the cluster's CTAs with rows of this one in their windows
};

// The vectors of a solve, where they live: shared memory (offset so that row
// indices apply) or global.  p is the window, or the global vector that the
// whole team gathers; zh holds the window's halo of z (clusters), zg the z
// that the grid's CTAs read their halos from.
struct TeamVecs {
  double *q, *r, *z, *dv, *x, *p, *zh, *zg;
};

struct TeamShared {
  // (here, not in registers: a pass over the rows loads the few it needs)
  TeamPart g;
  TeamVecs V;
  SellView sv;
  const double *sval;
  double lanes[2 * 128];                    // block_sums' lane partials
  double box[2][2][TEAM_MAX_CLUSTER];       // partial sums of the cluster's CTAs, by parity
  double pub[2];
  int ipub[2];
  // thread 0's scalars (in shared memory, not in every thread's registers)
  SysState S;                               // bb, rr, thr and its bounds, rho, rnorm0
  int it, status, timed, zero;
  int abort;                                // a bounded wait ran out
  // the rows each CTA of the cluster takes into its halo of z, and where
  int32_t lo[TEAM_MAX_CLUSTER], hi[TEAM_MAX_CLUSTER];
  uint32_t to[TEAM_MAX_CLUSTER];
  CallArgs call;                            // (global loads would wait on L2: L1 is dropped
                                            // at every meeting)
  unsigned long long ns[5], last;           // phase timers (one thread of rank 0)
  TeamCfg cfg;                              // batches: this system's layout,
  int next;                                 //   and the system the cluster solves
};

// (The aligned forms want the whole warp at once: callers come from code that some of
// its lanes skip.)
__device__ __forceinline__ void cluster_meet() {
  __syncwarp();
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::
          : "memory");
}

// The address that p (this CTA's shared memory) has in the cluster's CTA `rank`.
__device__ __forceinline__ uint32_t remote(const void *p, int rank) {
  const uint32_t l = (uint32_t)__cvta_generic_to_shared(p);
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(l), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote(uint32_t to, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(to), "d"(v) : "memory");
}

template <bool GRID>
struct Team {
  int rank, size;
  TeamShared &sh;
  double *red;      // 2 blockDim doubles
  const TeamCfg &cfg;
  DevCtl *ctl;
  unsigned target;  // grid: arrivals that complete the next meeting
  int par;

  // Warp 0 counts the CTA in and waits for the whole grid.
  __device__ __forceinline__ void arrive_and_wait() {
    target += (unsigned)size;
    if (threadIdx.x == 0)
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(cfg.ctr) : "memory");
    unsigned v;
    uint64_t t0 = 0;
    for (unsigned polls = 0;; ++polls) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cfg.ctr) : "memory");
      if ((int)(v - target) >= 0) break;
      if ((polls & 1023u) == 1023u) {
        const uint64_t t = global_ns();
        if (t0 == 0) t0 = t;
        else if (polls > cfg.wait_polls && t - t0 > (uint64_t)cfg.wait_ns) {
          sh.abort = 1;
          break;
        }
      }
    }
    __syncwarp();
  }

  // Sums over the team of NV <= 2 values a thread, valid in warp 0 of every
  // CTA (the same bits in all of them).
  template <int NV>
  __device__ __forceinline__ void sum(double (&v)[NV]) {
    block_sums<double, NV>(v, red, sh.lanes);
    if (size == 1) return;
    const int lane = threadIdx.x & 31;
    if constexpr (GRID) {
      if ((threadIdx.x >> 5) != 0) return;
      double *s = cfg.slots + (size_t)par * 2 * size;
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) s[k * size + rank] = v[k];
      }
      arrive_and_wait();
      // lane l adds slots l, l + 32, ...; all loads of a batch in flight
      constexpr int BATCH = 6;
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] = 0.0;
      for (int i0 = 0; i0 < size; i0 += 32 * BATCH) {
        double u[BATCH][NV];
#pragma unroll
        for (int j = 0; j < BATCH; ++j)
#pragma unroll
          for (int k = 0; k < NV; ++k) {
            const int i = i0 + 32 * j + lane;
            u[j][k] = i < size ? ldcg(s + k * size + i) : 0.0;
          }
#pragma unroll
        for (int j = 0; j < BATCH; ++j)
#pragma unroll
          for (int k = 0; k < NV; ++k)
            if (i0 + 32 * j < size) v[k] += u[j][k];
      }
      warp_sums<double, NV>(v);
    } else {
      if ((threadIdx.x >> 5) == 0 && lane < size) {
#pragma unroll
        for (int k = 0; k < NV; ++k) st_remote(remote(&sh.box[par][k][rank], lane), v[k]);
      }
      cluster_meet();
      if ((threadIdx.x >> 5) == 0) {
        // value lane / 16 of CTA lane % 16: four steps add either one value or two
        const int k = NV == 2 ? lane >> 4 : 0, c = lane & 15;
        double t = c < size ? sh.box[par][k][c] : 0.0;
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) t += __shfl_xor_sync(FULL_MASK, t, d);
#pragma unroll
        for (int q = 0; q < NV; ++q) v[q] = __shfl_sync(FULL_MASK, t, 16 * q);
      }
    }
    par ^= 1;
  }

  // Every thread's global writes before it are visible to every thread of the
  // team after it.
  __device__ __forceinline__ void barrier() {
    if constexpr (GRID) {
      __syncthreads();
      if ((threadIdx.x >> 5) == 0) arrive_and_wait();
      __syncthreads();
    } else {
      if (size > 1) cluster_meet();
      else __syncthreads();
    }
  }
  __device__ __forceinline__ bool aborted() const { return GRID && sh.abort != 0; }
};

// FP64 PCG on one system: cta_pcg_fp64's steps, tests and statuses, over a
// team.
//
// WIN: the CTA holds p for every row that its row products read, its own and
// a halo of col_span rows on either side.  The update hands z's halo rows over
// together with the partial sums (to the other CTAs' shared memory, or through
// L2), and after the sum every CTA forms p = z + beta p over its whole window
// -- the same operations on the same values as the owner's, so the same bits
// -- and needs no third meeting; the row products then gather from shared
// memory.  Without windows (a span too wide for them) p is a global vector and
// the third meeting publishes it.
template <bool GRID, bool SM, bool WIN>
__device__ __forceinline__ void team_pcg(const PcgArgs &a, Team<GRID> &tm, bool timers) {
  TeamShared &sh = tm.sh;
  // The element-wise passes copy the pointers they use: read through sh, every
  // store of the pass might change them, and each row would load them again.
  // (The streaming row products leave them there: their loads in flight take
  // the registers.)
  const TeamVecs &V = sh.V;
  const TeamPart &g = sh.g;
  const CallArgs &C = sh.call;
  const double *b = C.b;
  double *xg = C.x;
  const bool t0 = threadIdx.x == 0, lead = tm.rank == 0;
  const bool clk = timers && lead && threadIdx.x == 32;
  auto mark = [&](int k) {
    if (clk) {
      const unsigned long long t = global_ns();
      sh.ns[k] += t - sh.last;
      sh.last = t;
    }
  };
  if (clk) {
    for (int k = 0; k < 5; ++k) sh.ns[k] = 0;
    sh.last = global_ns();
  }
  auto rows = [&](auto gather, const double *v, auto &f) {
    constexpr int NC = decltype(gather)::value;
    if constexpr (SM) {
      const SellView sv = sh.sv;
      sell_rows<double, false, NC, true, 2>(sv, sh.sval, v, g.s0, g.s1, f);
    } else {
      if (a.stream_matrix) sell_rows<double, true, NC, false, 4>(a.sv, a.sval, v, g.s0, g.s1, f);
      else sell_rows<double, false, NC, false, 4>(a.sv, a.sval, v, g.s0, g.s1, f);
    }
  };
  std::integral_constant<int, GATHER_CA> from_global;
  std::integral_constant<int, WIN ? GATHER_SM : GATHER_CA> from_p;
  auto p_at = [](const double *p, int i) -> double {
    if constexpr (WIN) return p[i];
    else return __ldca(p + i);
  };
  // z of an own row, handed to the CTAs that hold the row in their halos
  auto hand_z = [&](double *zown, double *zg, int i, double z) {
    if constexpr (WIN && GRID) {
      if (zown != zg) zg[i] = z;
    } else if constexpr (WIN) {
      for (int d = g.dlo, e = g.dhi; d <= e; ++d)
        if (i >= sh.lo[d] && i < sh.hi[d]) st_remote(sh.to[d] + 8u * (uint32_t)i, z);
    }
  };
  // p = z (+ beta p), over the window or the own rows
  auto direction = [&](bool first, double be) {
    constexpr int U = 2;
    double *const p = V.p;
    const double *const z = V.z, *const zg = V.zg, *const zh = V.zh;
    double pv[U], zv[U];
    auto ld = [&](int i, int k) {
      pv[k] = first ? 0.0 : p_at(p, i);
      zv[k] = z[i];
    };
    auto use = [&](int i, int k) { p[i] = first ? zv[k] : fma(be, pv[k], zv[k]); };
    const int r0 = g.r0, r1 = g.r1;
    cta_rows_by<U>(r0, r1, ld, use);
    if constexpr (WIN) {
      const int w0 = g.w0, nlo = r0 - w0, nh = nlo + g.w1 - r1;
      for (int h = threadIdx.x; h < nh; h += blockDim.x) {
        const int i = h < nlo ? w0 + h : r1 + (h - nlo);
        const double zi = GRID ? __ldcg(zg + i) : zh[h];
        p[i] = first ? zi : fma(be, p[i], zi);
      }
      __syncthreads();
    }
  };
  // setup: r = b - A x0, z = D^-1 r; r.z, r.r, then b.b, missing diagonals
  double u[2] = {0.0, 0.0}, w[2] = {0.0, 0.0};
  {
    double *const r = V.r, *const z = V.z, *const zg = V.zg, *const dv = V.dv, *const x = V.x;
    auto start = [&](int i, double t) {
      const double bv = b[i], rv = bv - t, d = a.dinv[i], zv = d * rv;
      if (dv != a.dinv) dv[i] = d;
      r[i] = rv;
      z[i] = zv;
      hand_z(z, zg, i, zv);
      u[0] = fma(rv, zv, u[0]);
      u[1] = fma(rv, rv, u[1]);
      w[0] = fma(bv, bv, w[0]);
      w[1] += (d == 0.0) ? 1.0 : 0.0;
    };
    if (C.nonzero_guess) {
      if (x != xg)
        for (int i = g.r0 + threadIdx.x; i < g.r1; i += blockDim.x) x[i] = xg[i];
      rows(from_global, xg, start);
    } else {
      for (int i = g.r0 + threadIdx.x; i < g.r1; i += blockDim.x) {
        x[i] = 0.0;
        start(i, 0.0);
      }
    }
  }
  tm.template sum<2>(u);
  __syncthreads();  // (block_sums' scratch)
  tm.template sum<2>(w);
  SysState &S = sh.S;
  if (t0) {  // the scalars, the same in every CTA
    int status = -1;
    sh.it = sh.timed = sh.zero = 0;
    S.rho = u[0];
    S.rr = u[1];
    S.bb = w[0];
    set_thr(S, C.rtol * sqrt(S.bb));
    S.rnorm0 = sqrt(S.rr);
    if (w[1] > 0.0) status = GBS_ERR_NOT_SPD;
    else if (!isfinite(S.bb)) status = GBS_ERR_NAN;
    else if (S.bb == 0.0) {
      status = GBS_OK;
      sh.zero = 1;
      S.rr = S.rnorm0 = 0.0;
    } else if (!isfinite(S.rr) || !isfinite(S.rho)) status = GBS_ERR_NAN;
    else if (S.rnorm0 <= S.thr) status = GBS_OK;
    else if (C.maxit <= 0) status = GBS_ERR_MAXIT;
    sh.status = sh.ipub[0] = status;
  }
  __syncthreads();
  direction(true, 0.0);
  if constexpr (!WIN) tm.barrier();
  const bool zero_x = sh.zero != 0, limited = C.timeout_ns > 0;
  const bool go = sh.ipub[0] < 0 && !tm.aborted();
  mark(0);
  while (go) {
    // q = A p, p.q -> alpha
    double pq[1] = {0.0};
    {
      double *const ql = V.q;
      const double *const pl = V.p;
      auto fa = [&](int i, double y) {
        if constexpr (SM) {
          ql[i] = y;
          pq[0] = fma(p_at(pl, i), y, pq[0]);
        } else {
          V.q[i] = y;
          pq[0] = fma(p_at(V.p, i), y, pq[0]);
        }
      };
      rows(from_p, pl, fa);
    }
    tm.template sum<1>(pq);
    if (t0) {
      int status = -1;
      sh.it += 1;
      if (nan64(pq[0])) status = GBS_ERR_NAN;
      else if (!positive64(pq[0])) status = GBS_ERR_BREAKDOWN;
      else sh.pub[0] = S.rho / pq[0];
      sh.status = sh.ipub[0] = status;
    }
    __syncthreads();
    mark(1);
    if (sh.ipub[0] >= 0 || tm.aborted()) break;
    const double al = sh.pub[0];
    // x += alpha p, r -= alpha q, z = D^-1 r, r.z, r.r -> tests, beta
    {
      constexpr int U = 2;
      const double *const q = V.q, *const p = V.p, *const dv = V.dv;
      double *const r = V.r, *const z = V.z, *const zg = V.zg, *const x = V.x;
      double rz = 0.0, rr = 0.0;
      double qv[U], rv0[U], d[U], pv[U], xv[U];
      auto ld = [&](int i, int k) {
        qv[k] = q[i];
        rv0[k] = r[i];
        d[k] = dv[i];
        pv[k] = p_at(p, i);
        xv[k] = x[i];
      };
      auto use = [&](int i, int k) {
        const double rv = fma(-al, qv[k], rv0[k]);
        const double zv = d[k] * rv;
        x[i] = fma(al, pv[k], xv[k]);
        r[i] = rv;
        z[i] = zv;
        hand_z(z, zg, i, zv);
        rz = fma(rv, zv, rz);
        rr = fma(rv, rv, rr);
      };
      const int r0 = g.r0, r1 = g.r1;
      cta_rows_by<U>(r0, r1, ld, use);
      u[0] = rz;
      u[1] = rr;
    }
    // the time limit is the lead's clock: its verdict goes round with the sums
    double late[1] = {0.0};
    if (limited && lead && t0) late[0] = cta_timed_out(a.ctl, C.timeout_ns) ? 1.0 : 0.0;
    tm.template sum<2>(u);
    if (limited) {
      __syncthreads();
      tm.template sum<1>(late);
    }
    if (t0) {
      int status = -1;
      S.rr = u[1];
      if (!finite64(u[1]) || !finite64(u[0])) status = GBS_ERR_NAN;
      else if (meets_thr(u[1], S)) status = GBS_OK;
      else if (sh.it >= C.maxit) status = GBS_ERR_MAXIT;
      else if (late[0] != 0.0) sh.timed = 1;
      else {
        sh.pub[1] = u[0] / S.rho;
        S.rho = u[0];
      }
      sh.status = status;
      sh.ipub[1] = (status < 0 && late[0] == 0.0) ? -1 : 0;
    }
    __syncthreads();
    mark(2);
    if (sh.ipub[1] >= 0 || tm.aborted()) break;
    direction(false, sh.pub[1]);
    if constexpr (!WIN) {
      tm.barrier();
      if (tm.aborted()) break;
    }
    mark(3);
  }
  // x out, then ||b - A x||^2 (x = 0 where b = 0)
  if (const double *const x = V.x; zero_x || x != xg)
    for (int i = g.r0 + threadIdx.x; i < g.r1; i += blockDim.x) xg[i] = zero_x ? 0.0 : x[i];
  if (!tm.aborted()) tm.barrier();
  double tt[1] = {0.0};
  auto ft = [&](int i, double t) {
    const double d = b[i] - t;
    tt[0] = fma(d, d, tt[0]);
  };
  rows(from_global, xg, ft);
  if (!tm.aborted()) tm.template sum<1>(tt);
  if (lead && t0) {
    const bool stopped = sh.timed || tm.aborted();
    SysState &O = a.st[sh.g.s];
    memset(&O, 0, sizeof(SysState));
    O.bb = S.bb;
    O.rnorm0 = S.rnorm0;
    O.rnorm = sqrt(S.rr);
    O.tt = tt[0];
    O.iterations = sh.it;
    O.zero_x = sh.zero;
    O.status = stopped ? GBS_OK : sh.status;
    O.active = stopped ? 1 : 0;  // reported as the control word's error
    if (stopped) a.ctl->err = GBS_ERR_TIMEOUT;
  }
  mark(4);
  if (clk)
    for (int k = 0; k < 5; ++k) a.ctl->phase_ns[k] += (int64_t)sh.ns[k];
}

__device__ __forceinline__ size_t up16(size_t n) { return (n + 15) & ~(size_t)15; }

// Copies the CTA's part of the sliced copy into shared memory at m (cap
// bytes); the view and the values are rebased so that global slice, entry and
// pool indices apply.  Returns false (nothing copied) where it does not fit.
__device__ bool team_cache(const SellView &S, const double *sval, const TeamPart &g,
                           unsigned char *m, size_t cap, SellView &V, const double **vals) {
  const int ns = g.s1 - g.s0;
  if (ns <= 0) return false;
  const int e0 = __ldg(S.ptr + g.s0), e1 = __ldg(S.ptr + g.s1);
  const size_t ne = (size_t)(e1 - e0);
  int pool0 = 0, npool = 0;
  if (S.pat) {
    pool0 = __ldg(S.pat + g.s0);
    const int wl = (e1 - __ldg(S.ptr + g.s1 - 1)) >> 5;
    npool = __ldg(S.pat + g.s1 - 1) + ((wl + 1) & ~1) - pool0;
  }
  const size_t o_ptr = up16(ne * 8), o_row = o_ptr + up16(4 * (size_t)(ns + 1));
  const size_t o_a = o_row + up16(4 * (size_t)(ns + 1));
  size_t o_pool = 0, o_mask = 0, need = o_a;
  if (S.pat) {
    o_pool = o_a + up16(4 * (size_t)ns);
    o_mask = o_pool + up16(4 * (size_t)npool);
    need = o_mask + 128 * (size_t)ns;
  } else {
    need = o_a + (S.off ? 2 : 4) * ne;
  }
  if (need > cap) return false;
  auto copy = [&](auto *dst, const auto *src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = __ldg(src + i);
  };
  copy(reinterpret_cast<double2 *>(m), reinterpret_cast<const double2 *>(sval + e0), (int)(ne >> 1));
  copy(reinterpret_cast<int32_t *>(m + o_ptr), S.ptr + g.s0, ns + 1);
  copy(reinterpret_cast<int32_t *>(m + o_row), S.row0 + g.s0, ns + 1);
  V = S;
  V.ptr = reinterpret_cast<int32_t *>(m + o_ptr) - g.s0;
  V.row0 = reinterpret_cast<int32_t *>(m + o_row) - g.s0;
  *vals = reinterpret_cast<double *>(m) - e0;
  if (S.pat) {
    copy(reinterpret_cast<int32_t *>(m + o_a), S.pat + g.s0, ns);
    copy(reinterpret_cast<int32_t *>(m + o_pool), S.pool + pool0, npool);
    copy(reinterpret_cast<uint32_t *>(m + o_mask), S.mask + 32 * (int64_t)g.s0, 32 * ns);
    V.pat = reinterpret_cast<int32_t *>(m + o_a) - g.s0;
    V.pool = reinterpret_cast<int32_t *>(m + o_pool) - pool0;
    V.mask = reinterpret_cast<uint32_t *>(m + o_mask) - 32 * (int64_t)g.s0;
  } else if (S.off) {
    copy(reinterpret_cast<int32_t *>(m + o_a), reinterpret_cast<const int32_t *>(S.off + e0),
         (int)(ne >> 1));
    V.off = reinterpret_cast<int16_t *>(m + o_a) - e0;
  } else {
    copy(reinterpret_cast<int32_t *>(m + o_a), S.col + e0, (int)ne);
    V.col = reinterpret_cast<int32_t *>(m + o_a) - e0;
  }
  __syncthreads();
  return true;
}

// One system on the CTA's team: lays the CTA's part out in shared memory as c
// says (the same in every CTA of a cluster, whose halo tables point into one
// another) and solves.
template <bool GRID>
__device__ __forceinline__ void team_system(const PcgArgs &a, const TeamCfg &c, TeamShared &sh,
                                            double *red, const SysRange &sys, uint32_t rank,
                                            uint32_t size, bool timers) {
  double *win = red + 2 * blockDim.x, *zh = win + c.win_cap, *vec = zh + c.zh_cap;
  unsigned char *mat = reinterpret_cast<unsigned char *>(vec + (size_t)c.nvec * c.rows_cap);
  Team<GRID> tm{(int)rank, (int)size, sh, red, c, a.ctl, 0u, 0};
  const int64_t ns = sys.s1 - sys.s0;
  auto part = [&](int k, int &r0, int &r1) {  // rows of the team's CTA k
    r0 = min(sys.r1, sys.r0 + 32 * (int)(ns * k / size));
    r1 = min(sys.r1, sys.r0 + 32 * (int)(ns * (k + 1) / size));
  };
  auto window = [&](int r0, int r1, int &w0, int &w1) {  // (r1 - halo: no overflow)
    w0 = r0 < r1 ? max(sys.r0, r0 - c.halo) : r0;
    w1 = r0 < r1 ? (sys.r1 - r1 < c.halo ? sys.r1 : r1 + c.halo) : r1;
  };
  TeamPart g;
  g.s = sys.s;
  g.s0 = sys.s0 + (int)(ns * rank / size);
  g.s1 = sys.s0 + (int)(ns * (rank + 1) / size);
  part(rank, g.r0, g.r1);
  window(g.r0, g.r1, g.w0, g.w1);
  g.dlo = 0;
  g.dhi = -1;
  if constexpr (!GRID) {
    if (c.window && size > 1) {
      if (threadIdx.x < size) {
        const int d = threadIdx.x;
        int r0, r1, w0, w1;
        part(d, r0, r1);
        window(r0, r1, w0, w1);
        sh.lo[d] = d == (int)rank ? INT32_MAX : max(g.r0, w0);
        sh.hi[d] = min(g.r1, w1);
        // rows below d's own start its halo, rows above follow them
        sh.to[d] = remote(zh, d) - 8u * (uint32_t)((int)rank < d ? w0 : r1 - (r0 - w0));
      }
      __syncthreads();
      for (int d = 0; d < (int)size; ++d)
        if (sh.lo[d] < sh.hi[d]) {
          if (g.dhi < 0) g.dlo = d;
          g.dhi = d;
        }
    }
  }
  // q, r, [z,] D^-1, x: without windows z is kept over q
  const bool w = c.window != 0;
  if (threadIdx.x == 0) {
    int k = 0;
    auto home = [&](double *global) {
      const int at = k++;
      return at < c.nvec ? vec + (int64_t)at * c.rows_cap - g.r0 : global;
    };
    TeamVecs &V = sh.V;
    V.q = home(w ? a.p : a.q);
    V.r = home(a.r);
    V.z = w ? home(a.q) : V.q;
    V.dv = home(const_cast<double *>(a.dinv));
    V.x = home(sh.call.x);
    V.p = w ? win - g.w0 : a.p;
    V.zh = zh;
    V.zg = a.q;
    sh.g = g;
  }
  SellView C;
  const double *vals = nullptr;
  const bool cached = c.mat_cap > 0 && team_cache(a.sv, a.sval, g, mat, c.mat_cap, C, &vals);
  if (threadIdx.x == 0 && cached) {
    sh.sv = C;
    sh.sval = vals;
  }
  __syncthreads();
  if (w) {
    if (cached) team_pcg<GRID, true, true>(a, tm, timers);
    else team_pcg<GRID, false, true>(a, tm, timers);
  } else {
    if (cached) team_pcg<GRID, true, false>(a, tm, timers);
    else team_pcg<GRID, false, false>(a, tm, timers);
  }
}

// One system (an ensemble solve).
template <bool GRID, int TPB>
__global__ void __launch_bounds__(TPB, 1) k_team(PcgArgs a, const __grid_constant__ TeamCfg cfg) {
  extern __shared__ __align__(16) unsigned char team_smem[];
  __shared__ TeamShared sh;
  uint32_t rank, size;
  if constexpr (GRID) {
    rank = blockIdx.x;
    size = gridDim.x;
  } else {
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(size));
  }
  if (threadIdx.x == 0) {
    sh.abort = 0;
    sh.call = *a.call;
  }
  __syncthreads();
  if (!GRID && size > 1) cluster_meet();  // every CTA runs before its shared memory is written
  team_system<GRID>(a, cfg, sh, reinterpret_cast<double *>(team_smem), cta_system(a, 0), rank,
                    size, true);
  if (!GRID && size > 1) cluster_meet();  // no CTA leaves while others may write to its boxes
}

// Shared memory of a batch's systems: windows where the halo's work stays
// below the meeting they save, then as many vectors as fit, then the matrix.
__device__ __forceinline__ TeamCfg team_layout(int n, int per_rows, int halo, int size,
                                               int smem) {
  TeamCfg c;
  c.window = c.halo = c.win_cap = c.zh_cap = c.mat_cap = 0;
  c.ctr = nullptr;
  c.slots = nullptr;
  c.wait_polls = TEAM_WAIT_POLLS;
  c.wait_ns = TEAM_WAIT_NS;
  c.rows_cap = max(per_rows, 32);
  int room = smem / 8 - 2 * (int)blockDim.x;  // doubles
  const int h = min(halo, n), win = (min(n, c.rows_cap + 2 * h) + 31) & ~31;
  const int zh = (min(2 * h, n) + 31) & ~31;
  if (2 * h <= max(c.rows_cap, 4096) && win + zh <= room / 2) {
    c.window = 1;
    c.halo = h;
    c.win_cap = win;
    c.zh_cap = zh;
    room -= win + zh;
  }
  const int nv = c.window ? 5 : 4;
  c.nvec = min(nv, room / c.rows_cap);
  if (c.nvec == nv) c.mat_cap = 8 * (room - nv * c.rows_cap) & ~15;
  return c;
}

// (Not inlined: what the systems share would be hoisted out of the loop over
// them and spilled -- 2.6 KB a thread at 64 registers.)
__device__ __noinline__ void batch_system(const PcgArgs &a, TeamShared &sh, double *red,
                                          uint32_t rank, uint32_t size) {
  team_system<false>(a, sh.cfg, sh, red, cta_system(a, sh.next), rank, size,
                     blockIdx.x == 0);  // (the first cluster's phase times)
}

// A batch (FP64 CG, each system on its own): a persistent grid of clusters, each
// taking system order[cluster], then the next unsolved one from a queue -- the
// per-CTA solver's scheme with `size` SMs to a system: a batch of fewer systems
// than SMs leaves none idle, and the largest systems end the batch sooner.
template <int TPB>
__global__ void __launch_bounds__(TPB, 1)
    k_team_batch(const __grid_constant__ PcgArgs a, int32_t halo, int32_t smem) {
  extern __shared__ __align__(16) unsigned char team_smem[];
  __shared__ TeamShared sh;
  uint32_t rank, size, cluster;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(size));
  asm("mov.u32 %0, %%clusterid.x;" : "=r"(cluster));
  if (threadIdx.x == 0) {
    sh.abort = 0;
    sh.call = *a.call;
  }
  __syncthreads();
  if (threadIdx.x == 0) sh.next = (int)cluster;
  __syncthreads();
  cluster_meet();  // every CTA runs before its shared memory is written
  while (sh.next < a.cta_n) {
    {
      const SysRange sys = cta_system(a, sh.next);
      if (threadIdx.x == 0)
        sh.cfg = team_layout(sys.r1 - sys.r0, 32 * ((sys.s1 - sys.s0 + (int)size - 1) / (int)size),
                             halo, (int)size, smem);
      __syncthreads();
      batch_system(a, sh, reinterpret_cast<double *>(team_smem), rank, size);
    }
    // the next system, from the lead's queue to every CTA of the cluster: after
    // a meeting, so that no CTA still reads this one, its boxes or its halos
    cluster_meet();
    if (rank == 0 && threadIdx.x == 0) {
      uint32_t nclusters;
      asm("mov.u32 %0, %%nclusterid.x;" : "=r"(nclusters));
      const int nx = (int)nclusters + atomicAdd(&a.ctl->queue, 1);
      for (int d = 0; d < (int)size; ++d)
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote(&sh.next, d)), "r"(nx)
                     : "memory");
    }
    cluster_meet();
  }
}

// A batch of few systems, larger than a cluster should hold: the CTAs of one
// cooperative grid shared out among them, system order[k] on CTAs [first[k],
// first[k + 1]), a grid team of its own with its own counter and slots.
constexpr int TEAM_PARTS_MAX = 64;
constexpr int TEAM_CTR_STRIDE = 32;  // words from one team's counter to the next: a line each
struct TeamParts {
  int16_t first[TEAM_PARTS_MAX + 1];
};

template <int TPB>
__global__ void __launch_bounds__(TPB, 1)
    k_team_parts(const __grid_constant__ PcgArgs a, const __grid_constant__ TeamParts parts,
                 int32_t halo, int32_t smem, int32_t streams, unsigned *ctr, double *slots,
                 unsigned wait_polls, int64_t wait_ns) {
  extern __shared__ __align__(16) unsigned char team_smem[];
  __shared__ TeamShared sh;
  int k = 0;
  while (k + 1 < a.cta_n && (int)blockIdx.x >= parts.first[k + 1]) ++k;
  const int first = parts.first[k], size = parts.first[k + 1] - first;
  const SysRange sys = cta_system(a, k);
  if (threadIdx.x == 0) {
    sh.abort = 0;
    sh.call = *a.call;
    TeamCfg c = team_layout(sys.r1 - sys.r0, 32 * ((sys.s1 - sys.s0 + size - 1) / size), halo,
                            size, smem);
    if (streams) {  // (as one system's: p through L1, and room left for it)
      c.window = c.halo = c.win_cap = c.zh_cap = c.mat_cap = 0;
      c.nvec = min(4, (smem / 8 - 2 * (int)blockDim.x) / c.rows_cap);
    }
    c.ctr = ctr + k * TEAM_CTR_STRIDE;
    c.slots = slots + 4 * first;
    c.wait_polls = wait_polls;
    c.wait_ns = wait_ns;
    sh.cfg = c;
  }
  __syncthreads();
  team_system<true>(a, sh.cfg, sh, reinterpret_cast<double *>(team_smem), sys,
                    blockIdx.x - first, size, blockIdx.x == 0);  // (the first team's phase times)
}

// ------------------------------------------------------------------ host side

constexpr int64_t TEAM_SMEM = 219 * 1024;  // dynamic shared memory a CTA may take (of 227 KB)
constexpr int64_t TEAM_L1_SMEM = 128 * 1024;  // ... where the row products need L1 for p

// One system runs on a cluster up to this many FP64 operations an iteration
// (nonzeros plus eight a row): 16 SMs do 32 of them a clock, so beyond it the
// grid's dearer meetings are the cheaper part.  Measured, us an iteration on
// cluster / grid: 2D 64^2 (53k operations) 5.9 / 8.1, 3D 16^3 (60k) 6.4 / 8.7,
// 2D 101^2 (132k) 7.9 / 8.1, Q1 16^3 (157k) 9.6 / 10.4, 2D 128^2 (212k) 8.6 / 8.0.
constexpr int64_t TEAM_CLUSTER_WORK = 160000;
// Beyond this many rows the phase kernels take over: twice the threads an SM
// hide HBM's latency better than the saved meetings are worth (3D 7-point,
// us an iteration on team / phases: 128^3 70.4 / 72.9, 160^3 141.6 / 134.0).
// Rows of fewer than four entries are the vectors' traffic for the most part and
// end sooner (tridiagonal, 1.5M 45.0 / 48.0, 1.75M 52.8 / 54.0, 2M 58.7 / 56.5, 2.8M 84.6 /
// 75.3).
constexpr int64_t TEAM_GRID_ROWS = 3 << 20, TEAM_SHORT_ROWS = 7 << 18;
// A team's CTA owns one run of slices, alone on its SM, where the phase kernels'
// four CTAs an SM take blocks from four places of the matrix: where the rows'
// lengths differ from place to place the team waits for its longest run.  That
// pays while the longest has at most a quarter over the mean's nonzeros, or its
// excess takes less of the FP64 pipe than the phase kernels' boundaries (28,000
// FMAs: 7 us) on a system of up to 2^20 rows.  Measured, us an iteration on team /
// phases (27-point rows followed by diagonal or 7-point ones; the longest run over
// the mean, its excess): 200k rows 1.36 (10k) 24.9 / 29.3, 2.0 (18k) 24.8 / 26.8,
// 7.7 (30k) 22.3 / 24.0; 600k 1.25 50.7 / 55.0, 1.34 (27k) 50.5 / 54.6, 1.62 (41k)
// 50.0 / 48.2, 2.29 (59k) 47.8 / 46.2, 7.7 (90k) 46.7 / 35.1; 1.5M 1.24 104.7 / 105.9,
// 1.60 105.2 / 93.6; 7-point rows followed by 5-point ones 600k 1.34 (8k) 27.1 / 31.2,
// 1.5M 1.17 53.1 / 54.2, 1.34 (18k) 58.0 / 53.4.
constexpr int64_t TEAM_EXCESS = 28000, TEAM_EXCESS_ROWS = 1 << 20;
// Without column patterns (gathers from anywhere, columns to read) only while
// matrix and vectors keep to half of L2: random columns, 9 a row, 400k rows
// (59 MB) 30.8 / 34.1, 550k (81) 42.6 / 42.2, 850k 63.1 / 56.1; 25 a row 150k 26.1 /
// 30.2, 450k 69.3 / 65.9; 3D edges 300k 20.0 / 25.0, 1M (110) 51.8 / 47.0, 3M 131 / 106.
static bool team_suits(gbs_mat A) {
  const int64_t n = A->nrows, run = A->run_max_nnz, sms = sm_count(A);
  if (n > (A->nnz < 4 * n ? TEAM_SHORT_ROWS : TEAM_GRID_ROWS)) return false;
  if (4 * run * sms > 5 * A->nnz &&
      (n > TEAM_EXCESS_ROWS || run - A->nnz / sms > TEAM_EXCESS))
    return false;
  if (A->sell_npat > 0) return true;
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, A->device);
  return 2 * (A->sell_nnz * (A->col_span <= 32767 ? 10 : 12) + 40 * n) <= (int64_t)l2;
}

// How a batch runs under the automatic choice: an estimate of each engine's time
// for one iteration of every system (us; fitted to 536 measured batches: equal
// systems, 2 to 300 of 1,500 to 500,000 rows, 5- to 27-point, and mixed ones), the
// least wins.  A system's iterations count as its rows to the 0.385th power: the
// larger ones go on when the smaller have converged.  Systems of unlike size are
// unlike in iterations too: every second one then counts UNLIKE of them where a
// queue hands on the SMs that it leaves early, and the shared grid, whose SMs would
// idle, UNLIKE_SHARE of its time; and clusters take the size that gives every SM work,
// larger ones where their estimate is less than UNLIKE_SIZE of it.
//   phase kernels   PHASES_US, and the operations at the whole chip's rate, dearer
//                   where the systems' blocks do not fit one wave; refined, the bytes
//   per-CTA solver  one SM a system, from a queue
//   clusters        the same with `size` SMs, as many clusters as are resident
//   shared grid     every system its own share of the SMs (k_team_parts)
// Measured, ms per 100 iterations, phase kernels / per-CTA / clusters of 2, 4, 8, 16 /
// shared grid:
//   2D   2 x 1.5k      1.0 / 1.0 / 0.95 0.81 0.75 0.71 / 0.92
//        2 x 150k      2.5 / 49 / 32 17 8.7 5.3 / 1.9
//        8 x 40k       2.4 / 13 / 8.9 5.3 3.1 4.1 / 2.0
//        64 x 60k     17.5 / 22 / 18 17 22 25 / 12.8
//        140 x 20k    12.9 / 8.0 / 12 12 20 25
//        160 x 40k    28.7 / 30 / 29 29 34 47
//   Q1   4 x 20k       2.4 / 18 / 9.8 5.5 3.3 2.3 / 1.5
//        16 x 60k      8.8 / 52 / 33 18 18 15 / 7.6
//        16 x 150k    17.2 / 130 / 82 44 40 34 / 17.7
//        100 x 30k    30.9 / 27 / 35 29 36 40
//   mixed, to 1e-10: 9 Q1 5k-47k 3.1 / 40 / 21 11 6.6 3.7 / 2.6;  135 of 600-3.6k
//        8.8 / 6.1 / 4.7 4.6 8.6 17;  211 of 3k-12k 43 / 29 / 23 24 38 62
//   refined, phase kernels / per-CTA: 76 x 8k Q1 3.1 / 3.2, 2D 78 x 40k 118 / 99, Q1 78 x
//        40k 20.8 / 24.3, 140 x 40k 35.7 / 27.4, 160 x 40k 41 / 47, 2D 160 x 40k 260 / 206
// On the 536 the engine chosen takes 3% more than the fastest in the geometric mean
// and is 1.34 times faster than the choice between phase kernels and per-CTA solver
// by size alone; on eleven it is 3 to 13% slower than that.  On 70 others, drawn after
// the fit, 1.40 times and at worst 2% slower.
// (Clusters of a size that gave every SM work, whatever the systems' size, took 2.1
// times the phase kernels' time on 2D 2 x 150k, 2.0 on Q1 16 x 150k.)
// An SM's time goes with a system's nonzeros and, at the vectors' passes, its rows.
constexpr double PHASES_US = 15.5, PHASES_US_PER_OP = 2.1e-6, PHASES_US_PER_OP_TAIL = 3.05e-6,
                 PHASES_BYTES_PER_US32 = 2.8e6;
constexpr double CTA_US = 5.9, CTA_US_PER_NZ = 2.05e-4, CTA_US_PER_OP32 = 1.3e-4;
constexpr double CLUSTER_US = 6.0, CLUSTER_US_PER_NZ = 2.35e-4;
constexpr double PARTS_US = 8.4, PARTS_US_PER_NZ = 2.6e-4;
constexpr int64_t CTA_ROW_NZ = 11, CLUSTER_ROW_NZ = 16, PARTS_ROW_NZ = 11;  // nonzeros a row counts as
constexpr double UNLIKE = 0.57, UNLIKE_SHARE = 1.3, UNLIKE_SIZE = 0.8;
constexpr int64_t TEAM_BATCH_ROWS = 10240;  // rows a CTA of an unlike batch's clusters,
constexpr int64_t UNLIKE_ROWS = 40000;      // ... which take systems of up to so many

// The makespan of n systems on k machines that take them in the solvers' order as
// they fall free; us(q): system q's time on one.  Where it cannot be below limit, a
// lower bound that is not either.
template <class F>
static double makespan(int64_t n, int64_t k, double limit, F us) {
  k = std::min(std::max<int64_t>(k, 1), n);
  double sum = 0.0, most = 0.0;
  for (int64_t q = 0; q < n; ++q) {
    const double t = us(q);
    sum += t;
    most = std::max(most, t);
  }
  if (n <= k || std::max(most, sum / (double)k) >= limit) return std::max(most, sum / (double)k);
  std::vector<double> busy((size_t)k, 0.0);  // a heap: the machine that falls free first in front
  double end = 0.0;
  for (int64_t q = 0; q < n; ++q) {
    std::pop_heap(busy.begin(), busy.end(), std::greater<double>());
    busy.back() += us(q);
    end = std::max(end, busy.back());
    std::push_heap(busy.begin(), busy.end(), std::greater<double>());
  }
  return end;
}

typedef void (*BatchKernel)(PcgArgs, int32_t, int32_t);

// The launch of clusters of `size` CTAs for A's batch, and how many of them are
// resident at once (0: none) -- a matter of the kernel and the device alone, asked
// for once.
struct ClusterLaunch {
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute at[1];
  BatchKernel kernel;
  int fit;
};
static int cluster_launch(gbs_mat A, int size, ClusterLaunch &L) {
  const int64_t per = (A->max_sys_rows / 32 + size) / size * 32;
  L.kernel = per <= 1024 ? k_team_batch<512> : k_team_batch<1024>;
  memset(&L.lc, 0, sizeof(L.lc));
  memset(L.at, 0, sizeof(L.at));
  L.lc.gridDim = dim3((unsigned)(sm_count(A) / size * size));
  L.lc.blockDim = dim3(per <= 1024 ? 512u : 1024u);
  L.lc.dynamicSmemBytes = TEAM_SMEM;
  L.lc.attrs = L.at;
  L.lc.numAttrs = 1;
  L.at[0].id = cudaLaunchAttributeClusterDimension;
  L.at[0].val.clusterDim.x = (unsigned)size;
  L.at[0].val.clusterDim.y = L.at[0].val.clusterDim.z = 1;
  GBS_TRY_CUDA(cudaFuncSetAttribute(L.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)TEAM_SMEM));
  GBS_TRY_CUDA(cudaFuncSetAttribute(L.kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  static std::mutex mu;
  static std::map<std::tuple<int, int, unsigned>, int> known;
  std::lock_guard<std::mutex> lk(mu);
  const auto key = std::make_tuple(A->device, size, L.lc.blockDim.x);
  const auto at = known.find(key);
  if (at != known.end()) {
    L.fit = at->second;
    return GBS_OK;
  }
  if (cudaOccupancyMaxActiveClusters(&L.fit, L.kernel, &L.lc) != cudaSuccess) {
    cudaGetLastError();
    L.fit = 0;
  }
  known[key] = L.fit;
  return GBS_OK;
}

// Nonzeros plus per_row a row of the q-th system in the solvers' order.
static int64_t system_cost(gbs_mat A, int64_t q, int64_t per_row) {
  const int32_t sy = A->cta_order_h[q];
  return A->sys_nnz_h[q] + per_row * (A->row_off_h[sy + 1] - A->row_off_h[sy]);
}

// The first CTAs of the systems on the shared grid: one CTA each, then every
// further one to the system whose CTAs have the most to do.
static std::vector<int16_t> share_out(gbs_mat A) {
  const size_t n = A->cta_order_h.size();
  std::vector<int64_t> ops(n);
  for (size_t q = 0; q < n; ++q) ops[q] = system_cost(A, (int64_t)q, PARTS_ROW_NZ);
  std::vector<int16_t> size(n, 1), first(n + 1, 0);
  for (int64_t k = (int64_t)n; k < sm_count(A); ++k) {
    size_t most = 0;
    for (size_t q = 1; q < n; ++q)
      if (ops[q] * size[most] > ops[most] * size[q]) most = q;
    size[most] += 1;
  }
  for (size_t q = 0; q < n; ++q) first[q + 1] = (int16_t)(first[q] + size[q]);
  return first;
}

// Makes the choice for A's plan (kept until the plan changes).
int batch_choice(gbs_mat A) {
  if (A->batch_engine[0] >= 0) return GBS_OK;
  const int64_t n = A->nsys;
  A->batch_team = BATCH_PHASES;
  A->batch_cluster = 0;
  A->batch_parts.clear();
  if (A->nsys >= 2 * sm_count(A)) {  // (two per-CTA solvers an SM: cta_size_rule)
    A->batch_engine[0] = A->batch_engine[1] = BATCH_CTA;
    return GBS_OK;
  }
  // iterations: its for the engines that advance every system at once, queued for
  // those that take them from a queue
  std::vector<double> its(n), queued(n);
  std::vector<int64_t> ops(n);
  for (int64_t q = 0; q < n; ++q) ops[q] = system_cost(A, q, 8);
  const auto ends = std::minmax_element(ops.begin(), ops.end());
  const bool unlike = 4 * *ends.second > 5 * *ends.first;
  double most_its = 1e-9, work = 0.0;
  for (int64_t q = 0; q < n; ++q) {
    const int32_t sy = A->cta_order_h[q];
    its[q] = pow((double)(A->row_off_h[sy + 1] - A->row_off_h[sy]), 0.385);
    queued[q] = unlike && (q & 1) ? UNLIKE * its[q] : its[q];
    most_its = std::max(most_its, its[q]);
    work += its[q] * (double)ops[q];
  }
  double team_us = 1e300;
  if (A->nsys >= 2 && A->nslices > 0 && A->nnz > 0) {
    // rows of uneven lengths: the CTA with the longest keeps its team waiting
    const double uneven = std::max(1.0, (double)A->run_uneven / (1.25 * RUN_EVEN));
    int small = 2;
    if (unlike)
      while (small < TEAM_MAX_CLUSTER && ((int64_t)A->nsys * small < sm_count(A) ||
                                          A->max_sys_rows > TEAM_BATCH_ROWS * small))
        small *= 2;
    for (int size = small; size <= TEAM_MAX_CLUSTER; size *= 2) {
      if (unlike && A->max_sys_rows > UNLIKE_ROWS) break;
      ClusterLaunch L;
      GBS_TRY(cluster_launch(A, size, L));
      if (L.fit < 1) continue;
      const double below = (unlike && size > small ? UNLIKE_SIZE : 1.0) * team_us;
      const double us = makespan(n, L.fit, below, [&](int64_t q) {
        return queued[q] * (CLUSTER_US + uneven * CLUSTER_US_PER_NZ *
                                             (double)system_cost(A, q, CLUSTER_ROW_NZ) / size);
      });
      if (us >= below) continue;
      team_us = us;
      A->batch_team = BATCH_CLUSTER;
      A->batch_cluster = size;
    }
    if (A->nsys <= TEAM_PARTS_MAX && A->nsys <= sm_count(A)) {
      A->batch_parts = share_out(A);
      double us = 0.0;
      for (int64_t q = 0; q < n; ++q)
        us = std::max(us, its[q] * (PARTS_US + uneven * PARTS_US_PER_NZ *
                                                   (double)system_cost(A, q, PARTS_ROW_NZ) /
                                                   (A->batch_parts[q + 1] - A->batch_parts[q])));
      if (unlike) us *= UNLIKE_SHARE;
      if (us < team_us) {
        team_us = us;
        A->batch_team = BATCH_PARTS;
      }
    }
  }
  const double op = A->ta.nblocks <= A->ta.grid ? PHASES_US_PER_OP : PHASES_US_PER_OP_TAIL;
  const double phases[2] = {
      PHASES_US * most_its + op * work,
      most_its * (PHASES_US + (4.0 * (double)A->nnz + 44.0 * (double)A->nrows) / PHASES_BYTES_PER_US32)};
  for (int refined = 0; refined < 2; ++refined) {
    const double cta = makespan(n, sm_count(A), phases[refined], [&](int64_t q) {
      return queued[q] * (CTA_US + (refined ? CTA_US_PER_OP32 * (double)ops[q]
                                            : CTA_US_PER_NZ * (double)system_cost(A, q, CTA_ROW_NZ)));
    });
    int32_t e = cta < phases[refined] ? BATCH_CTA : BATCH_PHASES;
    if (!refined && team_us < std::min(cta, phases[0])) e = A->batch_team;
    A->batch_engine[refined] = e;
  }
  return GBS_OK;
}

// FP64 CG, and the solver left to the automatic choice: an explicit solver, plan or
// single-reduction form is what the caller asked for.  team_tuned: the autotuner
// measured the team fastest.
static bool team_allowed(gbs_mat A, const ksp_opts &o) {
  return o.method == GBS_KSP_CG && o.precision == GBS_FP64 && !o.host_loop &&
         A->lanes == GBS_SPMV_SELL && A->nrows > 0 &&
         (A->team_tuned ||
          (A->solver == GBS_SOLVER_AUTO && A->cg_form == GBS_CG_TEXTBOOK && A->plan_auto));
}

// How a batch runs under the automatic choice (batch_choice), or, tuned for
// teams, the better of theirs.
int32_t batch_team(gbs_mat A, const ksp_opts &o) {
  if (!team_allowed(A, o) || A->nsys < 2 || batch_choice(A) != GBS_OK) return BATCH_PHASES;
  const int32_t e = A->team_tuned ? A->batch_team : A->batch_engine[0];
  return e == BATCH_CLUSTER || e == BATCH_PARTS ? e : BATCH_PHASES;
}
bool batch_teams(gbs_mat A) {
  return A->nsys >= 2 && batch_choice(A) == GBS_OK && A->batch_team != BATCH_PHASES;
}

bool use_team(gbs_mat A, bool per_system, const ksp_opts &o) {
  if (per_system) return batch_team(A, o) != BATCH_PHASES;
  return A->nsys == 1 && team_allowed(A, o) && (A->team_tuned || team_suits(A));
}

// The team of a solve on A: its CTAs, their threads and their shared memory.
struct TeamShape {
  TeamCfg cfg;
  bool cluster;
  int size, tpb;
  size_t smem;
};

static TeamShape team_shape(gbs_mat A) {
  TeamShape T;
  memset(&T, 0, sizeof(T));
  TeamCfg &c = T.cfg;
  const int64_t n = A->nrows, ns = A->nslices;
  T.cluster = A->nnz + 8 * n <= TEAM_CLUSTER_WORK;
  T.size = T.cluster ? TEAM_MAX_CLUSTER : sm_count(A);
  while (T.size > 1 && ns < T.size) T.size = (T.size + 1) / 2;  // every CTA has a slice
  const int64_t per = (ns + T.size - 1) / T.size, rows = 32 * per;
  T.tpb = rows <= 256 ? 256 : 512;
  c.rows_cap = (int32_t)rows;
  int64_t left = TEAM_SMEM - 16 * T.tpb;
  // windows where the halo's extra work (one FMA a row, two rows a clock) stays
  // below the meeting they save
  const auto up32 = [](int64_t k) { return (k + 31) & ~(int64_t)31; };
  const int64_t halo = std::min<int64_t>(A->col_span, n), win = up32(std::min(n, rows + 2 * halo));
  const int64_t zh = T.cluster ? up32(std::min(2 * halo, n)) : 0;
  const bool window = 2 * halo <= std::max<int64_t>(rows, 4096) && 8 * (win + zh) <= left / 3;
  const int64_t per_entry = A->sell_npat ? 8 : (A->col_span <= 32767 ? 10 : 12);
  const int64_t mat = A->sell_nnz / ns * per * per_entry * 9 / 8 +
                      per * (136 + (A->sell_npat ? 256 : 0)) + 1024;
  const int nv = window ? 5 : 4;
  const int64_t used = (window ? 8 * (win + zh) : 0) + nv * 8 * rows;
  if (used + mat <= left) {  // vectors, windows and matrix all stay
    c.nvec = nv;
    c.mat_cap = (int32_t)std::min<int64_t>((left - used) & ~(int64_t)15,
                                           (mat + 1023) & ~(int64_t)1023);
    if (window) {
      c.window = 1;
      c.halo = (int32_t)halo;
      c.win_cap = (int32_t)win;
      c.zh_cap = (int32_t)zh;
    }
  } else {
    // the matrix streams past: every thread the registers allow, to have loads
    // in flight (2D 1024^2, us an iteration: 1024 threads 35.1, 512 40.3), and
    // p gathered through L1 rather than from windows (35.1 against 36.9)
    if (!T.cluster) T.tpb = 1024;
    c.nvec = (int32_t)std::min<int64_t>(4, TEAM_L1_SMEM / (8 * rows));
  }
  T.smem = (size_t)(16 * T.tpb + 8 * (c.win_cap + c.zh_cap) + c.nvec * 8 * rows + c.mat_cap);
  return T;
}

// Batches on teams; *ran stays false (and nothing has started) where the device
// cannot hold a team at once.
static int solve_clusters(gbs_mat A, const double *b, double *x, const ksp_opts &o,
                          cudaStream_t s, bool *ran) {
  ClusterLaunch L;
  GBS_TRY(cluster_launch(A, A->batch_cluster, L));
  if (L.fit < 1) return GBS_OK;
  L.lc.stream = s;
  L.lc.gridDim = dim3((unsigned)(std::min<int64_t>(L.fit, A->nsys) * A->batch_cluster));
  PcgArgs a = make_args(A, true, false);
  a.stream_matrix = 0;  // (a system's matrix is read again by the same SMs, from L2)
  a.order = A->cta_order;
  a.cta_n = A->nsys;
  GBS_TRY_CUDA(cudaMemsetAsync(A->ctl, 0, sizeof(DevCtl), s));
  GBS_TRY(put_call(A->call, call_args(b, x, o), s, A->ctl));
  GBS_TRY_CUDA(cudaLaunchKernelEx(&L.lc, L.kernel, a, A->col_span, (int32_t)TEAM_SMEM));
  count_launches(1);
  *ran = true;
  return GBS_OK;
}

static int solve_parts(gbs_mat A, const double *b, double *x, const ksp_opts &o,
                       cudaStream_t s, bool *ran) {
  TeamParts parts;
  memset(&parts, 0, sizeof(parts));
  // the largest part's rows, and whether every part keeps its matrix and vectors
  int64_t rows = 0, bytes = 0;
  const int64_t per_entry = A->sell_npat ? 8 : (A->col_span <= 32767 ? 10 : 12);
  for (int32_t k = 0; k < A->nsys; ++k) {
    parts.first[k] = A->batch_parts[k];
    const int32_t q = A->cta_order_h[k];
    const int64_t size = A->batch_parts[k + 1] - A->batch_parts[k];
    const int64_t per = (A->sell_slice0_h[q + 1] - A->sell_slice0_h[q] + size - 1) / size;
    const int64_t halo = std::min<int64_t>(A->col_span, A->row_off_h[q + 1] - A->row_off_h[q]);
    rows = std::max(rows, 32 * per);
    bytes = std::max(bytes, per * (32 * 5 * 8 + (A->slice_max_nnz * per_entry) * 9 / 8 + 136 +
                                   (A->sell_npat ? 256 : 0)) + 16 * std::max(32 * per, halo));
  }
  parts.first[A->nsys] = A->batch_parts[A->nsys];
  const bool streams = bytes > TEAM_SMEM - 16 * 512;
  const int tpb = streams ? 1024 : 512;
  const int64_t smem = streams ? 16 * tpb + std::min<int64_t>(4, TEAM_L1_SMEM / (8 * rows)) * 8 * rows
                               : TEAM_SMEM;
  void (*const kernel)(PcgArgs, TeamParts, int32_t, int32_t, int32_t, unsigned *, double *,
                       unsigned, int64_t) =
      streams ? k_team_parts<1024> : k_team_parts<512>;
  GBS_TRY_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)TEAM_SMEM));
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute at[1];
  memset(&lc, 0, sizeof(lc));
  memset(at, 0, sizeof(at));
  lc.gridDim = dim3((unsigned)parts.first[A->nsys]);
  lc.blockDim = dim3((unsigned)tpb);
  lc.dynamicSmemBytes = (size_t)smem;
  lc.stream = s;
  lc.attrs = at;
  lc.numAttrs = 1;
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  PcgArgs a = make_args(A, true, false);
  a.stream_matrix = stream_matrix(A, 8);
  a.order = A->cta_order;
  a.cta_n = A->nsys;
  // slots: four doubles a CTA; then the teams' counters (ensure_solver_workspace)
  unsigned *const ctr = reinterpret_cast<unsigned *>(A->part + 4 * sm_count(A));
  GBS_TRY_CUDA(cudaMemsetAsync(ctr, 0, sizeof(unsigned) * TEAM_CTR_STRIDE * A->nsys, s));
  GBS_TRY_CUDA(cudaMemsetAsync(A->ctl, 0, sizeof(DevCtl), s));
  GBS_TRY(put_call(A->call, call_args(b, x, o), s, A->ctl));
  const cudaError_t e = cudaLaunchKernelEx(&lc, kernel, a, parts, A->col_span, (int32_t)smem,
                                           (int32_t)streams, ctr, A->part, TEAM_WAIT_POLLS,
                                           TEAM_WAIT_NS);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorLaunchOutOfResources) {
    cudaGetLastError();
    return GBS_OK;
  }
  GBS_TRY_CUDA(e);
  count_launches(1);
  *ran = true;
  return GBS_OK;
}

int solve_team(gbs_mat A, const double *b, double *x, const ksp_opts &o, bool per_system,
               cudaStream_t s, bool *ran) {
  *ran = false;
  if (per_system)
    return batch_team(A, o) == BATCH_PARTS ? solve_parts(A, b, x, o, s, ran)
                                           : solve_clusters(A, b, x, o, s, ran);
  TeamShape T = team_shape(A);
  PcgArgs a = make_args(A, false, false);
  a.stream_matrix = stream_matrix(A, 8);
  T.cfg.slots = A->part;
  T.cfg.ctr = reinterpret_cast<unsigned *>(&A->ctl->queue);
  T.cfg.wait_polls = TEAM_WAIT_POLLS;
  T.cfg.wait_ns = TEAM_WAIT_NS;
  void (*const kernel)(PcgArgs, TeamCfg) =
      T.cluster ? k_team<false, 512> : T.tpb <= 512 ? k_team<true, 512> : k_team<true, 1024>;
  GBS_TRY_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)TEAM_SMEM));
  cudaLaunchConfig_t lc = {};
  cudaLaunchAttribute at[1];
  memset(at, 0, sizeof(at));
  lc.gridDim = dim3((unsigned)T.size);
  lc.blockDim = dim3((unsigned)T.tpb);
  lc.dynamicSmemBytes = T.smem;
  lc.stream = s;
  lc.attrs = at;
  lc.numAttrs = 1;
  if (T.cluster) {
    GBS_TRY_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)T.size;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  GBS_TRY_CUDA(cudaMemsetAsync(A->ctl, 0, sizeof(DevCtl), s));
  GBS_TRY(put_call(A->call, call_args(b, x, o), s, A->ctl));
  const cudaError_t e = cudaLaunchKernelEx(&lc, kernel, a, T.cfg);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorInvalidClusterSize ||
      e == cudaErrorLaunchOutOfResources) {
    cudaGetLastError();
    return GBS_OK;
  }
  GBS_TRY_CUDA(e);
  count_launches(1);
  *ran = true;
  return GBS_OK;
}

}  // namespace gbs
