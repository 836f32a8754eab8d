// Coarse-grid solver of the all-at-once multigrid (Sec. 3.7) as a routine of
// one team (a thread-block cluster, or one block; hhg_team.cuh): MINRES on the
// full saddle-point system, preconditioned block-diagonally (Sec. 3.2) with a
// CG solve on each velocity block of A and the inverse lumped pressure mass.
// Always FP64, on the compact unknown vector x = (u_0, u_1, u_2, p) of the
// coarsest level with K and A in CSR (CoarseSys), so no work is spent on the
// ghost frame, Dirichlet nodes or inactive nodes of the lattice.  Loops have
// fixed upper trip counts (max iterations).  Used by the coarse-solve kernel
// and by the fused coarse-levels cycle.
//
// Row products and dot products are chains of fused multiply-adds in row
// order, and the sums of the team have a fixed order (hhg_team.cuh): an
// inexact solve amplifies its rounding, so the order is part of the result.
//
// Recurrences (start from zero):
//   CG:     stop before an iteration when r.r <= rtol^2 r0.r0 (or r.r = 0),
//           or when d.Ad = 0; at most cg_max iterations.
//   MINRES: Lanczos with Givens rotations; z_j <- z_j / gamma_j,
//           delta_j = (K z_j).z_j, v_{j+1} = K z_j - delta_j/gamma_j v_j
//           - gamma_j/gamma_{j-1} v_{j-1}, z_{j+1} = P^{-1} v_{j+1},
//           gamma_{j+1} = sqrt(z_{j+1}.v_{j+1}); rotation a0..a3, c, s;
//           w_{j+1} = (z_j - a3 w_{j-1} - a2 w_j)/a1; x += c_{j+1} eta w_{j+1};
//           eta <- -s_{j+1} eta; stop when |eta| <= rtol gamma_1.
#pragma once
#include "hhg_kernels.h"
#include "hhg_team.cuh"

namespace hhg {
namespace coarse {

struct Ctx {
  CoarseSys S;
  Team T;
  int n;  // 3 nv + np
};

__device__ __forceinline__ double csr_row(const int32_t* ptr, const int32_t* col, const double* val, int r,
                                          const double* x) {
  double s = 0.0;
  const int e = ptr[r + 1];
  for (int k = ptr[r]; k < e; ++k) s = fma(val[k], x[col[k]], s);
  return s;
}

// This thread's part of a.b.
__device__ __forceinline__ double dot_part(const Ctx& C, const double* a, const double* b) {
  double s = 0;
  for (int q = (int)C.T.rank(); q < C.n; q += (int)C.T.size()) s = fma(a[q], b[q], s);
  return s;
}

// y = K x
__device__ inline void applyK(const Ctx& C, const double* x, double* y) {
  for (int r = (int)C.T.rank(); r < C.n; r += (int)C.T.size()) y[r] = csr_row(C.S.kptr, C.S.kcol, C.S.kval, r, x);
  C.T.sync();
}

// ---- team CG -----------------------------------------------------------------
// x_s = CG(A, b_s) from zero for NSYS systems in lockstep over the team: the
// three velocity components with the scalar A (NSYS = 3, N = nv rows each) or
// the coupled block of the D form and of free slip (NSYS = 1, N = 3 nv rows).
// Each system follows the stopping rule of a single CG on its own (it stops
// before an iteration when r.r <= rtol^2 r0.r0 or r.r = 0, or when d.Ad = 0);
// the others go on.  b, x: NSYS N entries.  Returns the iterations summed
// over the systems.
//
// cg_team_regs: a CTA holds a run of groups of 32 rows of every system and a
// warp at most one (system, group), a row per lane, whose x, r, d, A d and
// first CG_ROW matrix entries (with the addresses of their directions) stay
// in registers.  The directions lie in the shared memory of their CTAs, dir,
// and are read through the cluster's shared window.  An iteration is three
// cluster barriers: d.Ad, r.r and the new directions.  It is bound by the
// latencies of the FP64 chain (64 cycles per dependent operation, 560 per
// division) and of the barriers (480 cycles each): on the obstacle channel's
// level 1 (1,427 rows, 16 CTAs) an iteration takes 5.5 us, against 27 us
// with every thread evaluating the scalars and the vectors in global memory.
constexpr int CG_ROW = COARSE_ELL_ROUND;

template <int NSYS>
__device__ __noinline__ int cg_team_regs(const Ctx& C, const double* b, double* x, double* dir, int max_it,
                                         double rtol) {
  const Team T = C.T;  // local copies: the context is in memory
  const int N = NSYS == 3 ? C.S.nv : 3 * C.S.nv;
  const int groups = (N + 31) / 32;
  const int each = (groups + (int)T.nblocks - 1) / (int)T.nblocks;  // groups of a system per CTA
  const int rc = 32 * each;                                            // its rows
  const int warp = threadIdx.x >> 5, sys = warp / each;
  const bool used = sys < NSYS;
  const int mine = used ? sys : 0;
  const int l = (int)threadIdx.x - sys * rc;  // row within the CTA
  const int row = (int)blockIdx.x * rc + l, group = row >> 5;
  const bool live = used && group < groups;   // (uniform in the warp)
  const bool on = live && row < N;
  const int idx = on ? sys * N + row : -1;
  const uint32_t dir0 = (uint32_t)__cvta_generic_to_shared(dir) + 8u * (uint32_t)(mine * rc);
  const uint32_t inv = 0xffffffffu / (uint32_t)rc + 1u;  // col / rc = umulhi(col, inv): col, rc < 2^13
  auto addr_of = [&](int col) {
    const uint32_t o = __umulhi((uint32_t)col, inv);
    return team_shared_addr(dir0 + 8u * ((uint32_t)col - o * (uint32_t)rc), o);
  };
  // entries of the warp's longest row (the others' absent ones are zeros on
  // their own directions; a thread without a row reads row 0 and drops it)
  const int len = __reduce_max_sync(0xffffffffu, on ? C.S.aptr[row + 1] - C.S.aptr[row] : 0);
  const double* ev = C.S.eval + (on ? row : 0);
  const int32_t* ec = C.S.ecol + (on ? row : 0);
  double av[CG_ROW];
  uint32_t ad[CG_ROW];
#pragma unroll
  for (int e = 0; e < CG_ROW; ++e) {
    av[e] = ev[(int64_t)e * N];
    ad[e] = addr_of(ec[(int64_t)e * N]);
  }
  double xv = 0.0, qv = 0.0, rv = on ? b[idx] : 0.0, dv = rv;
  if (used) dir[mine * rc + l] = dv;
  // state of the handler warps: r.r, the stopping bound, running, iterations
  double rr = 0.0, stop = 0.0;
  bool run = false;
  int its = 0;
  if (live) team_publish(T, rv * rv, mine, group);
  double res[2 * NSYS];
  team_finish<NSYS, 2>(T, groups, res, [&](double tot, double* out) {
    rr = tot;
    stop = rtol * rtol * tot;
    run = !(rr <= stop || rr == 0.0);
    out[0] = run ? 1.0 : 0.0;
    out[1] = 0.0;
  });
  for (int it = 0; it < max_it; ++it) {
    // the directions are published: by the sum above (first iteration) or the barrier below
    bool any = false;
#pragma unroll
    for (int s = 0; s < NSYS; ++s) any |= res[2 * s] != 0.0;
    if (!any) break;
    bool go = live && res[2 * mine] != 0.0;
    if (go) {
      double dn[CG_ROW];
#pragma unroll
      for (int e = 0; e < CG_ROW; ++e) dn[e] = ld_team_shared(ad[e]);
      qv = 0.0;
#pragma unroll
      for (int e = 0; e < CG_ROW; ++e)
        if (e < len) qv = fma(av[e], dn[e], qv);
      for (int k = CG_ROW; k < len; k += CG_ROW) {
        double a[CG_ROW];
        uint32_t at[CG_ROW];
#pragma unroll
        for (int e = 0; e < CG_ROW; ++e) {
          a[e] = __ldg(ev + (int64_t)(k + e) * N);
          at[e] = addr_of(__ldg(ec + (int64_t)(k + e) * N));
        }
#pragma unroll
        for (int e = 0; e < CG_ROW; ++e) dn[e] = ld_team_shared(at[e]);
#pragma unroll
        for (int e = 0; e < CG_ROW; ++e)
          if (k + e < len) qv = fma(a[e], dn[e], qv);
      }
      if (!on) qv = 0.0;
      team_publish(T, dv * qv, mine, group);
    }
    team_finish<NSYS, 2>(T, groups, res, [&](double tot, double* out) {
      if (run && tot == 0.0) run = false;
      out[0] = run ? 1.0 : 0.0;
      out[1] = run ? rr / tot : 0.0;
    });
    go = go && res[2 * mine] != 0.0;
    if (go) {
      const double alpha = res[2 * mine + 1];
      rv = fma(-alpha, qv, rv);
      team_publish(T, rv * rv, mine, group);
      xv = fma(alpha, dv, xv);
    }
    team_finish<NSYS, 2>(T, groups, res, [&](double tot, double* out) {
      out[0] = out[1] = 0.0;
      if (run) {
        out[1] = tot / rr;
        rr = tot;
        ++its;
        run = !(rr <= stop || rr == 0.0);
        out[0] = run ? 1.0 : 0.0;
      }
    });
    if (go) {
      dv = fma(res[2 * mine + 1], dv, rv);
      dir[mine * rc + l] = dv;
    }
    T.sync();
  }
  if (on) x[idx] = xv;
  team_finish<NSYS, 1>(T, 0, res, [&](double, double* out) { out[0] = (double)its; });
  double n = 0.0;
#pragma unroll
  for (int s = 0; s < NSYS; ++s) n += res[s];
  C.T.calls = T.calls;
  return (int)n;
}

// The same for any number of rows per thread, on vectors in global memory
// (cg: r, d and A d, NSYS N entries each); a thread takes its rows in every
// system.
template <int NSYS>
__device__ __noinline__ int cg_team_mem(const Ctx& C, const double* b, double* x, double* cg, int max_it,
                                        double rtol) {
  const Team T = C.T;  // local copies: the context is in memory
  const int N = NSYS == 3 ? C.S.nv : 3 * C.S.nv;
  const int32_t *aptr = C.S.aptr, *acol = C.S.acol;
  const double* aval = C.S.aval;
  double* R = cg;
  double* D = cg + NSYS * N;
  double* Q = cg + 2 * NSYS * N;
  const int t0 = (int)T.rank(), step = (int)T.size();
  const int group = t0 >> 5, groups = (min(N, step) + 31) / 32;
  auto publish = [&](const double (&v)[NSYS]) {
    if (group < groups)
#pragma unroll
      for (int s = 0; s < NSYS; ++s) team_publish(T, v[s], s, group);
  };
  double acc[NSYS];
#pragma unroll
  for (int s = 0; s < NSYS; ++s) acc[s] = 0.0;
  for (int q = t0; q < N; q += step)
#pragma unroll
    for (int s = 0; s < NSYS; ++s) {
      const double v = b[s * N + q];
      x[s * N + q] = 0.0;
      R[s * N + q] = v;
      D[s * N + q] = v;
      acc[s] = fma(v, v, acc[s]);
    }
  double rr = 0.0, stop = 0.0;
  bool run = false;
  int its = 0;
  publish(acc);
  double res[2 * NSYS];
  team_finish<NSYS, 2>(T, groups, res, [&](double tot, double* out) {
    rr = tot;
    stop = rtol * rtol * tot;
    run = !(rr <= stop || rr == 0.0);
    out[0] = run ? 1.0 : 0.0;
    out[1] = 0.0;
  });
  for (int it = 0; it < max_it; ++it) {
    bool any = false;
#pragma unroll
    for (int s = 0; s < NSYS; ++s) any |= res[2 * s] != 0.0;
    if (!any) break;
#pragma unroll
    for (int s = 0; s < NSYS; ++s) {
      acc[s] = 0.0;
      if (res[2 * s] == 0.0) continue;
      for (int q = t0; q < N; q += step) {
        const double aq = csr_row(aptr, acol, aval, q, D + s * N);
        Q[s * N + q] = aq;
        acc[s] = fma(D[s * N + q], aq, acc[s]);
      }
    }
    publish(acc);
    team_finish<NSYS, 2>(T, groups, res, [&](double tot, double* out) {
      if (run && tot == 0.0) run = false;
      out[0] = run ? 1.0 : 0.0;
      out[1] = run ? rr / tot : 0.0;
    });
    bool go[NSYS];
#pragma unroll
    for (int s = 0; s < NSYS; ++s) {
      go[s] = res[2 * s] != 0.0;
      const double alpha = res[2 * s + 1];
      acc[s] = 0.0;
      if (go[s])
        for (int q = t0; q < N; q += step) {
          x[s * N + q] += alpha * D[s * N + q];
          const double rq = R[s * N + q] - alpha * Q[s * N + q];
          R[s * N + q] = rq;
          acc[s] = fma(rq, rq, acc[s]);
        }
    }
    publish(acc);
    team_finish<NSYS, 2>(T, groups, res, [&](double tot, double* out) {
      out[0] = out[1] = 0.0;
      if (run) {
        out[1] = tot / rr;
        rr = tot;
        ++its;
        run = !(rr <= stop || rr == 0.0);
        out[0] = run ? 1.0 : 0.0;
      }
    });
#pragma unroll
    for (int s = 0; s < NSYS; ++s)
      if (go[s]) {
        const double beta = res[2 * s + 1];
        for (int q = t0; q < N; q += step) D[s * N + q] = R[s * N + q] + beta * D[s * N + q];
      }
    T.sync();
  }
  team_finish<NSYS, 1>(T, 0, res, [&](double, double* out) { out[0] = (double)its; });
  double n = 0.0;
#pragma unroll
  for (int s = 0; s < NSYS; ++s) n += res[s];
  C.T.calls = T.calls;
  return (int)n;
}

// Team CG of the preconditioner; cg: 9 nv entries of global scratch, dir:
// team_dirs entries of shared memory.  One row per lane covers nv <= 2,560 on
// 16 CTAs of 512 threads.
template <int NSYS>
__device__ inline int cg_team(const Ctx& C, const double* b, double* x, double* cg, double* dir, int max_it,
                              double rtol) {
  const int N = NSYS == 3 ? C.S.nv : 3 * C.S.nv;
  if (N == 0) return 0;  // no velocity unknown (the unit cube's level 0): A has no rows
  const int each = ((N + 31) / 32 + (int)C.T.nblocks - 1) / (int)C.T.nblocks;
  if (C.S.eval && 32 * NSYS * each <= min((int)blockDim.x, team_dirs(C.T.nblocks)))
    return cg_team_regs<NSYS>(C, b, x, dir, max_it, rtol);
  return cg_team_mem<NSYS>(C, b, x, cg, max_it, rtol);
}

// The coupled block on one thread block (few rows: vectors and matrix in
// L1), every thread evaluating the scalars.  block_sum: the groups of 32
// values in order, as team_finish forms them.
__device__ __forceinline__ double block_sum(const Team& T, double x) {
  double* part = T.part(T.calls & 1u, 0);
  ++T.calls;
  x = warp_sum(x);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
  __syncthreads();
  double tot = part[0];
  for (int g = 1; g < (int)(blockDim.x >> 5); ++g) tot += part[g];
  return tot;
}

__device__ inline int cg_coupled_block(const Ctx& C, const double* b, double* x, double* cg, int max_it, double rtol) {
  const int n = 3 * C.S.nv;
  double* R = cg;
  double* D = cg + n;
  double* Q = cg + 2 * n;
  double rr = 0.0;
  for (int q = (int)threadIdx.x; q < n; q += (int)blockDim.x) {
    x[q] = 0.0;
    R[q] = b[q];
    D[q] = b[q];
    rr = fma(b[q], b[q], rr);
  }
  rr = block_sum(C.T, rr);
  const double stop = rtol * rtol * rr;
  int it = 0;
  for (; it < max_it; ++it) {
    if (rr <= stop || rr == 0.0) break;
    double dq = 0.0;
    for (int q = (int)threadIdx.x; q < n; q += (int)blockDim.x) {
      const double aq = csr_row(C.S.aptr, C.S.acol, C.S.aval, q, D);
      Q[q] = aq;
      dq = fma(D[q], aq, dq);
    }
    dq = block_sum(C.T, dq);
    if (dq == 0.0) break;
    const double alpha = rr / dq;
    double rn = 0.0;
    for (int q = (int)threadIdx.x; q < n; q += (int)blockDim.x) {
      x[q] = fma(alpha, D[q], x[q]);
      const double rq = fma(-alpha, Q[q], R[q]);
      R[q] = rq;
      rn = fma(rq, rq, rn);
    }
    rn = block_sum(C.T, rn);
    const double beta = rn / rr;
    for (int q = (int)threadIdx.x; q < n; q += (int)blockDim.x) D[q] = fma(beta, D[q], R[q]);
    __syncthreads();
    rr = rn;
  }
  return it;
}

// ---- warp-level CG: the three velocity blocks are solved concurrently ------

// x = CG(A, b) from zero by one warp (the same stopping rule), up to NR rows
// per lane with x, r, d, A d and the first CG_ROW entries of each row in
// registers; dir: the search direction in shared memory, nv entries of this
// warp.  One lane per row and a butterfly per sum; an iteration of the cube's
// level 2 (27 rows) is a chain of 7 row products, two trees of 5 additions
// and two divisions in FP64, 64 cycles per operation and 560 per division.
template <int NR>
__device__ __noinline__ int cg_warp(const CoarseSys& S, const double* b, double* x, double* dir, int max_it, double rtol) {
  const int lane = threadIdx.x & 31, nv = S.nv;
  const double* eval = S.eval;
  const int32_t* ecol = S.ecol;
  constexpr bool KEEP = NR == 1;
  double xv[NR], rv[NR], dv[NR], qv[NR], av[CG_ROW];
  int at[NR], len[NR], ac[CG_ROW];  // a lane without a row reads row 0 and drops it
  double rr = 0.0;
#pragma unroll
  for (int m = 0; m < NR; ++m) {
    const int q = lane + 32 * m;
    const bool on = q < nv;
    at[m] = on ? q : 0;
    len[m] = __reduce_max_sync(0xffffffffu, on ? S.aptr[q + 1] - S.aptr[q] : 0);
    if (KEEP) {
#pragma unroll
      for (int e = 0; e < CG_ROW; ++e) {
        av[e] = eval[e * nv + at[m]];
        ac[e] = ecol[e * nv + at[m]];
      }
    }
    xv[m] = 0.0;
    qv[m] = 0.0;
    rv[m] = dv[m] = on ? b[q] : 0.0;
    if (on) dir[q] = dv[m];
    rr = fma(rv[m], rv[m], rr);
  }
  rr = warp_sum(rr);
  __syncwarp();
  const double stop = rtol * rtol * rr;
  int it = 0;
  for (; it < max_it; ++it) {
    if (rr <= stop || rr == 0.0) break;
    double dq = 0.0;
#pragma unroll
    for (int m = 0; m < NR; ++m) {
      double s = 0.0;
      if (KEEP) {
        double dn[CG_ROW];
#pragma unroll
        for (int e = 0; e < CG_ROW; ++e) dn[e] = dir[ac[e]];
#pragma unroll
        for (int e = 0; e < CG_ROW; ++e)
          if (e < len[m]) s = fma(av[e], dn[e], s);
      }
      for (int k = KEEP ? CG_ROW : 0; k < len[m]; k += CG_ROW) {
        double a[CG_ROW], dn[CG_ROW];
#pragma unroll
        for (int e = 0; e < CG_ROW; ++e) {
          a[e] = __ldg(eval + (k + e) * nv + at[m]);
          dn[e] = dir[__ldg(ecol + (k + e) * nv + at[m])];
        }
#pragma unroll
        for (int e = 0; e < CG_ROW; ++e)
          if (k + e < len[m]) s = fma(a[e], dn[e], s);
      }
      if (lane + 32 * m >= nv) s = 0.0;
      qv[m] = s;
      dq = fma(dv[m], s, dq);
    }
    dq = warp_sum(dq);
    if (dq == 0.0) break;
    const double alpha = rr / dq;
    double rn = 0.0;
#pragma unroll
    for (int m = 0; m < NR; ++m) {
      xv[m] = fma(alpha, dv[m], xv[m]);
      rv[m] = fma(-alpha, qv[m], rv[m]);
      rn = fma(rv[m], rv[m], rn);
    }
    rn = warp_sum(rn);
    const double beta = rn / rr;
    // every lane has read dir before any lane rewrites it (the sums above)
#pragma unroll
    for (int m = 0; m < NR; ++m) {
      dv[m] = fma(beta, dv[m], rv[m]);
      if (lane + 32 * m < nv) dir[lane + 32 * m] = dv[m];
    }
    __syncwarp();
    rr = rn;
  }
#pragma unroll
  for (int m = 0; m < NR; ++m)
    if (lane + 32 * m < nv) x[lane + 32 * m] = xv[m];
  return it;
}

// The same for any number of rows per lane, on vectors in memory (r, d, w: nv
// entries each).  Rows in CSR: side by side (ecol), two at a time, they
// measured between half and 1.4 times the time, as L1 held them or not.
__device__ inline int cg_warp_mem(const CoarseSys& S, const double* b, double* x, double* r, double* d, double* w,
                                  int max_it, double rtol) {
  const int lane = threadIdx.x & 31, nv = S.nv;
  double rr = 0.0;
  for (int q = lane; q < nv; q += 32) {
    x[q] = 0.0;
    r[q] = b[q];
    d[q] = b[q];
    rr = fma(b[q], b[q], rr);
  }
  rr = warp_sum(rr);
  __syncwarp();
  const double stop = rtol * rtol * rr;
  int it = 0;
  for (; it < max_it; ++it) {
    if (rr <= stop || rr == 0.0) break;
    double dq = 0.0;
    for (int q = lane; q < nv; q += 32) {
      const double aq = csr_row(S.aptr, S.acol, S.aval, q, d);
      w[q] = aq;
      dq = fma(d[q], aq, dq);
    }
    dq = warp_sum(dq);
    if (dq == 0.0) break;
    const double alpha = rr / dq;
    double rn = 0.0;
    for (int q = lane; q < nv; q += 32) {
      x[q] = fma(alpha, d[q], x[q]);
      const double rq = fma(-alpha, w[q], r[q]);
      r[q] = rq;
      rn = fma(rq, rq, rn);
    }
    rn = warp_sum(rn);
    const double beta = rn / rr;
    // every lane has read d (the products above) before any lane rewrites it
    __syncwarp();
    for (int q = lane; q < nv; q += 32) d[q] = fma(beta, d[q], r[q]);
    __syncwarp();
    rr = rn;
  }
  return it;
}

// Largest velocity block solved by one warp in the single-block solver, and
// the largest with its vectors in registers (four rows per lane).
constexpr int WARP_CG_MAX_NV = 1024, WARP_CG_REG_NV = 128;

// z = P^{-1} v: CG on each velocity block, lumped mass on the pressure.  On a
// single block with small blocks the three CG solves run concurrently, warp
// w solving block w with warp-level synchronisation only; otherwise the team
// runs them in lockstep (cg_team).  cg holds 9 nv scratch entries.
__device__ inline int precond(const Ctx& C, const double* v, double* z, double* cg, int cg_max, double cg_rtol) {
  __shared__ int its_sh[3];
  double* dir_sh = C.T.dirs();  // directions of the three warp CGs, or of this CTA's rows in the team CG
  int its = 0;
  const int nv = C.S.nv;
  const int warp = threadIdx.x >> 5;
  const bool par = !C.S.coupled && C.T.nblocks == 1 && blockDim.x >= 128 && nv <= WARP_CG_MAX_NV && nv > 0;
  // the pressure part on the warps that no CG keeps busy
  const int skip = par ? 96 : 0;
  const int t0 = par ? (int)threadIdx.x - skip : (int)C.T.rank();
  const int ts = (int)C.T.size() - skip;
  if (t0 >= 0)
    for (int q = t0; q < C.S.np; q += ts) z[3 * nv + q] = v[3 * nv + q] / C.S.mass[q];
  if (C.S.coupled && C.T.nblocks == 1 && blockDim.x <= 128) {
    its = cg_coupled_block(C, v, z, cg, cg_max, cg_rtol);
  } else if (C.S.coupled) {
    its = cg_team<1>(C, v, z, cg, dir_sh, cg_max, cg_rtol);
  } else if (par) {
    if (warp < 3) {
      const double* b = v + warp * nv;
      double* x = z + warp * nv;
      double* dir = dir_sh + warp * WARP_CG_REG_NV;
      double* mem = cg + 3 * warp * nv;
      const int n = nv <= 32               ? cg_warp<1>(C.S, b, x, dir, cg_max, cg_rtol)
                    : nv <= 64             ? cg_warp<2>(C.S, b, x, dir, cg_max, cg_rtol)
                    : nv <= WARP_CG_REG_NV ? cg_warp<4>(C.S, b, x, dir, cg_max, cg_rtol)
                                           : cg_warp_mem(C.S, b, x, mem, mem + nv, mem + 2 * nv, cg_max, cg_rtol);
      if ((threadIdx.x & 31) == 0) its_sh[warp] = n;
    }
  } else {
    its = cg_team<3>(C, v, z, cg, dir_sh, cg_max, cg_rtol);
  }
  C.T.sync();
  if (par) {
    its = its_sh[0] + its_sh[1] + its_sh[2];
    C.T.sync();
  }
  return its;
}

// (U, P) += PMINRES correction of the residual equation (F, G) - K (U, P) on
// the coarsest level L (fields of type T, the solve in FP64); every thread of
// the team must call it.  scratch: coarse_scratch_doubles(S) entries.
template <class T>
__device__ __noinline__ void minres_team(const Team& tm, const CoarseSys& S, const LevelDev<T>& L, double* scratch,
                                   const CoarseParams& prm, double* info) {
  const int nv = S.nv, n = 3 * S.nv + S.np;
  Ctx C{S, tm, n};
  double* vec[11];
  for (int f = 0; f < 11; ++f) vec[f] = scratch + (int64_t)f * n;
  double* cg = scratch + (int64_t)11 * n;
  double *b = vec[0], *x = vec[1], *Kz = vec[2];
  double* vv[3] = {vec[3], vec[4], vec[5]};  // v_prev, v, v_next (rotating)
  double* zz[2] = {vec[6], vec[7]};          // z, z_next
  double* ww[3] = {vec[8], vec[9], vec[10]};  // w_prev, w, w_next

  // gather (U, P) into Kz and (F, G) into b; zero x, v_prev, w_prev, w
  for (int q = (int)tm.rank(); q < n; q += (int)tm.size()) {
    double up, fg;
    if (q < 3 * nv) {
      const int d = q / nv;
      const int c = S.vidx[q - d * nv];
      up = (double)L.u[d][c];
      if (L.flags[c] & F_SLIP) {
        // the admissible part of f at a free-slip node: the assembled rows
        // carry the identity in the constrained directions (Sec. 6.1)
        T fv[3] = {L.f[0][c], L.f[1][c], L.f[2][c]};
        slip_project(class_row(L, c), fv);
        fg = (double)fv[d];
      } else {
        fg = (double)L.f[d][c];
      }
    } else {
      const int c = S.pidx[q - 3 * nv];
      up = (double)L.p[c];
      fg = (double)L.g[c];
    }
    Kz[q] = up;
    b[q] = fg;
    x[q] = 0.0;
    vv[0][q] = 0.0;
    ww[0][q] = 0.0;
    ww[1][q] = 0.0;
  }
  tm.sync();
  // b = (F, G) - K (U, P), v_1 = b
  for (int r = (int)tm.rank(); r < n; r += (int)tm.size()) {
    const double br = b[r] - csr_row(S.kptr, S.kcol, S.kval, r, Kz);
    b[r] = br;
    vv[1][r] = br;
  }
  tm.sync();

  int iv_prev = 0, iv = 1, iv_next = 2, iz = 0, iz_next = 1, iw_prev = 0, iw = 1, iw_next = 2;
  int cg_total = precond(C, vv[iv], zz[iz], cg, prm.cg_max, prm.cg_rtol);
  // the scalars of the recurrence are evaluated by the handler warp of each
  // sum (team_finish) and published
  double gamma;
  team_reduce1<1>(C.T, dot_part(C, zz[iz], vv[iv]), n, &gamma,
                  [](double tot, double* out) { out[0] = sqrt(fmax(tot, 0.0)); });
  int its = 0;
  double rel = 0.0;
  if (gamma > 0.0) {
    const double gamma1 = gamma;
    double gamma_prev = 1.0, eta = gamma;
    double c_prev = 1.0, cc = 1.0, s_prev = 0.0, ss = 0.0;
    for (; its < prm.minres_max;) {
      for (int q = (int)tm.rank(); q < n; q += (int)tm.size()) zz[iz][q] /= gamma;
      tm.sync();
      applyK(C, zz[iz], Kz);
      double r[3];
      team_reduce1<3>(C.T, dot_part(C, Kz, zz[iz]), n, r, [=](double tot, double* out) {
        out[0] = tot;
        out[1] = tot / gamma;
        out[2] = gamma / gamma_prev;
      });
      const double delta = r[0], r1 = r[1], r2 = r[2];
      for (int q = (int)tm.rank(); q < n; q += (int)tm.size())
        vv[iv_next][q] = Kz[q] - r1 * vv[iv][q] - r2 * vv[iv_prev][q];
      tm.sync();
      cg_total += precond(C, vv[iv_next], zz[iz_next], cg, prm.cg_max, prm.cg_rtol);
      double g[6];
      team_reduce1<6>(C.T, dot_part(C, zz[iz_next], vv[iv_next]), n, g, [=](double tot, double* out) {
            const double gamma_next = sqrt(fmax(tot, 0.0));
            const double a0 = fma(cc, delta, -(c_prev * ss * gamma));
            const double a1 = sqrt(fma(a0, a0, gamma_next * gamma_next));
            out[0] = gamma_next;
            out[1] = a1;
            out[2] = fma(c_prev * cc, gamma, ss * delta);
            out[3] = s_prev * gamma;
            out[4] = a0 / a1;
            out[5] = gamma_next / a1;
          });
      const double gamma_next = g[0], a1 = g[1], a2 = g[2], a3 = g[3], c_next = g[4], s_next = g[5];
      if (a1 == 0.0) break;
      const double step = c_next * eta;
      for (int q = (int)tm.rank(); q < n; q += (int)tm.size()) {
        const double wn = (zz[iz][q] - a3 * ww[iw_prev][q] - a2 * ww[iw][q]) / a1;
        ww[iw_next][q] = wn;
        x[q] += step * wn;
      }
      tm.sync();
      eta = -s_next * eta;
      ++its;
      // shift the recurrences
      int t = iv_prev;
      iv_prev = iv;
      iv = iv_next;
      iv_next = t;
      t = iz;
      iz = iz_next;
      iz_next = t;
      t = iw_prev;
      iw_prev = iw;
      iw = iw_next;
      iw_next = t;
      gamma_prev = gamma;
      gamma = gamma_next;
      c_prev = cc;
      cc = c_next;
      s_prev = ss;
      ss = s_next;
      rel = eta;
      if (fabs(eta) <= prm.minres_rtol * gamma1 || gamma == 0.0) break;
    }
    rel = fabs(rel) / gamma1;
  }
  // (U, P) += x
  for (int q = (int)tm.rank(); q < n; q += (int)tm.size()) {
    if (q < 3 * nv) {
      const int d = q / nv;
      const int c = S.vidx[q - d * nv];
      L.u[d][c] = (T)((double)L.u[d][c] + x[q]);
    } else {
      const int c = S.pidx[q - 3 * nv];
      L.p[c] = (T)((double)L.p[c] + x[q]);
    }
  }
  if (tm.rank() == 0 && info) {
    info[0] = (double)its;
    info[1] = rel;
    info[2] = (double)cg_total;
  }
}

}  // namespace coarse
}  // namespace hhg
