// A "team" is every thread of a one-cluster grid: a thread-block cluster of
// nblocks CTAs (or a single block when nblocks == 1).  Phases of a fused
// multigrid kernel are separated by the cluster barrier (a hardware barrier
// with release/acquire semantics at cluster scope, so global-memory writes
// of one phase are seen by every CTA in the next), and sums over the team
// are formed in a fixed order through distributed shared memory, so every
// CTA gets the same, run-to-run reproducible value.
#pragma once
#include <cooperative_groups.h>
#include <stdint.h>

namespace hhg {

constexpr int TEAM_MAX_WARPS = 16;   // per CTA (512 threads)
constexpr int TEAM_MAX_BLOCKS = 16;  // CTAs of a cluster

// Shared memory of a team's sums and search directions, in doubles: groups
// per sum and directions per CTA.  One block needs 3.8 KB, a cluster 16.4 KB;
// it is dynamic shared memory, because a block's solver lives in what the
// shared memory leaves of L1 (16 KB more took the solve of 3,000 unknowns
// from 11 to 18 ms).
constexpr int TEAM_MAX_SUMS = 3, TEAM_MAX_OUT = 6;
__host__ __device__ constexpr int team_groups(unsigned nblocks) {
  return nblocks > 1 ? TEAM_MAX_BLOCKS * TEAM_MAX_WARPS : TEAM_MAX_WARPS;
}
__host__ __device__ constexpr int team_dirs(unsigned nblocks) { return nblocks > 1 ? 512 : 384; }
__host__ __device__ constexpr unsigned team_bytes(unsigned nblocks) {
  return (unsigned)sizeof(double) * (2 * TEAM_MAX_SUMS * team_groups(nblocks) + team_dirs(nblocks));
}

struct Team {
  unsigned nblocks;            // CTAs in the cluster; the grid is exactly one cluster
  double* mem;                 // team_bytes(nblocks) of shared memory (at the same offset in every CTA)
  mutable unsigned calls = 0;  // sums formed so far (the same in every thread): picks the exchange buffer

  // groups of sum w in exchange buffer `buf`; the search directions
  __device__ __forceinline__ double* part(unsigned buf, int w) const {
    return mem + (buf * TEAM_MAX_SUMS + w) * team_groups(nblocks);
  }
  __device__ __forceinline__ double* dirs() const { return mem + 2 * TEAM_MAX_SUMS * team_groups(nblocks); }

  // Consecutive warps of the ranking sit on different CTAs, so that a loop
  // over fewer items than threads loads every SM alike (a ranking CTA by CTA
  // left the 1,500 rows of the obstacle channel's coarsest level on 3 of 16).
  __device__ __forceinline__ unsigned rank() const {
    return ((threadIdx.x >> 5) * nblocks + blockIdx.x) * 32 + (threadIdx.x & 31);
  }
  __device__ __forceinline__ unsigned size() const { return nblocks * blockDim.x; }
  __device__ __forceinline__ void sync() const {
    if (nblocks > 1)
      cooperative_groups::this_cluster().sync();
    else
      __syncthreads();
  }
};

// Sum over the warp, in every lane.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums over the team are formed from groups of 32 values, a warp each: the
// sum of group g of sum w is published to slot [w][g] of every CTA
// (team_publish), and the handler warp of sum w adds the groups in runs of
// blockDim.x / 32, each run in order, then the runs in order (team_finish).
// That fixes the rounding by the order of the values alone, wherever in the
// cluster a group is held.
// The calling warp's 32 values as group `group` of sum w.
__device__ __forceinline__ void team_publish(const Team& T, double x, int w, int group) {
  const int lane = threadIdx.x & 31;
  x = warp_sum(x);
  double* at = T.part(T.calls & 1u, w) + group;
  if (T.nblocks > 1) {
    if (lane < (int)T.nblocks) *cooperative_groups::this_cluster().map_shared_rank(at, lane) = x;
  } else if (lane == 0) {
    *at = x;
  }
}

// Totals of the W sums just published (groups 0 .. ngroups - 1 of each).
// Warp w < W of every CTA is the handler of sum w: it evaluates
// fin(total, out) in all its lanes (out: W_OUT doubles published to the
// CTA), so that the scalar recurrences of a Krylov step run in one warp per
// CTA.  On GB300 an FP64 instruction occupies a quarter of an SM for 64
// cycles per warp: evaluated by every thread, the partials of sixteen CTAs,
// the divisions and the square roots of a step cost several times its
// vectors.  Every thread must call it; blockDim.x is a multiple of 32, at
// least 32 W and at most 32 TEAM_MAX_WARPS.  vals receives the published
// values, vals[w * W_OUT + e].  A single sum of a block of at most four warps
// is formed by every warp (each has a quarter of the SM to itself), without
// the exchange of the values.
template <int W, int W_OUT, class F>
__device__ __forceinline__ void team_finish(const Team& T, int ngroups, double* vals, F&& fin) {
  static_assert(W <= TEAM_MAX_SUMS && W * W_OUT <= TEAM_MAX_OUT, "team_finish buffers");
  __shared__ double res[2][TEAM_MAX_OUT];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned buf = T.calls & 1u;
  ++T.calls;
  // one barrier per sum: a CTA reaches the barrier of the next sum (the other
  // buffer) only after it has read this one's groups
  T.sync();
  const bool every = W == 1 && T.nblocks == 1 && blockDim.x <= 128;
  if (warp < W || every) {
    const int per = (int)(blockDim.x >> 5), g0 = lane * per;
    const int most = min(per, ngroups);
    const double* at = T.part(buf, every ? 0 : warp);
    double run = g0 < ngroups ? at[g0] : 0.0;
    for (int j = 1; j < most; j += 4) {
      double v[4];  // four loads in flight, then the additions in order
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = at[min(g0 + j + e, team_groups(T.nblocks) - 1)];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j + e < most) run += g0 + j + e < ngroups ? v[e] : 0.0;
    }
    double tot = __shfl_sync(0xffffffffu, run, 0);
    for (int c = 1; c * per < ngroups; ++c) tot += __shfl_sync(0xffffffffu, run, c);
    double out[W_OUT];
    fin(tot, out);
    if (every) {
#pragma unroll
      for (int e = 0; e < W_OUT; ++e) vals[e] = out[e];
      return;
    }
    if (lane == 0)
#pragma unroll
      for (int e = 0; e < W_OUT; ++e) res[buf][warp * W_OUT + e] = out[e];
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < W * W_OUT; ++e) vals[e] = res[buf][e];
}

// One sum of a value per thread of the ranking, n items in the loop that formed them.
template <int W_OUT, class F>
__device__ __forceinline__ void team_reduce1(const Team& T, double x, int n, double* vals, F&& fin) {
  const int group = (int)(T.rank() >> 5), ngroups = (min(n, (int)T.size()) + 31) / 32;
  if (group < ngroups) team_publish(T, x, 0, group);
  team_finish<1, W_OUT>(T, ngroups, vals, fin);
}

// A double at a shared-memory address of this CTA or of another CTA of the
// cluster (volatile: ordered with the barriers, free to overlap other loads).
__device__ __forceinline__ double ld_team_shared(uint32_t addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr));
  return v;
}
// Address in CTA r of the cluster of the shared-memory address addr of this CTA.
__device__ __forceinline__ uint32_t team_shared_addr(uint32_t addr, uint32_t r) {
  uint32_t v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(v) : "r"(addr), "r"(r));
  return v;
}

}  // namespace hhg
