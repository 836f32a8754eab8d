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

struct Team {
  unsigned nblocks;            // CTAs in the cluster; the grid is exactly one cluster
  mutable unsigned calls = 0;  // sums formed so far (the same in every thread): picks the exchange buffer

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

// Sum over the warp, in every lane.  The addends are aligned to the largest
// exponent as 58-bit integers (five bits below its last place, where shorter
// addends are cut off: together less than one unit in the last place of the
// largest), and summed exactly, in three limbs by the warp's integer
// reduction: 260 cycles on GB300 against 547 for a tree of five FP64
// additions, each of which occupies the FP64 pipe for 64.  Addends that are
// not finite or whose largest is below 2^-959 take the tree.
__device__ __forceinline__ double warp_sum(double x) {
  const int hi = __double2hiint(x), ah = hi & 0x7fffffff;
  const int top = __reduce_max_sync(0xffffffffu, ah) & 0x7ff00000;
  if (top >= 0x7ff00000 || top < (64 << 20)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  }
  // subnormal addends lie more than 58 bits below the largest: shifted out
  const int sh = ((top | 0xfffff) - ah) >> 20;
  int64_t m = ((int64_t)((ah & 0xfffff) | 0x100000) << 32) | (uint32_t)__double2loint(x);
  m = sh < 58 ? (m << 5) >> sh : 0;
  m = hi < 0 ? -m : m;
  const uint32_t s0 = __reduce_add_sync(0xffffffffu, (uint32_t)m & 0x3ffffffu);
  const uint32_t s1 = __reduce_add_sync(0xffffffffu, (uint32_t)(m >> 26) & 0x3ffffffu);
  const int s2 = __reduce_add_sync(0xffffffffu, (int)(m >> 52));
  const int64_t sum = (int64_t)s0 + ((int64_t)s1 << 26) + ((int64_t)s2 << 52);
  return (double)sum * __hiloint2double(top - (57 << 20), 0);
}

// a / b and 1 / c of values that are the same in every lane, by one division:
// even lanes form the first, odd lanes the second.
__device__ __forceinline__ void div_and_rcp(double a, double b, double c, double& q, double& r) {
  const bool odd = threadIdx.x & 1;
  const double v = (odd ? 1.0 : a) / (odd ? c : b);
  q = __shfl_sync(0xffffffffu, v, 0);
  r = __shfl_sync(0xffffffffu, v, 1);
}

// Exchange buffers of team_reduce, one set per kernel.
constexpr int TEAM_MAX_SUMS = 3, TEAM_MAX_OUT = 6;
struct TeamShared {
  double val[32 * TEAM_MAX_WARPS];
  double part[2][TEAM_MAX_SUMS][TEAM_MAX_BLOCKS];
  double res[2][TEAM_MAX_OUT];
};
__device__ __forceinline__ TeamShared& team_shared() {
  __shared__ TeamShared s;
  return s;
}

// W sums over the team of one value per thread, x: the warps [w * each,
// (w + 1) * each) of every CTA contribute to sum w, the others to none.  Warp
// w < W of every CTA is the handler of sum w: it adds its warps' values lane by lane, then
// over its lanes, exchanges the CTA's partial through distributed shared
// memory, and evaluates fin(w, total, out) in all its lanes (out: W_OUT
// doubles published to the CTA), so that the scalar recurrences of a Krylov
// step run in one warp per CTA.  On GB300 an FP64 instruction occupies a
// quarter of an SM for 64 cycles per warp: evaluated by every thread, the
// warp trees, the sixteen partials, the divisions and the square roots of a
// step cost several times its vectors.  Every thread must call it;
// blockDim.x is a multiple of 32, at least 32 W and at most
// 32 TEAM_MAX_WARPS.  Returns the published values: res[w * W_OUT + e].
template <int W, int W_OUT, class F>
__device__ __forceinline__ const double* team_reduce(const Team& T, double x, int each, F&& fin) {
  static_assert(W <= TEAM_MAX_SUMS && W * W_OUT <= TEAM_MAX_OUT, "team_reduce buffers");
  TeamShared& B = team_shared();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned buf = T.calls & 1u;
  ++T.calls;
  B.val[threadIdx.x] = x;
  __syncthreads();
  double tot = 0.0;
  if (warp < W) {
    tot = B.val[32 * warp * each + lane];
    for (int w = warp * each + 1; w < (warp + 1) * each; ++w) tot += B.val[32 * w + lane];
    tot = warp_sum(tot);
    if (T.nblocks > 1 && lane < (int)T.nblocks) {
      // this CTA's partial into slot blockIdx.x of every CTA
      double* at = &B.part[buf][warp][blockIdx.x];
      *cooperative_groups::this_cluster().map_shared_rank(at, lane) = tot;
    }
  }
  if (T.nblocks > 1) {
    // one barrier per sum: a CTA reaches the barrier of the next sum (the
    // other buffer) only after it has read this one's partials
    cooperative_groups::this_cluster().sync();
    if (warp < W) tot = warp_sum(lane < (int)T.nblocks ? B.part[buf][warp][lane] : 0.0);
  }
  if (warp < W) {
    double out[W_OUT];
    fin(warp, tot, out);
    if (lane == 0)
#pragma unroll
      for (int e = 0; e < W_OUT; ++e) B.res[buf][warp * W_OUT + e] = out[e];
  }
  __syncthreads();
  return B.res[buf];
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
