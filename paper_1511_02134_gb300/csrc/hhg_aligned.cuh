// FP64 stencil sums in aligned 64-bit integers.
//
// The closed-form stencils of regular nodes are integer combinations of the
// field: the 7-point Laplacian, and twelve times the divergence differences
// along the seven Kuhn directions (hhg_device.cuh).  On GB300 an FP64
// operation occupies a quarter of an SM for 64 cycles per warp, a 64-bit
// integer addition for 2 and a shift or logical operation on a word for 2.  So
// the values of one stencil are aligned to the largest exponent among them,
// as integers with G bits below the last place of that largest value, summed
// exactly, and converted back once: about 27 cycles per value and 70 per sum
// in place of 64 per addition (the divergence sums of one field take 16
// operations per component).
// Measured (cube level 7, with boundary nodes in blocks of their own): Uzawa
// step 567 -> 347 us, its pressure sweep 275 -> 134 us, residual 448 -> 223 us;
// level 8 Uzawa step 4.75 (unsplit) -> 2.56 ms.
//
// Accuracy (u = 2^-53): where every value of a stencil that is not zero has an
// exponent within G of the largest, no bit is cut off: the sum is exact,
// rounded once, and no order of FP64 operations comes closer.  In other
// stencils (mixed magnitudes, a zero crossing) a value loses less than one
// unit of 2^-G last places of the largest.  The FP64 operations combine
// opposite neighbours first, without error where these cancel, and the small
// values then count in full; so a stencil with cut values is summed in
// integers only where the largest pair (the difference of two opposite
// neighbours in a divergence, their sum in a Laplacian, or the centre) is
// within 2^-K of the largest value (AlSums::note).  The sum is then off by at
// most 3 u (six neighbours), 6 u (Laplacian) or 9 u (divergence) of that pair
// and one rounding, where the FP64 operations may round that pair and each of
// the up to nine sums it enters.  Over ten kinds of random stencils (one and
// many magnitudes, equal, close and opposite pairs, ramps) the rms error of
// those with cut values is 0.45 to 1.0 of the FP64 operations'.  (Two pairs
// that cancel each other are not looked for.)
//
// All other stencils take the FP64 operations: those without such a pair, and
// those whose largest value is not finite, or so large that the sum could
// overflow, or below 2^-959 (shifts and subnormals).  The integer sums only
// note that (AlSums::bad); such a sum is formed again by a function of its own
// (al_fp64_*), which reads the values again: kept in registers beside their
// integers they would cost all nodes.
// Measured (cube level 7, a solve's last state): FP64 wherever a value is cut
// off 65.2 ms per solve, K smaller by two 59.9, by one 57.7, as here 57.3,
// every stencil in integers 56.8.
#pragma once
#include <type_traits>

#include "hhg_device.cuh"

namespace hhg {

// Twice the high word: exponent (11 bits) and leading mantissa bits, without the sign.
__device__ __forceinline__ uint32_t al_mag(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x);
  return h + h;
}

// top: the largest al_mag of a stencil with its mantissa bits set (exponent top >> 21).
__device__ __forceinline__ bool al_range(uint32_t top) { return top - (64u << 21) < ((0x7f0u - 64u) << 21); }

template <int G>
__device__ __forceinline__ int64_t al_int(double x, uint32_t top) {
  const uint32_t hi = (uint32_t)__double2hiint(x);
  const uint32_t sh = (top - (hi + hi)) >> 21;  // exponent below the largest
  uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | (uint32_t)__double2loint(x)) << G;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(sh));  // shifts beyond 63 give zero (zeros, subnormals)
  const int64_t s = (int32_t)hi >> 31;
  return ((int64_t)m ^ s) - s;
}

// The FP64 value of a sum of al_int<G>(., top).
template <int G>
__device__ __forceinline__ double al_value(int64_t s, uint32_t top) {
  const double d = (double)s;
  const int hi = __double2hiint(d) + (((int)(top >> 21) - 1075 - G) << 20);
  return s == 0 ? 0.0 : __hiloint2double(hi, __double2loint(d));
}

// Alignment of one stencil: top, and whether its integers hold it: in range,
// and no bit is cut off by G bits below the last place of the largest value
// (zeros count as cut off, one operation per value) or the largest pair is
// close to it.  Stencils of zeros hold (their values shift out).
template <int G>
struct AlTop {
  uint32_t top;
  bool in, whole;

  template <int N>
  __device__ __forceinline__ explicit AlTop(const double (&v)[N]) {
    uint32_t hi = al_mag(v[0]), lo = hi;
#pragma unroll
    for (int n = 1; n < N; ++n) {
      hi = max(hi, al_mag(v[n]));
      lo = min(lo, al_mag(v[n]));
    }
    top = hi | 0x1fffffu;
    in = al_range(top);
    whole = lo >= (top & ~0x1fffffu) - ((uint32_t)G << 21);
    if (hi == 0) {
      uint32_t any = 0;
#pragma unroll
      for (int n = 0; n < N; ++n) any |= (uint32_t)__double2loint(v[n]);
      top = 0x3fffffffu;
      in = whole = any == 0;
    }
  }
  // pair: the high word of the largest pair; at least 2^-K of the largest
  // value's leading bit (one unit allows for the low word).
  template <int K>
  __device__ __forceinline__ bool holds(int32_t pair) const {
    return in && (whole || pair > (1 << (20 + G - K)) + 1);
  }
};

__device__ __forceinline__ int32_t al_pair(int64_t d) { return abs((int32_t)(d >> 32)); }

// The 14 neighbours along +-(e1, e2, e3, e1+e2, e2+e3, e1+e3, e1+e2+e3).
template <class V>
__device__ __forceinline__ void al_load14(const V& x, double (&v)[14]) {
  v[0] = x(1, 0, 0);
  v[1] = x(-1, 0, 0);
  v[2] = x(0, 1, 0);
  v[3] = x(0, -1, 0);
  v[4] = x(0, 0, 1);
  v[5] = x(0, 0, -1);
  v[6] = x(1, 1, 0);
  v[7] = x(-1, -1, 0);
  v[8] = x(0, 1, 1);
  v[9] = x(0, -1, -1);
  v[10] = x(1, 0, 1);
  v[11] = x(-1, 0, -1);
  v[12] = x(1, 1, 1);
  v[13] = x(-1, -1, -1);
}

template <class T, class I>
__device__ __forceinline__ Diff7<T> al_diff7(const I (&v)[14]) {
  return Diff7<T>{v[0] - v[1], v[2] - v[3], v[4] - v[5], v[6] - v[7], v[8] - v[9], v[10] - v[11], v[12] - v[13]};
}

__device__ __forceinline__ int32_t al_pair14(const Diff7<int64_t>& d) {
  return max(max(max(al_pair(d.e1), al_pair(d.e2)), max(al_pair(d.e3), al_pair(d.f12))),
             max(max(al_pair(d.f23), al_pair(d.f13)), al_pair(d.b)));
}

// Sum of three pairs of integers, and the largest of the pairs.
__device__ __forceinline__ int64_t al_sum6(const int64_t* i, int32_t& pair) {
  const int64_t a = i[0] + i[1], b = i[2] + i[3], c = i[4] + i[5];
  pair = max(max(al_pair(a), al_pair(b)), al_pair(c));
  return (a + b) + c;
}

// Stencil sums of one node in aligned integers.  Each sum has a bit, set in bad
// if it has to be formed in FP64.  (The divergences leave a stencil that is
// out of range at once: that branch keeps the compiler from loading all fields
// ahead, which costs half the warps, and leaves it the next field's loads
// beside this one's conversions.)
struct AlSums {
  unsigned bad = 0;

  template <int K, int G>
  __device__ __forceinline__ void note(const AlTop<G>& t, int32_t pair, unsigned bit) {
    if (!t.holds<K>(pair)) bad |= bit;
  }

  // Sum of the six axis neighbours (6 2^60 < 2^63).
  __device__ __forceinline__ double nb6(const GNb<double>& x, unsigned bit) {
    constexpr int G = 7;
    const double v[6] = {x(-1, 0, 0), x(1, 0, 0), x(0, -1, 0), x(0, 1, 0), x(0, 0, -1), x(0, 0, 1)};
    const AlTop<G> t(v);
    int64_t i[6];
#pragma unroll
    for (int n = 0; n < 6; ++n) i[n] = al_int<G>(v[n], t.top);
    int32_t pair;
    const int64_t s = al_sum6(i, pair);
    note<5>(t, pair, bit);
    return al_value<G>(s, t.top);
  }

  // 6 x(c) minus the six axis neighbours (12 2^59 < 2^63).
  __device__ __forceinline__ double lap7(const GNb<double>& x, double xc, unsigned bit) {
    constexpr int G = 6;
    const double v[7] = {x(-1, 0, 0), x(1, 0, 0), x(0, -1, 0), x(0, 1, 0), x(0, 0, -1), x(0, 0, 1), xc};
    const AlTop<G> t(v);
    int64_t i[6];
#pragma unroll
    for (int n = 0; n < 6; ++n) i[n] = al_int<G>(v[n], t.top);
    int32_t pair;
    const int64_t nb = al_sum6(i, pair), c = al_int<G>(xc, t.top);
    note<4>(t, max(pair, al_pair(c)), bit);
    return al_value<G>(6 * c - nb, t.top);
  }

  // 12 Div of one field, component comp, or all three when comp < 0 (weights
  // 18 in all, partial sums below 30 2^58 < 2^63), from the integers i of its
  // values.
  static constexpr int DG = 5;
  __device__ __forceinline__ void div12_in(const AlTop<DG>& t, const int64_t (&i)[14], int comp, double* div, unsigned bit) {
    const Diff7<int64_t> d = al_diff7<int64_t>(i);
    note<3>(t, al_pair14(d), bit);
    if (comp < 0) {
      int64_t o[3];
      div12_all(d, o);
#pragma unroll
      for (int q = 0; q < 3; ++q) div[q] = al_value<DG>(o[q], t.top);
    } else {
      div[0] = al_value<DG>(div12(d, comp), t.top);
    }
  }
  __device__ __forceinline__ void div12_of(const GNb<double>& x, int comp, double* div, unsigned bit) {
    double v[14];
    al_load14(x, v);
    const AlTop<DG> t(v);
    if (!t.in) {
      bad |= bit;
      return;
    }
    int64_t i[14];
#pragma unroll
    for (int n = 0; n < 14; ++n) i[n] = al_int<DG>(v[n], t.top);
    div12_in(t, i, comp, div, bit);
  }
  // The residual's stencils of one field: the Laplacian 6 x(c) - sum of the
  // axis neighbours, and 12 Div (component comp, or all three into div[0..3)
  // when comp < 0).  The Laplacian takes the divergence's integers where the
  // largest of its own seven values is at most one exponent below the largest
  // of the divergence's fourteen (a smooth field), else its own alignment: a
  // neighbour with no weight in a row must not set what the row cuts off.  bit:
  // the Laplacian's, 16 bit the divergence's.
  __device__ __forceinline__ double lap_div(const GNb<double>& x, int comp, double* div, unsigned bit) {
    constexpr int G = DG;
    double v[14];
    al_load14(x, v);
    const double l[7] = {v[0], v[1], v[2], v[3], v[4], v[5], x(0, 0, 0)};
    const AlTop<G> t(v);
    AlTop<G> tl(l);
    if (!t.in || !tl.in) {
      bad |= 17 * bit;
      return 0.0;
    }
    const uint32_t below = (t.top >> 21) - (tl.top >> 21);  // wraps where the centre is the largest
    int64_t i[14];
#pragma unroll
    for (int n = 0; n < 14; ++n) i[n] = al_int<G>(v[n], t.top);
    div12_in(t, i, comp, div, 16 * bit);
    if (below > 1u) {
#pragma unroll
      for (int n = 0; n < 6; ++n) i[n] = al_int<G>(l[n], tl.top);
    } else {
      tl.whole = tl.whole && t.whole;
      tl.top = t.top;
    }
    int32_t pair;
    const int64_t nb = al_sum6(i, pair), c = al_int<G>(l[6], tl.top);
    note<3>(tl, max(pair, al_pair(c)), bit);
    return al_value<G>(6 * c - nb, tl.top);
  }
};

// FP64 fields in global memory are summed in aligned integers.  The
// cluster-resident levels keep the FP64 sums: their phases are latency bound,
// with fewer warps than FP64 pipes would need to be busy, and the integers
// spill (cube level 4 FP64 solve 8.50 -> 8.60 ms).
template <class V>
constexpr bool ALIGNED = std::is_same<V, GNb<double>>::value;

struct AlDiv {
  double d[3];
};
static __device__ __noinline__ double al_fp64_nb6(GNb<double> x) { return nb6v(x); }
static __device__ __noinline__ double al_fp64_lap7(GNb<double> x) { return 6.0 * x(0, 0, 0) - nb6v(x); }
static __device__ __noinline__ AlDiv al_fp64_div12(GNb<double> x) {
  AlDiv o;
  div12_all(diff7v<double>(x), o.d);
  return o;
}

// ---- the stencil sums of one regular node ---------------------------------------
// Plain sums in FP32 and on views of shared memory.

// Sums of the six axis neighbours of three fields.
template <class T, class V>
__device__ __forceinline__ void st_nb6x3(const V* u, T nb[3]) {
  if constexpr (ALIGNED<V>) {
    AlSums S;
#pragma unroll
    for (int d = 0; d < 3; ++d) nb[d] = S.nb6(u[d], 1u << d);
    if (S.bad)
#pragma unroll
      for (int d = 0; d < 3; ++d)
        if (S.bad & (1u << d)) nb[d] = al_fp64_nb6(u[d]);
  } else {
#pragma unroll
    for (int d = 0; d < 3; ++d) nb[d] = nb6v(u[d]);
  }
}

// ... of one field.
template <class T, class V>
__device__ __forceinline__ T st_nb6(const V& x) {
  if constexpr (ALIGNED<V>) {
    AlSums S;
    const double nb = S.nb6(x, 1u);
    return S.bad ? al_fp64_nb6(x) : nb;
  } else {
    return nb6v(x);
  }
}

// 12 Div_d x for d = 0, 1, 2.
template <class T, class V>
__device__ __forceinline__ void st_div12_all(const V& x, T out[3]) {
  if constexpr (ALIGNED<V>) {
    AlSums S;
    S.div12_of(x, -1, out, 1u);
    if (S.bad) {
      const AlDiv o = al_fp64_div12(x);
#pragma unroll
      for (int d = 0; d < 3; ++d) out[d] = o.d[d];
    }
  } else {
    div12_all(diff7v<T>(x), out);
  }
}

// 12 Div_d u_d (div[d]) and 6 p(c) minus the six axis neighbours of p; pc = p(c).
template <class T, class V>
__device__ __forceinline__ T st_pres(const V* u, const V& p, T pc, T div[3]) {
  if constexpr (ALIGNED<V>) {
    AlSums S;
#pragma unroll
    for (int d = 0; d < 3; ++d) S.div12_of(u[d], d, div + d, 1u << d);
    double lap = S.lap7(p, pc, 8u);
    if (S.bad) {
#pragma unroll
      for (int d = 0; d < 3; ++d)
        if (S.bad & (1u << d)) div[d] = al_fp64_div12(u[d]).d[d];
      if (S.bad & 8u) lap = al_fp64_lap7(p);
    }
    return lap;
  } else {
    div[0] = div12(diff7v<T>(u[0]), 0);
    div[1] = div12(diff7v<T>(u[1]), 1);
    div[2] = div12(diff7v<T>(u[2]), 2);
    return (T)6 * pc - nb6v(p);
  }
}

// The residual's sums, each field aligned once for its Laplacian and its
// divergence part: Laplacians of u and p, 12 Div_d u_d, 12 Div_d p.
__device__ __forceinline__ double st_residual(const GNb<double>* u, const GNb<double>& p, double lap[3], double du[3],
                                              double dp[3]) {
  AlSums S;
#pragma unroll
  for (int d = 0; d < 3; ++d) lap[d] = S.lap_div(u[d], d, du + d, 1u << d);
  double lp = S.lap_div(p, -1, dp, 8u);
  if (S.bad) {
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      if (S.bad & (1u << d)) lap[d] = al_fp64_lap7(u[d]);
      if (S.bad & (16u << d)) du[d] = al_fp64_div12(u[d]).d[d];
    }
    if (S.bad & 8u) lp = al_fp64_lap7(p);
    if (S.bad & 128u) {
      const AlDiv o = al_fp64_div12(p);
#pragma unroll
      for (int d = 0; d < 3; ++d) dp[d] = o.d[d];
    }
  }
  return lp;
}

}  // namespace hhg
