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
// step 567 -> 351 us, its pressure sweep 275 -> 134 us, residual 448 -> 215 us;
// level 8 Uzawa step 4.75 (unsplit) -> 2.65 ms.
//
// Accuracy: a value whose exponent is within G of the largest is represented
// exactly; of the others at most one unit of 2^-G last places of the largest
// value is cut off per value.  Sums of values of similar size, the smooth
// fields of a solve, are then exact up to the one rounding of the conversion,
// where a chain of FP64 operations rounds each partial sum; in every case
// the error is below that of the first rounding the chain would make of the
// largest value.  Over random fields of one and of many magnitudes its rms is
// 0.5 to 0.6 of the FP64 chain's, and both are exact on smooth ones.
//
// Ranges: a stencil whose largest value is not finite, or so large that the
// sum could overflow, or below 2^-959 (shifts and subnormals), takes the FP64
// operations; one of zeros is zero.
#pragma once
#include "hhg_device.cuh"

namespace hhg {

// Twice the high word: exponent (11 bits) and leading mantissa bits, without the sign.
__device__ __forceinline__ uint32_t al_mag(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x);
  return h + h;
}

// top: the largest al_mag with its mantissa bits set (exponent top >> 21).
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

template <int N>
__device__ __forceinline__ uint32_t al_top(const double (&v)[N]) {
  uint32_t t = al_mag(v[0]);
#pragma unroll
  for (int n = 1; n < N; ++n) t = max(t, al_mag(v[n]));
  return t | 0x1fffffu;
}

template <int N>
__device__ __forceinline__ bool al_zero(const double (&v)[N]) {
  uint32_t t = 0;
#pragma unroll
  for (int n = 0; n < N; ++n) t |= al_mag(v[n]) | (uint32_t)__double2loint(v[n]);
  return t == 0;
}

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

// Sum of the six axis neighbours (6 2^60 < 2^63).
template <class V>
__device__ __forceinline__ double al_nb6(const V& x) {
  constexpr int G = 7;
  const double v[6] = {x(-1, 0, 0), x(1, 0, 0), x(0, -1, 0), x(0, 1, 0), x(0, 0, -1), x(0, 0, 1)};
  const uint32_t top = al_top(v);
  if (!al_range(top)) return al_zero(v) ? 0.0 : ((v[0] + v[1]) + (v[2] + v[3])) + (v[4] + v[5]);
  int64_t s = 0;
#pragma unroll
  for (int n = 0; n < 6; ++n) s += al_int<G>(v[n], top);
  return al_value<G>(s, top);
}

// 6 x(c) minus the six axis neighbours (12 2^59 < 2^63).
template <class V>
__device__ __forceinline__ double al_lap7(const V& x) {
  constexpr int G = 6;
  const double v[7] = {x(-1, 0, 0), x(1, 0, 0), x(0, -1, 0), x(0, 1, 0), x(0, 0, -1), x(0, 0, 1), x(0, 0, 0)};
  const uint32_t top = al_top(v);
  if (!al_range(top)) return al_zero(v) ? 0.0 : 6.0 * v[6] - (((v[0] + v[1]) + (v[2] + v[3])) + (v[4] + v[5]));
  int64_t s = 0;
#pragma unroll
  for (int n = 0; n < 6; ++n) s -= al_int<G>(v[n], top);
  return al_value<G>(s + 6 * al_int<G>(v[6], top), top);
}

// 12 Div_d x for d = 0, 1, 2 (weights 18 in all, partial sums below 30 2^58 < 2^63).
template <class V>
__device__ __forceinline__ void al_div12_all(const V& x, double out[3]) {
  constexpr int G = 5;
  double v[14];
  al_load14(x, v);
  const uint32_t top = al_top(v);
  if (!al_range(top)) {
    if (al_zero(v))
      out[0] = out[1] = out[2] = 0.0;
    else
      div12_all(al_diff7<double>(v), out);
    return;
  }
  int64_t i[14], o[3];
#pragma unroll
  for (int n = 0; n < 14; ++n) i[n] = al_int<G>(v[n], top);
  div12_all(al_diff7<int64_t>(i), o);
#pragma unroll
  for (int d = 0; d < 3; ++d) out[d] = al_value<G>(o[d], top);
}

// 12 Div_comp x.
template <class V>
__device__ __forceinline__ double al_div12(const V& x, int comp) {
  constexpr int G = 5;
  double v[14];
  al_load14(x, v);
  const uint32_t top = al_top(v);
  if (!al_range(top)) return al_zero(v) ? 0.0 : div12(al_diff7<double>(v), comp);
  int64_t i[14];
#pragma unroll
  for (int n = 0; n < 14; ++n) i[n] = al_int<G>(v[n], top);
  return al_value<G>(div12(al_diff7<int64_t>(i), comp), top);
}

// The residual's stencils of one field: the Laplacian 6 x(c) - sum of the
// axis neighbours, and 12 Div (component comp, or all three into div[0..3)
// when comp < 0).  The Laplacian takes the divergence's integers where the
// largest of its own seven values is at most one exponent below the largest
// of the divergence's fourteen (a smooth field), else its own alignment: a
// neighbour with no weight in a row must not set what the row cuts off.
template <class V>
__device__ __forceinline__ double al_lap_div(const V& x, int comp, double* div) {
  constexpr int G = 5;
  double v[14];
  al_load14(x, v);
  const double l[7] = {v[0], v[1], v[2], v[3], v[4], v[5], x(0, 0, 0)};
  const uint32_t top = al_top(v), topl = al_top(l);
  if (!al_range(top) || !al_range(topl)) {
    const Diff7<double> d = al_diff7<double>(v);
    if (comp < 0)
      div12_all(d, div);
    else
      div[0] = div12(d, comp);
    return 6.0 * l[6] - (((v[1] + v[0]) + (v[3] + v[2])) + (v[5] + v[4]));
  }
  int64_t i[14];
#pragma unroll
  for (int n = 0; n < 14; ++n) i[n] = al_int<G>(v[n], top);
  const Diff7<int64_t> d = al_diff7<int64_t>(i);
  if (comp < 0) {
    int64_t o[3];
    div12_all(d, o);
#pragma unroll
    for (int q = 0; q < 3; ++q) div[q] = al_value<G>(o[q], top);
  } else {
    div[0] = al_value<G>(div12(d, comp), top);
  }
  const uint32_t below = (top >> 21) - (topl >> 21);  // wraps where the centre is the largest
  int64_t nb;
  uint32_t t = top;
  if (below <= 1u) {
    nb = ((i[0] + i[1]) + (i[2] + i[3])) + (i[4] + i[5]);
  } else {
    t = topl;
    nb = 0;
#pragma unroll
    for (int n = 0; n < 6; ++n) nb += al_int<G>(l[n], t);
  }
  return al_value<G>(6 * al_int<G>(l[6], t) - nb, t);
}

}  // namespace hhg
