// leg64.cuh -- the argument record of the FP64 Legendre kernels (legendre_fp64.cu,
// legendre_tc64.cu).
#pragma once
#include "sht_device.cuh"

namespace sht {

struct LegArgs {
  int lmax, spin, npairs, nm;
  const int *mval;
  const int64_t *coef_off;
  const double2 *coef;  // {a, b} of p_{l+1} = (a x + b) p_l - p_{l-1}
  const double2 *pm;    // alpha_l times a_lm (spin: P = E + iB, M = E - iB) per (array, m, l), indexed like coef
  int64_t ncoef;        // pm's entries per array
  const double2 *mpre;
  const PairDev *pairs;
  double2 *phase;  // [nmaps][nm][npairs][2]
  const int2 *syn_items;
  const int4 *ana_items;
  const int64_t *part_off;
  double *part;
  // tensor-core form (legendre_tc64.cu): 2^lexp bounds |p_l| of (m index, pair); ref[m index]:
  // the pair whose value at the first degree is nearest to its bound (RefPair)
  const signed char *lexp;
  const unsigned long long *ref;
  // per m index, a byte per job: the columns of a synthesis that its fixed-point operands
  // do not hold to an IEEE sum's accuracy
  const unsigned *wide_syn;
  int *err;  // device status word (bounded waits)
};

// An m's reference pair, as one number that orders: from the top 1 for the pair next to the
// equator where all its values at the first degree lie within 2^-kRefNear of the bound (the
// equator serves then), the exponent of the largest value over the bound plus 2^16, the
// pair, and a bit for each value (+s, -s) that near to the bound.
constexpr int kRefNear = 6;
__device__ __forceinline__ unsigned long long ref_key(bool equator, int exponent, int pair, int lanes) {
  return ((unsigned long long)(equator ? 1u : 0u) << 63) | ((unsigned long long)(unsigned)(max(exponent, -60000) + 65536) << 36) |
         ((unsigned long long)(unsigned)pair << 2) | (unsigned)lanes;
}
struct RefPair {
  int pair, lanes;
  bool near;  // no pair is near its bound where not
};
__device__ __forceinline__ RefPair ref_of(unsigned long long k) {
  return {(int)((k >> 2) & 0x3ffffffffull), (int)(k & 3u), (int)((k >> 36) & 0x7ffffffu) - 65536 >= -kRefNear};
}

// The tensor-core form rounds a column's inputs to 2^-54 of the largest and Lambda to 2^-56
// of its bound, so what a term loses is relative to the largest of its column.  kWideRange
// is the range, in powers of two, of the inputs that meet at one result (see alm_to_pm and
// tc64_ana_body) up to which the loss stays below the error of Lambda itself (2^-43, or
// 1e-13, against some 1e-13 to 1e-12 from the recursion on the rings and degrees where
// such ranges meet).  Beyond it the column or item runs in IEEE double.
constexpr int kWideRange = 14;
// the exponent field of a double as an order-preserving integer (denormals: 1; zero: 0)
__device__ __forceinline__ int size_field(double v) {
  const int e = (int)(((unsigned)__double2hiint(v) >> 20) & 0x7ffu);
  return e > 0 ? e : (v != 0.0 ? 1 : 0);
}
// fields within which scaled values and results neither overflow nor underflow
constexpr int kFieldMin = 100, kFieldMax = 1990;

}  // namespace sht
