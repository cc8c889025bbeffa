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
  // tensor-core form (legendre_tc64.cu): 2^lexp bounds |p_l| of (m index, pair); geo[m index]:
  // the equator-most ring reaches that from the first degree on
  const signed char *lexp;
  const unsigned char *geo;
  // per m index, a byte per job: the columns of a synthesis that its fixed-point operands
  // do not hold to an IEEE sum's accuracy
  const unsigned *wide_syn;
  int *err;  // device status word (bounded waits)
};

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
