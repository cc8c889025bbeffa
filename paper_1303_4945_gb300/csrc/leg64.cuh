// leg64.cuh -- the argument record of the FP64 Legendre kernels (legendre_fp64.cu,
// legendre_tc64.cu).
#pragma once
#include "sht_device.cuh"

namespace sht {

struct LegArgs {
  int lmax, spin, npairs, nm, astride;
  const int *mval;
  const int64_t *mstart;
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
  int ppt;
  const signed char *lexp;  // tensor-core form: 2^lexp bounds |p_l| of (m index, pair)
  int *err;                 // device status word (bounded waits)
};

}  // namespace sht
