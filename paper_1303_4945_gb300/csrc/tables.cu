// tables.cu -- plan-time kernels: recursion coefficients and start-value prefactors.
//
// Recursion of Sect. 4.1 (the Wigner-d recursion it takes from Kostelec &
// Rockmore), restated for d^l_{a b} with
// a = -m, b = s:
//   [cos t + m s / (l (l+1))] d^l = c1_l d^{l-1} + c2_l d^{l+1},
//   c1_l = sqrt((l^2 - m^2)(l^2 - s^2)) / (l (2l+1)),
//   c2_l = sqrt(((l+1)^2 - m^2)((l+1)^2 - s^2)) / ((l+1)(2l+1)).
// With lambda_l = (-1)^m N_l d^l, N_l = sqrt((2l+1)/(4 pi)), this becomes
//   lambda_{l+1} = (A_l cos t + AK_l) lambda_l - C_l lambda_{l-1},
//   A_l  = N_{l+1} / (N_l c2_l)  = (l+1) sqrt((2l+3)(2l+1)) / sqrt(((l+1)^2 - m^2)((l+1)^2 - s^2)),
//   AK_l = A_l m s / (l (l+1)),
//   C_l  = N_{l+1} c1_l / (N_{l-1} c2_l)
//        = sqrt((2l+3)/(2l-1)) (l+1)/l sqrt((l^2-m^2)(l^2-s^2) / (((l+1)^2-m^2)((l+1)^2-s^2))).
// For -s the same table applies with AK_l -> -AK_l.  For s = 0 these reduce to
// the familiar A_l = sqrt((4(l+1)^2 - 1)/((l+1)^2 - m^2)), C_l = A_l sqrt((l^2 - m^2)/(4 l^2 - 1)).
#include "sht_device.cuh"

namespace sht {

// The kernels run the recursion on p_l = lambda_l / alpha_l with alpha_l alpha_{l+1} = A_l.
// C_l = A_l / A_{l-1}, so the coefficient of p_{l-1} becomes 1:
//   p_{l+1} = (a_l cos t + b_l) p_l - p_{l-1},   a_l = A_l alpha_l / alpha_{l+1} = alpha_l^2,
//   b_l = AK_l alpha_l / alpha_{l+1} = a_l m s / (l (l + 1)),
// one product less per step and one table entry less per (m, l).  The a_lm are
// multiplied by alpha_l before a synthesis and after an analysis.  a_l = A_l^2 / a_{l+1}
// runs downwards in double-double from a_{lmax+1} = A_lmax (A_l tends to 2 for large l,
// where the interleaved subsequences then agree) on the rational A_l^2.  In plain
// double the chain's roundings reach the values through the alternating products and
// cost a factor of 4 on the rings next to the poles (lmax 4095, m 1: 1.9e-11 against
// 3.4e-12; the form with three coefficients has 4e-12 there and twice this form's
// error elsewhere).
__device__ __forceinline__ dd dd_norm(double hi, double lo) {
  const double s = hi + lo;
  return {s, lo - (s - hi)};
}
__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const double p = a.hi * b.hi;
  return dd_norm(p, fma(a.hi, b.hi, -p) + (a.hi * b.lo + a.lo * b.hi));
}
__device__ __forceinline__ dd dd_div(dd a, dd b) {
  const double q = a.hi / b.hi;
  const double r = fma(-q, b.hi, a.hi) + (a.lo - q * b.lo);
  return dd_norm(q, r / b.hi);
}
// A_l^2 = (l+1)^2 / ((l+1)^2 - m^2) (2l+1)(2l+3) / ((l+1)^2 - s^2): quotients of integers
// exact in double
__device__ dd coef_A2(int l, int m, int s) {
  const double L1 = l + 1.0, dm = m, ds = s;
  return dd_mul(dd_div({L1 * L1, 0.0}, {(L1 - dm) * (L1 + dm), 0.0}),
                dd_div({(2.0 * L1 - 1.0) * (2.0 * L1 + 1.0), 0.0}, {(L1 - ds) * (L1 + ds), 0.0}));
}

// coef: the FP64 table's first ncoef64 entries (a mixed plan keeps only the prefix
// its FP64 columns read); coef32 (mixed plans) and alpha: every entry.  One block
// per m; thread t owns an even number of consecutive degrees (the last thread the
// rest).  a at the start of an even stretch is a at its end times the product of
// A_l^2 / A_{l+1}^2 over every second degree, so the stretches join in a short serial
// scan of one product each.
constexpr int kCoefThreads = 256;
__global__ void __launch_bounds__(kCoefThreads)
    coef_kernel(int lmax, int spin, int nm, const int *__restrict__ mval, const int64_t *__restrict__ coef_off,
                double2 *__restrict__ coef, int64_t ncoef64, float4 *__restrict__ coef32, double *__restrict__ alpha) {
  __shared__ dd start[kCoefThreads + 1];
  const int mi = blockIdx.x, t = threadIdx.x;
  if (mi >= nm) return;
  const int m = mval[mi];
  const int as = spin < 0 ? -spin : spin;
  const int l0 = m > as ? m : as, n = lmax - l0 + 1;
  const int len = 2 * ((n + 2 * kCoefThreads - 1) / (2 * kCoefThreads));
  const int i0 = min(t * len, n), i1 = min(i0 + len, n);
  const int last = (n - 1) / len;  // the thread holding degree lmax
  const dd top = {sqrt(coef_A2(lmax, m, as).hi), 0.0};
  if (i0 < i1) {
    dd q = t < last ? dd{1.0, 0.0} : top;
    if (t < last)
      for (int i = i0; i < i1; i += 2) q = dd_mul(q, dd_div(coef_A2(l0 + i, m, as), coef_A2(l0 + i + 1, m, as)));
    else
      for (int i = i1 - 1; i >= i0; --i) q = dd_div(coef_A2(l0 + i, m, as), q);
    start[t] = q;
  }
  __syncthreads();
  if (t == 0)
    for (int k = last - 1; k >= 0; --k) start[k] = dd_mul(start[k], start[k + 1]);
  __syncthreads();
  if (i0 >= i1) return;
  dd q = i1 < n ? start[t + 1] : top;  // a_{l+1}
  for (int k = i1 - 1; k >= i0; --k) {
    const int l = l0 + k;
    q = dd_div(coef_A2(l, m, as), q);
    const double r = sqrt(q.hi);
    const double f = l == 0 ? 0.0 : (double)m * (double)spin / ((double)l * (l + 1.0));
    const double b = q.hi * f;
    const int64_t i = coef_off[mi] + k;
    alpha[i] = r + 0.5 * q.lo / r;
    if (i < ncoef64) coef[i] = make_double2(q.hi, b);
    if (coef32) {
      const float ah = (float)q.hi, bh = (float)b;
      coef32[i] = make_float4(ah, (float)(q.hi - (double)ah), bh, (float)(b - (double)bh));
    }
  }
}

// sqrt((2 l0 + 1)/(4 pi)) * sqrt((2 l0)! / ((l0 + k)! (l0 - k)!)) as (mantissa, exponent),
// k = s if m >= |s| else m, over alpha_{l0} (the start value of the scaled recursion).  The factorial ratio is a product of min(u, v)
// ratios (hi + j)/j accumulated in double-double with a separate exponent.
__global__ void prefactor_kernel(int spin, int nm, const int *__restrict__ mval,
                                 const int64_t *__restrict__ coef_off, const double *__restrict__ alpha,
                                 double2 *__restrict__ pre) {
  const int mi = blockIdx.x * blockDim.x + threadIdx.x;
  if (mi >= nm) return;
  const int m = mval[mi];
  const int as = spin < 0 ? -spin : spin;
  const int l0 = m > as ? m : as;
  const int k = (m >= as) ? as : m;
  const int u = l0 - k, v = l0 + k;  // (2 l0)! / (u! v!)
  double hi = 1.0, lo = 0.0;
  int ex = 0;
  for (int j = 1; j <= u; ++j) {
    const double num = (double)(v + j), den = (double)j;
    const double q = num / den;
    const double qe = fma(-q, den, num) / den;  // q + qe = num/den to ~1e-32
    const double p = hi * q;
    double e = fma(hi, q, -p) + (hi * qe + lo * q);
    hi = p + e;
    lo = e - (hi - p);
    int t;
    hi = frexp(hi, &t);
    lo = ldexp(lo, -t);
    ex += t;
  }
  // square root of (hi + lo) 2^ex
  if (ex & 1) {
    hi *= 2.0;
    lo *= 2.0;
    ex -= 1;
  }
  const double r = sqrt(hi);
  const double rl = (fma(-r, r, hi) + lo) / (2.0 * r);
  const double nrm = sqrt((2.0 * l0 + 1.0) / (4.0 * 3.14159265358979323846));
  double mant = (r + rl) * nrm / alpha[coef_off[mi]];
  int t;
  mant = frexp(mant, &t);
  pre[mi] = make_double2(mant, (double)(ex / 2 + t));
}

cudaError_t launch_coef_tables(const sht_plan_s *P, cudaStream_t st) {
  if (P->nm > 0) {
    coef_kernel<<<P->nm, kCoefThreads, 0, st>>>(P->lmax, P->spin, P->nm, P->d_mval, P->d_coef_off, P->d_coef,
                                                P->ncoef64, P->d_coef32, P->d_alpha);
    prefactor_kernel<<<(P->nm + 127) / 128, 128, 0, st>>>(P->spin, P->nm, P->d_mval, P->d_coef_off, P->d_alpha,
                                                          P->d_mpre);
  }
  return cudaGetLastError();
}

}  // namespace sht
