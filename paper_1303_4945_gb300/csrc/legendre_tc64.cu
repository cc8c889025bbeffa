// legendre_tc64.cu -- the FP64 form's Legendre stage (Eqs. syn2, ana1) with the
// contraction on the tensor cores (tcgen05).
//
// The FP64 pipe issues one warp instruction in 16 cycles per SM, so the kernels of
// legendre_fp64.cu are bound by their FP64 instructions: per (m, l, ring pair) 12 at
// spin s with one E/B pair (4 of the two recursions, 8 multiply-adds) and 4 at spin 0
// with one map, more with more of them.  Here only the recursions stay on that pipe.
// Each value is turned into an exact fixed-point number by integer instructions and the
// contraction runs as bf16 products of its digits, error-free as in the mixed form's
// kernels (legendre_tc.cu, legendre_tc_ana.cu; the structure of both is theirs):
//
//  * Lambda / u_p, u_p = 2^lexp a bound on the pair's values (bound_kernel, once per
//    plan), is rounded to a multiple of 2^-55 and cut into seven 8-bit digits in
//    [-128, 127]: the bytes of its two's complement form after 0x80 is added to each.
//    An IEEE double of Lambda's typical size, a quarter of the bound, is itself a multiple
//    of 2^-55 of it.
//  * The other operand (a_lm per column and 256-degree window; G_m times u_p per column
//    and tile) is scaled by a power of two of its largest value (in FP64, so the full
//    exponent range passes) and cut the same way.
//  * Products of digits i and j belong to level i + j.  The levels 0 to 2 are exact whatever
//    the digits (sums of at most 2^24 units over 512 entries), and level 3 but for inputs
//    whose digits are all near their ends at once (the synthesis sums its four products in
//    one accumulator, 1.5 2^24 units at worst; beyond 2^24 its last bit, 2^-38 of sums above
//    2^-14); levels 4 to 6 (2^-32 and below) are added in FP32, rounding below 2^-56 of the
//    bound; higher levels are dropped.  Level sums meet in exact two-sums and are
//    added up in FP64.
//
// An IEEE sum loses 2^-53 of each term, these operands 2^-54 of the largest input of a
// column.  Where the inputs that meet at one result lie within 2^10 of one another that
// stays below the error of Lambda itself, and the errors against 64-bit references are the
// same (below).  Where they do not (a spectrum falling steeply over degrees a ring hardly
// sees, one ring far brighter than the rest, a geometry without the equator, infinities
// and NaN, the ends of the exponent range), the CTA runs the IEEE sums (leg64_ieee.cuh):
// alm_to_pm decides for a synthesis' columns, tc64_ana_body for an analysis' items.  (As
// kernels of their own behind these, over the same items, they cost 4 us a call when
// nothing needed them, and a column of two E/B pairs at lmax 511 alone 0.3 ms.)
//
// Every wait is bounded (see legendre_tc_ana.cu).
//
// What bounds it (GB300, ncu, spin 2, lmax 1023): the FP64 pipe, 87% busy in both
// kernels, with four instructions per step; issue 27 - 33%, ALU 29 - 31% (the fixed-point
// conversion takes about 27 integer instructions a value), tensor pipe 5 - 13%.
// Measured against legendre_fp64.cu's kernels: HEALPix Nside 256, lmax 767, spin 2
// synthesis 2.85 -> 1.40 ms, analysis 4.64 -> 1.57; Gauss-Legendre lmax 1023, spin 0 1.74 ->
// 1.19 and 2.35 -> 1.56; two maps at lmax 511 on 1025 rings 0.93 -> 0.56 and 1.75 -> 0.77.
// Errors against 64 bits: the same to three digits (2.6e-14 / 5.1e-14, 1.3e-13 / 9.3e-14,
// 5.8e-14 / 1.0e-13).  Analysis CTAs of 256 threads with four accumulators (as in the mixed
// form): 1.52 and 1.44 ms on the first two, but 429 against 280 us at lmax 511, spin 0.
#include "dual.cuh"
#include "leg64_ieee.cuh"
#include "tcgen05.cuh"

namespace sht {
namespace t64 {

constexpr int kDig = 7;

// |w| <= 127/128 (a digit of 128 would wrap) -> w 2^63 rounded to 2^7, every byte offset
// by 128: digit i is byte 7 - i of the result minus 128, in units of 2^(-7-8i)
__device__ __forceinline__ uint64_t fix64(double w) {
  const uint32_t hw = (uint32_t)__double2hiint(w), lw = (uint32_t)__double2loint(w);
  const int e = (int)((hw >> 20) & 0x7ffu);
  const uint32_t hi = (((hw & 0xfffffu) | 0x100000u) << 10) | (lw >> 22);
  const uint64_t m = ((uint64_t)hi << 32) | (lw << 10);  // |w| = m 2^(e - 1022 - 63)
  const uint64_t f = m >> max(0, min(63, 1022 - e));
  const uint64_t sg = (uint64_t)(int64_t)((int)hw >> 31);
  return ((f ^ sg) - sg) + 0x8080808080808080ull;
}
// digit i of a fixed-point value as a float
__device__ __forceinline__ float digit_raw(uint64_t f, int i) {  // 2^23 + 128 + digit
  const uint32_t w = i < 4 ? (uint32_t)(f >> 32) : (uint32_t)f;
  return __uint_as_float(__byte_perm(w, 0x4b000000u, 0x7650u + (3 - (i & 3))));
}
constexpr float kDigitOff = 8388608.0f + 128.0f;
__device__ __forceinline__ float digit(uint64_t f, int i) { return __fsub_rn(digit_raw(f, i), kDigitOff); }

// the exponent field of a double's magnitude, as an order-preserving integer: |v| <
// 2^(field - 1022); 2047 for infinities and NaN
__device__ __forceinline__ int exp_field(double v) { return (int)(((uint32_t)__double2hiint(v) >> 20) & 0x7ffu); }
// v 2^k (k split in two, so that neither factor over- or underflows)
__device__ __forceinline__ double scale_pow2(double v, int k) {
  const int a = k / 2, b = k - a;
  return (v * __hiloint2double((1023 + a) << 20, 0)) * __hiloint2double((1023 + b) << 20, 0);
}
__device__ __forceinline__ double pow2d(int k) {  // k clamped to the normal range
  return __hiloint2double((1023 + max(-1022, min(1023, k))) << 20, 0);
}

// The recursions of one thread in IEEE double (legendre_fp64.cu's steps), on p / u_p:
// lane 0 lambda(+s) and lane 1 (-1)^(l - l0) lambda(-s) of a ring pair (SPIN), or two ring
// pairs' lambda (spin 0; ONE: only lane 0).
template <bool SPIN, bool ONE>
struct Rec {
  double p0, q0, p1, q1, x0, x1;
  int s0, s1;
  __device__ __forceinline__ void start(const LegArgs &a, int mi, int m, int lane, int s, int pr, bool valid) {
    const PairDev pd = a.pairs[valid ? pr : 0];
    double mant, v = 0.0;
    int e, sc = 0;
    start_value(m, s, pd, a.mpre[mi], &mant, &e);
    if (valid) v = to_scaled(mant, e - a.lexp[(size_t)mi * a.npairs + pr], &sc);
    if (lane == 0) {
      p0 = v;
      q0 = 0.0;
      x0 = pd.x;
      s0 = sc;
    } else {
      p1 = v;
      q1 = 0.0;
      x1 = pd.x;
      s1 = sc;
    }
  }
  __device__ __forceinline__ void step(double2 c) {
    if (SPIN) {
      const double u = fma(c.x, x0, c.y), v = fma(-c.x, x0, c.y);
      const double n0 = fma(u, p0, -q0), n1 = fma(v, p1, -q1);
      q0 = p0;
      p0 = n0;
      q1 = p1;
      p1 = n1;
    } else {
      const double n0 = fma(c.x * x0, p0, -q0);
      q0 = p0;
      p0 = n0;
      if (!ONE) {
        const double n1 = fma(c.x * x1, p1, -q1);
        q1 = p1;
        p1 = n1;
      }
    }
  }
  __device__ __forceinline__ void rescale() {
    if (s0 < 0 && fabs(p0) > kScaleUp) {
      p0 *= kScaleFactor;
      q0 *= kScaleFactor;
      ++s0;
    }
    if (!ONE && s1 < 0 && fabs(p1) > kScaleUp) {
      p1 *= kScaleFactor;
      q1 *= kScaleFactor;
      ++s1;
    }
  }
  // both values zero or below 2^-250
  __device__ __forceinline__ bool dead() const {
    return (s0 < 0 || (p0 == 0.0 && q0 == 0.0)) && (s1 < 0 || (p1 == 0.0 && q1 == 0.0));
  }
  // the fixed-point values (zero below scale 0)
  __device__ __forceinline__ uint64_t fix0(bool settled) const { return fix64(settled || s0 == 0 ? p0 : 0.0); }
  __device__ __forceinline__ uint64_t fix1(bool settled) const { return fix64(settled || s1 == 0 ? p1 : 0.0); }
};

// Exact sum of levels 0 to 3 (D: the ten digit-product sums, integers of at most 2^23,
// or two-term sums of at most 2^24) and the FP32 sum lo of the rest in units of level
// 4, as a double in units of level 0.
__device__ __forceinline__ double level_sum(float L0, float L1, float L2a, float L2b, float L3a, float L3b, float lo) {
  const f2 a = two_sum(L0, L1 * 0x1p-8f);
  const f2 b = two_sum(L2a * 0x1p-16f, L2b * 0x1p-16f), c = two_sum(L3a * 0x1p-24f, L3b * 0x1p-24f);
  const f2 d = two_sum(a.l, b.h), e = two_sum(d.h, c.h);
  const float rest = __fadd_rn(__fadd_rn(__fadd_rn(d.l, e.l), __fadd_rn(b.l, c.l)), lo * 0x1p-32f);
  return (double)a.h + ((double)e.h + (double)rest);
}

// ---- synthesis shapes (see legendre_tc.cu) --------------------------------------
constexpr int kRows = 128, kK = 16, kWin = 16;
constexpr int kLevels = 8;  // TMEM levels: 0 .. 6, and the one the last window's zero digit fills
constexpr int kATile = kRows * kK * 2;
constexpr int kIssuerWarp = 3;
template <int NJ, bool SPIN>
struct Shape {
  static constexpr int NL = SPIN ? 2 : 1;
  static constexpr int NCOL = SPIN ? 8 * NJ : 4 * NJ;
  static constexpr int NCW = NCOL < 8 ? 8 : NCOL;
  static constexpr int N = 2 * NCW;
  static constexpr int NDT = kDig + 2;  // digit tiles per Lambda set: -1 .. 7 (the outer two zero)
  static constexpr int COLS = kLevels * NCW;
  static constexpr int TCOLS = COLS <= 64 ? 64 : (COLS <= 128 ? 128 : 256);
  static constexpr int NV = SPIN ? 4 * NJ : 2 * NJ;
  static constexpr int DTILE = NCW * kK * 2;
  static constexpr int A_BYTES = NL * kDig * kATile;
  static constexpr int B_BYTES = NL * NDT * DTILE;
  static constexpr int NARR = SPIN ? 2 * NJ : NJ;
  static constexpr int ROW = 1 + NARR;                  // double2 per degree: coefficients, a_lm
  static constexpr int STG = kK * ROW;
  static constexpr int PF = (STG + kRows - 1) / kRows;
  static constexpr int ST_BYTES = 2 * STG * 16;
  static constexpr int ACC_BYTES = NCOL * kRows * 8;
  static constexpr int SMEM = A_BYTES + ST_BYTES + B_BYTES + ACC_BYTES + 2 * NV * 4;
  static constexpr int SMEM_FLOOR = (228 * 1024) / (512 / TCOLS + 1) - 1024 + 1;
  static constexpr int SMEM_LAUNCH = SMEM > SMEM_FLOOR ? SMEM : SMEM_FLOOR;
  static constexpr int MINB = SMEM_LAUNCH <= 56 * 1024 ? 4 : (SMEM_LAUNCH <= 74 * 1024 ? 3 : 2);
  static_assert(N % 16 == 0 && N <= 256 && NCOL <= 32 && COLS <= TCOLS && 128 % NV == 0, "shape");
};

// largest exponent field of each a_lm value over a window's degrees lw0 .. lw1
template <int NJ, bool SPIN>
__device__ __forceinline__ void window_bounds(const LegArgs &a, int64_t co, int lw0, int lw1, int *emax) {
  using S = Shape<NJ, SPIN>;
  const int v = threadIdx.x % S::NV;
  int mx = 0;
  for (int l = lw0 + (int)threadIdx.x / S::NV; l <= lw1; l += kRows / S::NV) {
    const double2 q = __ldg(a.pm + (int64_t)(v / 2) * a.ncoef + co + l);
    mx = max(mx, exp_field((v & 1) ? q.y : q.x));
  }
#pragma unroll
  for (int o = S::NV; o < 32; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) < S::NV) atomicMax(emax + v, mx);
}

// the a_lm digit stacks of a K-step (legendre_tc.cu's build_b): array v / 2 holds P (even)
// or s M (odd) of job v / 4 at spin s, map v / 2 at spin 0
template <int NJ, bool SPIN>
__device__ __forceinline__ void build_b(const double2 *stg, const int *emax, unsigned char *Bt) {
  using S = Shape<NJ, SPIN>;
  auto at = [](int r, int k) { return (r / 8) * 256 + (r % 8) * 16 + (k / 8) * 128 + (k % 8) * 2; };
  for (int t = threadIdx.x; t < kK * S::NV; t += kRows) {
    const int k = t % kK, v = t / kK;
    const double2 q = stg[k * S::ROW + 1 + v / 2];
    const uint64_t f = fix64(scale_pow2((v & 1) ? q.y : q.x, 1021 - emax[v]));  // below 1/2
    int col0, col1 = 0, zcol = 0;
    if (SPIN) {
      const int j = v / 4, c = v % 4;
      col0 = 8 * j + c;
      col1 = 8 * j + (c < 2 ? 6 + c : 2 + c);
    } else {
      const int j = v / 2, c = v % 2, odd = k & 1;
      col0 = 4 * j + (odd ? 2 : 0) + c;
      zcol = 4 * j + (odd ? 0 : 2) + c;
    }
#pragma unroll
    for (int dj = 0; dj < kDig; ++dj) {
      const int r = (dj + 1) * S::NCW;
      const uint16_t b = tc::bf16_of(digit(f, dj));
      *reinterpret_cast<uint16_t *>(Bt + at(r + col0, k)) = b;
      if (SPIN)
        *reinterpret_cast<uint16_t *>(Bt + S::NDT * S::DTILE + at(r + col1, k)) = b;
      else
        *reinterpret_cast<uint16_t *>(Bt + at(r + zcol, k)) = 0;
    }
  }
}

// ---- analysis shapes (see legendre_tc_ana.cu) -----------------------------------
constexpr int kTile = 128, kBlk = 8, kN = kDig * kBlk, kColRows = 8, kDCols = 64, kM = 64;
constexpr int kEStride = kN + 4, kKStride = 144;
template <int NJ, bool SPIN>
struct AnaShape64 {
  static constexpr int TH = 128;
  static constexpr int WARPS = TH / 32;
  static constexpr int NP = SPIN ? 1 : 2;
  static constexpr int TILES = NP * TH / kTile;
  static constexpr int NACC = 2;
  static constexpr int LAG = 1;
  static constexpr int NC = 4 * NJ;
  static constexpr int CPW = NC / 4;
  static constexpr int KG = 2 * TH / 8;
  static constexpr int A_LBO = NC * kColRows * 16;
  static constexpr int A_SBO = CPW == 1 ? 64 : 128;
  static constexpr int A_BYTES = KG * A_LBO;
  __host__ __device__ static constexpr int a_at(int c, int j, int h) { return h * A_LBO + (kColRows * c + j) * 16; }
  static constexpr int B_SBO = KG * kKStride;
  static constexpr int B_BYTES = kDig * B_SBO;
  static constexpr int EROWS = CPW * kColRows;
  static constexpr int E_BYTES = WARPS * EROWS * kEStride * 4;
  static constexpr int SMEM = A_BYTES + B_BYTES + E_BYTES;
  static constexpr int TCOLS = NACC * kDCols;
  static constexpr int SMEM_FLOOR = (228 * 1024) / (512 / TCOLS + 1) - 1024 + 1;
  static constexpr int SMEM_LAUNCH = SMEM > SMEM_FLOOR ? SMEM : SMEM_FLOOR;
  static constexpr int V = (SPIN ? 4 : 2) * NJ;
  static constexpr int MINB = NJ == 1 ? 4 : 2;
  static_assert(kColRows * NC <= kM && CPW <= 2, "columns within the MMA's rows");
  static_assert(WARPS == 4 && LAG < NACC, "every warp reads a quarter of every block");
  static_assert((KG - 1) * A_LBO + 7 * A_SBO + 128 <= A_BYTES + B_BYTES, "A operand inside shared memory");
  static_assert(MINB * (SMEM_LAUNCH + 2048) <= 228 * 1024, "CTAs per SM");
};

}  // namespace t64

// ---------------------------------------------------------------------------
// The bound 2^lexp on |p_l| per (m, ring pair), once per plan, from a plain FP32 walk of
// the recursion in difference form (step_polar in mixed_common.cuh: relative errors
// well inside the margin of 1/16 next to the poles too, as cos(theta) >= 0 in every
// pair: 1 - cos(theta) keeps its digits there); not below 2^-90.  A thread
// walks kBoundPairs pairs, which share the conversions of the coefficients.
// ---------------------------------------------------------------------------
constexpr int kBoundPairs = 8;
template <bool SPIN>
__global__ void __launch_bounds__(128) bound_kernel(LegArgs a, signed char *__restrict__ out, unsigned long long *__restrict__ ref) {
  const int mi = blockIdx.y, pb = blockIdx.x * 128 * kBoundPairs + threadIdx.x;
  if (pb >= a.npairs) return;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax;
  const double2 *__restrict__ cf = a.coef + (a.coef_off[mi] - l0);
  float vmax[kBoundPairs];
  int e0[kBoundPairs], e1[kBoundPairs];  // the exponents of the values at the first degree
#pragma unroll
  for (int k = 0; k < kBoundPairs; ++k) {
    vmax[k] = 0.f;
    e1[k] = -70000;
  }
#pragma unroll 1
  for (int t = 0; t < (SPIN ? 2 : 1); ++t) {
    float p[kBoundPairs], d[kBoundPairs], y[kBoundPairs], w[kBoundPairs];  // values p 2^(64 sc), w their weight
    int sc[kBoundPairs];
#pragma unroll
    for (int k = 0; k < kBoundPairs; ++k) {
      const PairDev pd = a.pairs[min(pb + 128 * k, a.npairs - 1)];
      y[k] = (float)(1.0 - pd.x);
      double mant;
      int e;
      start_value(m, t ? -s : s, pd, a.mpre[mi], &mant, &e);
      sc[k] = 0;
      p[k] = 0.f;
      if (mant != 0.0) {
        sc[k] = (e + 32) >= 0 ? (e + 32) / 64 : -((-(e + 32) + 63) / 64);
        p[k] = (float)ldexp(mant, e - 64 * sc[k]);
      }
      (t ? e1[k] : e0[k]) = mant != 0.0 ? ilogb(mant) + e : -70000;
      d[k] = p[k];
      w[k] = sc[k] == 0 ? 1.f : (sc[k] == -1 ? 0x1p-64f : 0.f);
    }
    for (int l = l0; l <= lmax; ++l) {
      const double2 c = __ldg(cf + l);
      const float ca = (float)c.x, cb = (float)(c.x - 2.0 + (t ? -c.y : c.y));
      const bool check = ((l - l0) & 3) == 3;
#pragma unroll
      for (int k = 0; k < kBoundPairs; ++k) {
        vmax[k] = fmaxf(vmax[k], fabsf(p[k]) * w[k]);
        d[k] = fmaf(fmaf(-ca, y[k], cb), p[k], d[k]);
        p[k] += d[k];
        if (check && sc[k] < 0 && fabsf(p[k]) > 0x1p32f) {
          p[k] *= 0x1p-64f;
          d[k] *= 0x1p-64f;
          w[k] = ++sc[k] == 0 ? 1.f : (sc[k] == -1 ? 0x1p-64f : 0.f);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kBoundPairs; ++k) vmax[k] = fmaxf(vmax[k], fabsf(p[k]) * w[k]);
  }
  unsigned long long best = 0;
#pragma unroll
  for (int k = 0; k < kBoundPairs; ++k) {
    if (pb + 128 * k >= a.npairs) break;
    int e = -90;
    if (vmax[k] > 0.f) {
      int ev;
      frexpf(vmax[k] * 1.0625f, &ev);
      e = max(e, min(ev, 100));
    }
    out[(size_t)mi * a.npairs + pb + 128 * k] = (signed char)e;
    const int d0 = e0[k] - e, d1 = SPIN ? e1[k] - e : d0, lanes = (d0 >= -kRefNear ? 1 : 0) | (d1 >= -kRefNear ? 2 : 0);
    const int p = pb + 128 * k;
    const unsigned long long key = ref_key(p == a.npairs - 1 && lanes == 3, max(d0, d1), p, lanes);
    best = key > best ? key : best;
  }
  atomicMax(ref + mi, best);
}

// ---------------------------------------------------------------------------
// synthesis (columns and pipeline as in legendre_tc.cu)
// ---------------------------------------------------------------------------
template <int NJ, bool SPIN>
__device__ __forceinline__ void tc64_syn_body(const LegArgs &a, const int2 item, unsigned char *smem) {
  using namespace t64;
  using S = Shape<NJ, SPIN>;
  constexpr int NL = S::NL, NCOL = S::NCOL;
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tslot;
  __shared__ volatile int stop;
  __shared__ int kstart[kRows / 32];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int mi = item.x;
  const int p = item.y + tid;
  const bool valid = p < a.npairs;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax;
  const int nks = (lmax - l0 + kK) / kK;
  const int64_t co = a.coef_off[mi] - l0;
  const double2 *__restrict__ cf = a.coef + co;
  unsigned char *const Abuf = smem;
  double2 *const stage = reinterpret_cast<double2 *>(smem + S::A_BYTES);
  unsigned char *const Bt = smem + S::A_BYTES + S::ST_BYTES;
  double *const accs = reinterpret_cast<double *>(Bt + S::B_BYTES);
  int *const emax = reinterpret_cast<int *>(Bt + S::B_BYTES + S::ACC_BYTES);

  double2 pf[S::PF];
  auto prefetch = [&](int ks) {
    const int lb = l0 + ks * kK;
#pragma unroll
    for (int i = 0; i < S::PF; ++i) {
      const int e = tid + i * kRows;
      pf[i] = make_double2(0.0, 0.0);
      if (e < S::STG) {
        const int k = e / S::ROW, c = e % S::ROW, l = lb + k;
        if (l <= lmax) pf[i] = c < 1 ? __ldg(cf + l) : __ldg(a.pm + (int64_t)(c - 1) * a.ncoef + co + l);
        if (SPIN && c > 0 && !(c & 1) && (k & 1)) pf[i] = make_double2(-pf[i].x, -pf[i].y);  // s M
      }
    }
  };
  auto stage_store = [&](int ks) {
    double2 *dst = stage + (ks & 1) * S::STG;
#pragma unroll
    for (int i = 0; i < S::PF; ++i) {
      const int e = tid + i * kRows;
      if (e < S::STG) dst[e] = pf[i];
    }
  };
  if (warp == 0) tc::tmem_alloc(&tslot, S::TCOLS);
  if (tid == 0) {
    tc::bar_init(&mbar);
    stop = 0;
  }
  for (int i = tid; i < S::B_BYTES / 16; i += kRows) reinterpret_cast<uint4 *>(Bt)[i] = make_uint4(0, 0, 0, 0);
  if (tid < 2 * S::NV) emax[tid] = 0;

  // the recursions up to the warp's first K-step with a value at scale 0 (below, the
  // values are under 2^-250); the CTA starts at its warps' earliest
  Rec<SPIN, !SPIN> rec;
  rec.p1 = rec.q1 = rec.x1 = 0.0;
  rec.s1 = 0;
  rec.start(a, mi, m, 0, s, p, valid);
  if (SPIN) rec.start(a, mi, m, 1, -s, p, valid);
  int kw = 0;
  while (kw < nks && __all_sync(0xffffffffu, rec.dead())) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int l = l0 + kw * kK + 8 * h + q;
        rec.step(l <= lmax ? __ldg(cf + l) : make_double2(0.0, 0.0));
      }
      rec.rescale();
    }
    ++kw;
  }
  if ((tid & 31) == 0) kstart[warp] = kw;
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = tslot;
  const uint32_t lane = tbase + ((uint32_t)(warp * 32) << 16);
  int ks0 = kstart[0];
#pragma unroll
  for (int w = 1; w < kRows / 32; ++w) ks0 = min(ks0, kstart[w]);
  if (ks0 < nks) {
    prefetch(ks0);
    stage_store(ks0);
  }
#pragma unroll
  for (int c = 0; c < NCOL; ++c) accs[c * kRows + tid] = 0.0;
  bool settled = __all_sync(0xffffffffu, rec.s0 == 0 && rec.s1 == 0);

  // 8 degrees from the staged rows: the digits packed per pair of degrees
  auto part = [&](const bool st, const double2 *rows, uint32_t (&pk)[NL][kDig][4]) __attribute__((always_inline)) {
    float2 hold[kDig];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint64_t f0 = rec.fix0(st), f1 = SPIN ? rec.fix1(st) : 0ull;
#pragma unroll
      for (int i = 0; i < kDig; ++i) {
        float2 d;
        if (SPIN) d = add2(make_float2(digit_raw(f0, i), digit_raw(f1, i)), both(-kDigitOff));
        else d = make_float2(digit(f0, i), 0.f);
        if (!(q & 1)) {
          hold[i] = d;
        } else {
          pk[0][i][q >> 1] = tc::pack_bf16(hold[i].x, d.x);
          if (SPIN) pk[NL - 1][i][q >> 1] = tc::pack_bf16(hold[i].y, d.y);
        }
      }
      rec.step(rows[q * S::ROW]);
    }
  };
  auto store_a = [&](int q0, const uint32_t (&pk)[NL][kDig][4]) {
#pragma unroll
    for (int t = 0; t < NL; ++t)
#pragma unroll
      for (int i = 0; i < kDig; ++i)
        *reinterpret_cast<uint4 *>(Abuf + (t * kDig + i) * kATile + (tid / 8) * 256 + (q0 / 8) * 128 + (tid % 8) * 16) =
            make_uint4(pk[t][i][0], pk[t][i][1], pk[t][i][2], pk[t][i][3]);
  };
  // Lambda digit i of set t meets the a_lm digits (j0, j0 + 1), j0 = -(i mod 2), ..., while
  // i + j0 <= 6, into levels i + j0 and i + j0 + 1; in a window's first K-step the set-0,
  // digit-0 products overwrite levels 0 .. 7
  const uint64_t adesc0 = tc::mat_desc(tc::smem_u32(Abuf), 128, 256);
  const uint64_t bdesc0 = tc::mat_desc(tc::smem_u32(Bt), 128, 256);
  auto issue = [&](int ks) {
    tc::fence_after();
    constexpr uint32_t idesc = tc::instr_desc(kRows, S::N);
    const bool first = (ks % kWin) == 0 || ks == ks0;
#pragma unroll
    for (int t = 0; t < NL; ++t)
#pragma unroll
      for (int i = 0; i < kDig; ++i)
#pragma unroll
        for (int j0 = -(i & 1); i + j0 <= kDig - 1; j0 += 2) {
          const uint64_t ad = adesc0 + (uint64_t)(((t * kDig + i) * kATile) >> 4);
          const uint64_t bd = bdesc0 + (uint64_t)((t * S::NDT * S::DTILE + (j0 + 1) * S::DTILE) >> 4);
          tc::mma_bf16(tbase + (i + j0) * S::NCW, ad, bd, idesc, (first && t == 0 && i == 0) ? 0u : 1u);
        }
    tc::mma_commit(&mbar);
  };
  // the a_lm value whose column c is (its exponent scales the column)
  auto value_of = [](int c) {
    if (!SPIN) return 2 * (c / 4) + (c & 1);
    const int j = c / 8, k = c % 8;
    return 4 * j + (k < 4 ? k : (k < 6 ? k - 2 : k - 6));
  };
  auto readout = [&](const int *em) {
#pragma unroll
    for (int c0 = 0; c0 < NCOL; c0 += 4) {
      uint32_t dv[kLevels - 1][4];
#pragma unroll
      for (int k = 0; k < kLevels - 1; ++k) tc::tmem_ld4(lane + k * S::NCW + c0, dv[k]);
      tc::tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        auto L = [&](int k) { return __uint_as_float(dv[k][c]); };
        const float lo = __fadd_rn(__fadd_rn(L(6) * 0x1p-16f, L(5) * 0x1p-8f), L(4));
        const double t = level_sum(L(0), L(1), L(2), 0.f, L(3), 0.f, lo);
        const int e = em[value_of(c0 + c)];
        double &acc = accs[(c0 + c) * kRows + tid];
        acc += scale_pow2(t, e - 1021 - 14);
      }
    }
  };

  int ncommit = 0, nwaited = 0;
  bool ok = true;
  auto wait_mma = [&]() -> bool {
    const uint32_t par = (uint32_t)(ncommit - 1) & 1u;
    return tc::bar_try(&mbar, par) || tc::bar_wait_or(&mbar, par, &stop);
  };
  for (int ks = ks0; ks < nks; ++ks) {
    const int lb = l0 + ks * kK;
    int *const em = emax + ((ks / kWin) & 1) * S::NV;
    if (ks % kWin == 0 || ks == ks0) {
      const int lw1 = l0 + (ks / kWin + 1) * kWin * kK - 1;
      window_bounds<NJ, SPIN>(a, co, lb, lw1 < lmax ? lw1 : lmax, em);
      __syncthreads();
      // the other window's, for later: every thread has left the readout that reads it
      if (tid < S::NV) emax[(((ks / kWin) & 1) ^ 1) * S::NV + tid] = 0;
    }
    const bool wlive = ks >= kw;
    const double2 *rows = stage + (ks & 1) * S::STG;
    if (ks + 1 < nks) prefetch(ks + 1);
    bool fail = false;
#pragma unroll 1
    for (int q0 = 0; q0 < kK; q0 += 8) {
      uint32_t pk[NL][kDig][4];
      if (wlive) {
        if (settled) {
          part(true, rows + q0 * S::ROW, pk);
        } else {
          part(false, rows + q0 * S::ROW, pk);
          rec.rescale();
          settled = __all_sync(0xffffffffu, rec.s0 == 0 && rec.s1 == 0);
        }
      } else {
#pragma unroll
        for (int t = 0; t < NL; ++t)
#pragma unroll
          for (int i = 0; i < kDig; ++i)
#pragma unroll
            for (int q = 0; q < 4; ++q) pk[t][i][q] = 0u;
      }
      if (q0 == 0 && ncommit > nwaited) {
        fail = !wait_mma();
        nwaited = ncommit;
      }
      if (!fail) store_a(q0, pk);
      if (q0 == 0 && !fail) build_b<NJ, SPIN>(rows, em, Bt);
    }
    if (ks + 1 < nks) stage_store(ks + 1);
    tc::fence_async_smem();
    if (fail) stop = 1;
    __syncthreads();
    if (warp == kIssuerWarp && tc::elect_one()) issue(ks);
    ++ncommit;
    if (ks % kWin == kWin - 1 || ks == nks - 1) {
      fail = !wait_mma();
      nwaited = ncommit;
      if (__syncthreads_or(fail || stop)) {
        ok = false;
        break;
      }
      tc::fence_after();
      readout(em);
      tc::fence_before();
    }
  }
  if (!ok) {
    if (tid == 0) atomicOr(a.err, 1);
    if (ncommit > nwaited) tc::bar_wait(&mbar, (uint32_t)(ncommit - 1) & 1u);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, S::TCOLS);
  if (!ok || !valid) return;
  const double u = pow2d(a.lexp[(size_t)mi * a.npairs + p]);
  auto colsum = [&](int c) { return u * accs[c * kRows + tid]; };
  if (SPIN) {
    const double sig = (as & 1) ? -1.0 : 1.0;
    const double h0 = ((l0 + m) & 1) ? -0.5 : 0.5;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const double n1r = colsum(8 * j + 0), n1i = colsum(8 * j + 1);
      const double s4r = colsum(8 * j + 2), s4i = colsum(8 * j + 3);
      const double n2r = colsum(8 * j + 4), n2i = colsum(8 * j + 5);
      const double s3r = colsum(8 * j + 6), s3i = colsum(8 * j + 7);
      const double ar = n1r + sig * n2r, ai = n1i + sig * n2i;
      const double br = sig * n2r - n1r, bi = sig * n2i - n1i;
      const double cr = s3r + sig * s4r, ci = s3i + sig * s4i;
      const double dr = sig * s4r - s3r, di = sig * s4i - s3i;
      double2 qn = make_double2(-0.5 * ar, -0.5 * ai);
      double2 un = make_double2(0.5 * bi, -0.5 * br);
      double2 qs = make_double2(-h0 * cr, -h0 * ci);
      double2 us = make_double2(h0 * di, -h0 * dr);
      if (m == 0) qn.y = qs.y = un.y = us.y = 0.0;
      double2 *oq = a.phase + (((size_t)(2 * j) * a.nm + mi) * a.npairs + p) * 2;
      double2 *ou = a.phase + (((size_t)(2 * j + 1) * a.nm + mi) * a.npairs + p) * 2;
      oq[0] = qn;
      oq[1] = qs;
      ou[0] = un;
      ou[1] = us;
    }
  } else {
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const double e0 = colsum(4 * j + 0), e1 = colsum(4 * j + 1);
      const double o0 = colsum(4 * j + 2), o1 = colsum(4 * j + 3);
      double2 fn = make_double2(e0 + o0, e1 + o1), fs = make_double2(e0 - o0, e1 - o1);
      if (m == 0) fn.y = fs.y = 0.0;
      double2 *o = a.phase + (((size_t)j * a.nm + mi) * a.npairs + p) * 2;
      o[0] = fn;
      o[1] = fs;
    }
  }
}

// ---------------------------------------------------------------------------
// analysis (K entries, columns and pipeline as in legendre_tc_ana.cu; the partial
// sums, as in legendre_fp64.cu, in items that walk a group of tiles into one slot); false
// if the item is left to the IEEE sums
// ---------------------------------------------------------------------------
template <int NJ, bool SPIN>
__device__ __forceinline__ bool tc64_ana_body(const LegArgs &a, const int4 item, unsigned char *smem) {
  using namespace t64;
  using S = AnaShape64<NJ, SPIN>;
  constexpr int NC = S::NC, V = S::V, TH = S::TH, NP = S::NP;
  constexpr int NACC = S::NACC, LAG = S::LAG;
  __shared__ __align__(8) uint64_t full[NACC], freeb[NACC], mine[S::WARPS];
  __shared__ uint32_t tslot;
  __shared__ int vmax[NC], eqmax[NC];
  __shared__ int tstart[S::WARPS];
  __shared__ volatile int stop;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int mi = item.x, ng = item.z & 255;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax, nl = lmax - l0 + 1;
  const double2 *__restrict__ cf = a.coef + (a.coef_off[mi] - l0);
  double *const outp = a.part + a.part_off[mi] + (int64_t)(item.z >> 8) * nl * V;
  const double sg0 = ((l0 + m) & 1) ? -1.0 : 1.0;
  unsigned char *const Abuf = smem;
  unsigned char *const Bbuf = smem + S::A_BYTES;
  float *const Ebuf = reinterpret_cast<float *>(smem + S::A_BYTES + S::B_BYTES) + warp * S::EROWS * kEStride;

  if (warp == 0) tc::tmem_alloc(&tslot, S::TCOLS);
  if (tid == 0) {
#pragma unroll
    for (int x = 0; x < NACC; ++x) {
      tc::bar_init(&full[x], S::WARPS);
      tc::bar_init(&freeb[x], 4);
    }
#pragma unroll
    for (int w = 0; w < S::WARPS; ++w) tc::bar_init(&mine[w], 1);
    stop = 0;
  }
  for (int i = tid; i < S::A_BYTES / 16; i += TH) reinterpret_cast<uint4 *>(Abuf)[i] = make_uint4(0, 0, 0, 0);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tbase = tslot;
  const uint32_t tlane = tbase + ((uint32_t)((warp & 3) * 32) << 16);
  auto zero_acc = [&](uint32_t ta) {
#pragma unroll
    for (int q = 0; q < kN / 8; ++q) tc::tmem_zero8(ta + q * 8);
  };
  if (warp < 4) {
#pragma unroll
    for (int x = 0; x < NACC; ++x) zero_acc(tlane + x * kDCols);
    tc::tmem_wait_st();
  }
  tc::fence_before();
  const uint64_t adesc0 = tc::mat_desc(tc::smem_u32(Abuf), S::A_LBO, S::A_SBO);
  const uint64_t bdesc0 = tc::mat_desc(tc::smem_u32(Bbuf), kKStride, S::B_SBO);
  constexpr uint32_t idesc = tc::instr_desc(kM, kN, true);

  // the K entries of pair p (spin: both of its lanes; spin 0: lane t) for every column
  auto load_pair = [&](int p, int t, double (&gv)[2][NC]) __attribute__((always_inline)) {
    const bool south = a.pairs[p].south;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      if (!SPIN) {
        const double2 *gp = a.phase + (((size_t)j * a.nm + mi) * a.npairs + p) * 2;
        const double2 gn = gp[0], gs = south ? gp[1] : make_double2(0.0, 0.0);
        gv[t][4 * j + 0] = gn.x + gs.x;
        gv[t][4 * j + 1] = gn.y + gs.y;
        gv[t][4 * j + 2] = gn.x - gs.x;
        gv[t][4 * j + 3] = gn.y - gs.y;
      } else {
        const double2 *gq = a.phase + (((size_t)(2 * j) * a.nm + mi) * a.npairs + p) * 2;
        const double2 *gu = a.phase + (((size_t)(2 * j + 1) * a.nm + mi) * a.npairs + p) * 2;
        const double2 qn = gq[0], un = gu[0];
        const double2 qs = south ? gq[1] : make_double2(0.0, 0.0), us = south ? gu[1] : make_double2(0.0, 0.0);
        gv[0][4 * j + 0] = qn.x - un.y;          // T1: l+ W+_N
        gv[0][4 * j + 1] = qn.y + un.x;
        gv[0][4 * j + 2] = sg0 * (qs.x + us.y);  // s T2: l+ W-_S'
        gv[0][4 * j + 3] = sg0 * (qs.y - us.x);
        gv[1][4 * j + 0] = sg0 * (qs.x - us.y);  // T1: s l- W+_S'
        gv[1][4 * j + 1] = sg0 * (qs.y + us.x);
        gv[1][4 * j + 2] = qn.x + un.y;          // s T2: s l- W-_N
        gv[1][4 * j + 3] = qn.y - un.x;
      }
    }
  };
  // The size of column c's largest entry in gv, |G u_p|, as an exponent field (scaled by
  // 2^200, so that u_p keeps it positive; infinities and NaN: 4000)
  auto size_of = [&](const double (&gv)[2][NC], const int (&lexp)[NP], int c, int lanes) __attribute__((always_inline)) {
    int mx = 0;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int e = size_field(gv[t][c]);
      if (e > 0 && (lanes >> t & 1)) mx = max(mx, e == 2047 ? 4000 : e + 200 + lexp[SPIN ? 0 : t]);
    }
    return mx;
  };

  // Whether the item's values range too far for fixed point (it then returns false): at every
  // degree the sum comes from the pairs between two latitudes, which close in on the
  // reference pair towards the first degree (next to the equator, but for m about |s| > 5),
  // and the others' Lambda falls away exponentially; so no pair's |G u_p| may exceed
  // 2^kWideRange times the largest of the 32 about that pair (of the values +s, -s that are
  // near their bound there; columns of zeros there are zero).  One warp finds those; each
  // pass compares its own.
  if (warp == 0) {
    const RefPair rp = ref_of(a.ref[mi]);
    const int p = max(min(rp.pair + 15, a.npairs - 1) - lane, -1);
    int mx[NC];
    {
      double gv[2][NC];
      int lexp[NP];
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c) gv[t][c] = 0.0;
#pragma unroll
      for (int t = 0; t < NP; ++t) lexp[t] = p >= 0 ? a.lexp[(size_t)mi * a.npairs + p] : 0;
      if (p >= 0) load_pair(p, 0, gv);
#pragma unroll
      for (int c = 0; c < NC; ++c) mx[c] = size_of(gv, lexp, c, SPIN ? rp.lanes : 3);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int e = __reduce_max_sync(0xffffffffu, mx[c]);
      if (lane == 0) eqmax[c] = e;
    }
  }
  bool wide = false;

  int ib = 0;
  int nmine = 0, nmine_done = 0;
  bool ok = true;
  auto wait_warp = [&](uint64_t *bar, uint32_t parity) -> bool {
    if (__all_sync(0xffffffffu, tc::bar_try(bar, parity))) return true;
    const bool r = tc::bar_wait_or(bar, parity, &stop);
    return __all_sync(0xffffffffu, r);
  };
  auto give_up = [&]() {
    if (lane == 0) stop = 1;
    ok = false;
  };

#pragma unroll 1
  for (int gi = 0; gi < ng && !wide; gi += S::TILES) {
    int pr[NP], lexp[NP];
    bool valid[NP];
    double gv[2][NC];
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
      for (int c = 0; c < NC; ++c) gv[t][c] = 0.0;
#pragma unroll
    for (int t = 0; t < NP; ++t) {
      pr[t] = (item.y + gi) * kTile + NP * tid + t;
      valid[t] = pr[t] < min(a.npairs, (item.y + ng) * kTile);
      lexp[t] = valid[t] ? a.lexp[(size_t)mi * a.npairs + pr[t]] : 0;
      if (valid[t]) load_pair(pr[t], t, gv);
    }
    // the recursions up to the warp's first block with a value at scale 0
    Rec<SPIN, false> rec;
    rec.start(a, mi, m, 0, s, pr[0], valid[0]);
    rec.start(a, mi, m, 1, SPIN ? -s : 0, pr[NP - 1], valid[NP - 1]);
    int lw = l0;  // this warp's first block
    while (lw <= lmax && __all_sync(0xffffffffu, rec.dead())) {
#pragma unroll
      for (int q = 0; q < kBlk; ++q) rec.step(__ldg(cf + min(lw + q, lmax)));
      rec.rescale();
      lw += kBlk;
    }
    __syncthreads();  // the previous tile's products are complete (its last accumulator was read)
    if (stop) {
      ok = false;
      break;
    }
    if (tid < NC) vmax[tid] = 0;
    if (lane == 0) tstart[warp] = lw;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c) {  // column bounds over the tile
      const int mx = __reduce_max_sync(0xffffffffu, size_of(gv, lexp, c, 3));
      if (lane == 0) atomicMax(&vmax[c], mx);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NC; ++c)
      wide = wide || (vmax[c] > 0 && (vmax[c] > eqmax[c] + kWideRange || vmax[c] < kFieldMin + 200 || vmax[c] >= kFieldMax + 200));
    if (wide) break;  // the same for every thread; no product is in flight here
    int lstart = tstart[0];
#pragma unroll
    for (int w = 1; w < S::WARPS; ++w) lstart = min(lstart, tstart[w]);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        // |G u_p 2^(1221 - vmax)| < 1/2
        const uint64_t f = fix64(scale_pow2(gv[t][c], lexp[SPIN ? 0 : t] + 1221 - vmax[c]));
        unsigned char *dst = Abuf + S::a_at(c, 0, t * (TH / 8) + tid / 8) + (tid % 8) * 2;
#pragma unroll
        for (int j = 0; j < kDig; ++j) *reinterpret_cast<uint16_t *>(dst + j * 16) = tc::bf16_of(digit(f, j));
      }
    }
    if (gi == 0)
      for (int i = tid; i < (min(lstart, lmax + 1) - l0) * V; i += TH) outp[i] = 0.0;
    tc::fence_async_smem();
    __syncthreads();
    if (lstart > lmax) continue;

    bool settled = __all_sync(0xffffffffu, rec.s0 == 0 && rec.s1 == 0);
    auto part = [&](const bool st, int lb4, uint32_t (&pk)[2][kDig][2]) __attribute__((always_inline)) {
      float2 hold[kDig];
      double2 cv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) cv[q] = __ldg(cf + min(lb4 + q, lmax));
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint64_t f0 = rec.fix0(st), f1 = rec.fix1(st);
#pragma unroll
        for (int i = 0; i < kDig; ++i) {
          const float2 d = add2(make_float2(digit_raw(f0, i), digit_raw(f1, i)), both(-kDigitOff));
          if (!(q & 1)) {
            hold[i] = d;
          } else {
            pk[0][i][q >> 1] = tc::pack_bf16(hold[i].x, d.x);
            pk[1][i][q >> 1] = tc::pack_bf16(hold[i].y, d.y);
          }
        }
        rec.step(cv[q]);
      }
    };
    auto store_b = [&](int h, const uint32_t (&pk)[2][kDig][2]) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int i = 0; i < kDig; ++i)
          *reinterpret_cast<uint2 *>(Bbuf + i * S::B_SBO + (t * (TH / 8) + tid / 8) * kKStride + (tid % 8) * 16 + h * 8) =
              make_uint2(pk[t][i][0], pk[t][i][1]);
    };
    auto issue = [&](int xb) {
      tc::fence_after();
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const int kk = t * (TH / 16) + 2 * warp + hh;
          const uint64_t ad = adesc0 + (uint64_t)((2 * kk * S::A_LBO) >> 4);
          const uint64_t bd = bdesc0 + (uint64_t)((2 * kk * kKStride) >> 4);
          tc::mma_bf16(tbase + xb * kDCols, ad, bd, idesc, 1u);
        }
      tc::mma_commit(&mine[warp]);
      tc::mma_commit(&full[xb]);
    };
    auto epi_read = [&](int ibp) {
      const int xb = ibp % NACC;
      if (!wait_warp(&full[xb], (uint32_t)(ibp / NACC) & 1u)) {
        give_up();
        return;
      }
      tc::fence_after();
      const uint32_t ta = tlane + xb * kDCols;
      uint32_t v[kN / 8][8];
#pragma unroll
      for (int q = 0; q < kN / 8; ++q) tc::tmem_ld8(ta + q * 8, v[q]);
      tc::tmem_wait_ld();
      zero_acc(ta);
      if (lane < S::EROWS) {
        float4 *er = reinterpret_cast<float4 *>(Ebuf + lane * kEStride);
#pragma unroll
        for (int q = 0; q < kN / 8; ++q)
#pragma unroll
          for (int r = 0; r < 2; ++r)
            er[2 * q + r] = make_float4(__uint_as_float(v[q][4 * r]), __uint_as_float(v[q][4 * r + 1]),
                                        __uint_as_float(v[q][4 * r + 2]), __uint_as_float(v[q][4 * r + 3]));
      }
      tc::tmem_wait_st();
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::bar_arrive(&freeb[xb]);
    };
    const int odeg = lane & 7, epart = lane >> 3;
    const int ecol = S::CPW == 1 ? 0 : (epart & 1);
    const int ocol = S::CPW * (warp & 3) + ecol;
    const bool oact = S::CPW == 1 ? epart == 0 : epart < 2;
    auto out_at = [&](int lbp, bool &neg) -> double * {
      const int l = lbp + odeg, j = ocol >> 2, cc = ocol & 3;
      neg = false;
      if (!oact || l > lmax) return nullptr;
      if (SPIN) {
        neg = cc >= 2 && (odeg & 1);
        return outp + (int64_t)(l - l0) * V + 4 * j + cc;
      }
      return (cc >> 1) == (odeg & 1) ? outp + (int64_t)(l - l0) * V + 2 * j + (cc & 1) : nullptr;
    };
    const int vm = vmax[ocol];
    auto epi_sum = [&](double *o, bool neg, double prev) {
      const float *e = Ebuf + ecol * kColRows * kEStride + odeg;
      auto D = [&](int i, int j) { return e[j * kEStride + i * 8]; };  // sum of G_j L_i
      // levels 4 to 6 in FP32: a lane takes rows j = q and q + 4 (row 7 is zero); the
      // products it meets above level 6 belong to the sum too
      float lo = 0.f;
#pragma unroll
      for (int r = 0; r < (S::CPW == 1 ? 1 : 2); ++r) {
        const int q = S::CPW == 1 ? epart : (epart >> 1) + 2 * r;
        const float *er = e + q * (kEStride - 8) + 32;  // D(4 - q, q)
        const float *ew = e + (q + 4) * kEStride;       // D(0, q + 4)
        const float f = q == 0 ? 1.f : (q == 1 ? 0x1p-8f : (q == 2 ? 0x1p-16f : 0x1p-24f));
        lo = __fadd_rn(lo, __fmaf_rn(__fmaf_rn(er[16], 0x1p-8f, er[8]), 0x1p-8f, er[0]));
        lo = __fmaf_rn(f, __fmaf_rn(__fmaf_rn(ew[16], 0x1p-8f, ew[8]), 0x1p-8f, ew[0]), lo);
      }
      if (S::CPW == 1) lo = __fadd_rn(lo, __shfl_xor_sync(0xffffffffu, lo, 8));
      lo = __fadd_rn(lo, __shfl_xor_sync(0xffffffffu, lo, 16));
      if (o) {
        const double t = level_sum(D(0, 0), __fadd_rn(D(1, 0), D(0, 1)), __fadd_rn(D(2, 0), D(1, 1)), D(0, 2),
                                   __fadd_rn(D(3, 0), D(2, 1)), __fadd_rn(D(1, 2), D(0, 3)), lo);
        const double val = scale_pow2(t, vm - 1221 - 14);
        *o = prev + (neg ? -val : val);
      }
      __syncwarp();
    };

    int lb = lstart;
    const int ib0 = ib;
#pragma unroll 1
    for (; lb <= lmax; lb += kBlk, ++ib) {
      const int xb = ib % NACC;
      const bool turn = ib - LAG >= ib0;
      bool neg_prev = false;
      double *const o_prev = turn ? out_at(lb - LAG * kBlk, neg_prev) : nullptr;
      double prev = 0.0;
      if (o_prev && gi > 0) asm volatile("ld.global.f64 %0, [%1];" : "=d"(prev) : "l"(o_prev));
      const bool live = lb >= lw;
      if (live) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t pk[2][kDig][2];
          if (settled) part(true, lb + 4 * h, pk);
          else part(false, lb + 4 * h, pk);
          if (h == 0 && nmine > nmine_done) {
            if (!wait_warp(&mine[warp], (uint32_t)(nmine - 1) & 1u)) break;
            nmine_done = nmine;
          }
          store_b(h, pk);
        }
        if (nmine > nmine_done) {
          give_up();
          break;
        }
        if (!settled) {
          rec.rescale();
          settled = __all_sync(0xffffffffu, rec.s0 == 0 && rec.s1 == 0);
        }
        tc::fence_async_smem();
        __syncwarp();
      }
      if (ib >= NACC && !wait_warp(&freeb[xb], (uint32_t)(ib / NACC - 1) & 1u)) {
        give_up();
        break;
      }
      if (live) {
        if (tc::elect_one()) issue(xb);
        __syncwarp();
        ++nmine;
      } else if (lane == 0) {
        tc::bar_arrive(&full[xb]);
      }
      if (turn) {
        epi_read(ib - LAG);
        if (!ok) break;
        epi_sum(o_prev, neg_prev, prev);
      }
    }
    if (!ok) continue;
#pragma unroll 1
    for (int k = ib - LAG > ib0 ? ib - LAG : ib0; k < ib; ++k) {
      bool neg;
      double *o = out_at(lb - (ib - k) * kBlk, neg);
      const double prev = (o && gi > 0) ? *o : 0.0;
      epi_read(k);
      if (!ok) break;
      epi_sum(o, neg, prev);
    }
  }
  if (!ok && lane == 0) atomicOr(a.err, 1);  // each warp its own (see legendre_tc_ana.cu)
  if (nmine > nmine_done) tc::bar_wait(&mine[warp], (uint32_t)(nmine - 1) & 1u);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tbase, S::TCOLS);
  return !wide;
}

// ---------------------------------------------------------------------------
// kernels and launchers (plans, and batches: item.w selects the plan's record)
// ---------------------------------------------------------------------------
template <int NJ, bool SPIN>
__device__ __forceinline__ void tc64_syn_item(const LegArgs &a, const int2 item, unsigned char *smem) {
  if (!a.wide_syn[item.x]) tc64_syn_body<NJ, SPIN>(a, item, smem);
  else if constexpr (SPIN) leg_syn_spin_body<NJ>(a, item);
  else leg_syn_s0_body<NJ>(a, item);
}
template <int NJ, bool SPIN>
__device__ __forceinline__ void tc64_ana_item(const LegArgs &a, const int4 item, unsigned char *smem) {
  if (ref_of(a.ref[item.x]).near && tc64_ana_body<NJ, SPIN>(a, item, smem)) return;
  __syncthreads();
  double (*const red)[32] = reinterpret_cast<double (*)[32]>(smem);
#pragma unroll 1
  for (int gi = 0; gi < (item.z & 255); ++gi) {  // tile after tile into the item's slot
    if constexpr (SPIN) leg_ana_spin_body<NJ, 1>(a, item, gi, red);
    else leg_ana_s0_body<NJ, 1>(a, item, gi, red);
  }
}
template <int NJ, bool SPIN>
__global__ void __launch_bounds__(t64::kRows, (t64::Shape<NJ, SPIN>::MINB)) tc64_syn(LegArgs a) {
  extern __shared__ __align__(128) unsigned char tc64_smem[];
  tc64_syn_item<NJ, SPIN>(a, a.syn_items[blockIdx.x], tc64_smem);
}
template <int NJ, bool SPIN>
__global__ void __launch_bounds__(t64::kRows, (t64::Shape<NJ, SPIN>::MINB))
    tc64_syn_batch(const LegArgs *__restrict__ args, const int4 *__restrict__ items) {
  extern __shared__ __align__(128) unsigned char tc64_smem[];
  const int4 it = items[blockIdx.x];
  tc64_syn_item<NJ, SPIN>(args[it.w], make_int2(it.x, it.y), tc64_smem);
}
template <int NJ, bool SPIN>
__global__ void __launch_bounds__((t64::AnaShape64<NJ, SPIN>::TH), (t64::AnaShape64<NJ, SPIN>::MINB)) tc64_ana(LegArgs a) {
  extern __shared__ __align__(128) unsigned char tc64_smem[];
  tc64_ana_item<NJ, SPIN>(a, a.ana_items[blockIdx.x], tc64_smem);
}
template <int NJ, bool SPIN>
__global__ void __launch_bounds__((t64::AnaShape64<NJ, SPIN>::TH), (t64::AnaShape64<NJ, SPIN>::MINB))
    tc64_ana_batch(const LegArgs *__restrict__ args, const int4 *__restrict__ items) {
  extern __shared__ __align__(128) unsigned char tc64_smem[];
  const int4 it = items[blockIdx.x];
  tc64_ana_item<NJ, SPIN>(args[it.w], make_int4(it.x, it.y, it.z, 0), tc64_smem);
}

// f.template operator()<NJ, SPIN>() for the shapes the kernels are built for
template <int NJ, bool SPIN>
struct ShapeTag {
  static constexpr int nj = NJ;
  static constexpr bool spin = SPIN;
};
template <class F>
static cudaError_t syn_shape(int spin, int nj, F &&f) {
  if (spin == 0) {
    switch (nj) {
      case 1: return f(ShapeTag<1, false>{});
      case 2: return f(ShapeTag<2, false>{});
      case 4: return f(ShapeTag<4, false>{});
    }
  } else {
    switch (nj) {
      case 1: return f(ShapeTag<1, true>{});
      case 2: return f(ShapeTag<2, true>{});
    }
  }
  return cudaErrorInvalidValue;
}
template <class F>
static cudaError_t ana_shape(int spin, int nj, F &&f) {
  if (nj == 1) return spin ? f(ShapeTag<1, true>{}) : f(ShapeTag<1, false>{});
  if (nj == 2) return spin ? f(ShapeTag<2, true>{}) : f(ShapeTag<2, false>{});
  return cudaErrorInvalidValue;
}
bool tc64_syn_supported(int spin, int nj) { return spin ? nj <= 2 : nj <= 4; }
bool tc64_ana_supported(int, int nj) { return nj <= 2; }
int tc64_ana_tiles(int spin, int nj) {
  int t = 1;
  ana_shape(spin, nj, [&](auto sh) {
    t = t64::AnaShape64<decltype(sh)::nj, decltype(sh)::spin>::TILES;
    return cudaSuccess;
  });
  return t;
}

// shared-memory attributes of every instance (once per plan; the limits are only raised)
cudaError_t tc64_prepare_device() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void *k, int smem) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  };
  for (int spin = 0; spin < 2; ++spin)
    for (int nj = 1; nj <= 4; nj *= 2) {
      if (tc64_syn_supported(spin, nj))
        syn_shape(spin, nj, [&](auto sh) {
          using T = decltype(sh);
          const int b = t64::Shape<T::nj, T::spin>::SMEM_LAUNCH;
          set((const void *)tc64_syn<T::nj, T::spin>, b);
          set((const void *)tc64_syn_batch<T::nj, T::spin>, b);
          return cudaSuccess;
        });
      if (tc64_ana_supported(spin, nj))
        ana_shape(spin, nj, [&](auto sh) {
          using T = decltype(sh);
          const int b = t64::AnaShape64<T::nj, T::spin>::SMEM_LAUNCH;
          set((const void *)tc64_ana<T::nj, T::spin>, b);
          set((const void *)tc64_ana_batch<T::nj, T::spin>, b);
          return cudaSuccess;
        });
    }
  return e;
}

cudaError_t launch_leg_tc64_items(const sht_plan_s *P, int stage, const void *legargs, const void *items, int n,
                                  cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  LegArgs a;
  memcpy(&a, legargs, sizeof(a));
  if (stage == 0) {
    a.syn_items = static_cast<const int2 *>(items);
    return syn_shape(P->spin, P->njobs_pad, [&](auto sh) {
      using T = decltype(sh);
      tc64_syn<T::nj, T::spin><<<n, t64::kRows, t64::Shape<T::nj, T::spin>::SMEM_LAUNCH, st>>>(a);
      return cudaGetLastError();
    });
  }
  a.ana_items = static_cast<const int4 *>(items);
  return ana_shape(P->spin, P->njobs_pad, [&](auto sh) {
    using T = decltype(sh);
    using S = t64::AnaShape64<T::nj, T::spin>;
    tc64_ana<T::nj, T::spin><<<n, S::TH, S::SMEM_LAUNCH, st>>>(a);
    return cudaGetLastError();
  });
}

cudaError_t launch_leg_tc64_batch(int stage, int spin, int nj, const void *args, const int4 *items, int n,
                                  cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const LegArgs *a = static_cast<const LegArgs *>(args);
  if (stage == 0)
    return syn_shape(spin, nj, [&](auto sh) {
      using T = decltype(sh);
      tc64_syn_batch<T::nj, T::spin><<<n, t64::kRows, t64::Shape<T::nj, T::spin>::SMEM_LAUNCH, st>>>(a, items);
      return cudaGetLastError();
    });
  return ana_shape(spin, nj, [&](auto sh) {
    using T = decltype(sh);
    using S = t64::AnaShape64<T::nj, T::spin>;
    tc64_ana_batch<T::nj, T::spin><<<n, S::TH, S::SMEM_LAUNCH, st>>>(a, items);
    return cudaGetLastError();
  });
}

cudaError_t launch_bounds64(const sht_plan_s *P, cudaStream_t st) {
  if (P->nm == 0 || P->npairs == 0) return cudaSuccess;
  LegArgs a;
  leg_fp64_fill_args(P, 1, &a);
  const dim3 grid((P->npairs + 128 * kBoundPairs - 1) / (128 * kBoundPairs), P->nm);
  if (P->spin) bound_kernel<true><<<grid, 128, 0, st>>>(a, P->d_lexp, P->d_ref);
  else bound_kernel<false><<<grid, 128, 0, st>>>(a, P->d_lexp, P->d_ref);
  return cudaGetLastError();
}

}  // namespace sht
