// legendre_mixed.cu -- Legendre stage (Eqs. syn2, ana1) in the mixed form.
//
// On GB300 the FP64 pipe issues 1/64 of the FP32 rate, so this form moves
// the whole inner loop (the recursion of Sect. 4.1 and the accumulation of
// Fig. 1 / Fig. 2) onto the FP32 pipe in compensated "double-float" pairs
// (value = hi + lo, two FP32 numbers).  Products use the exact FMA split
// (Dekker / Kahan two-product), sums Knuth's two-sum; about 46 significant
// bits survive per operation, enough for ~1e-12 after thousands of steps.
// FP64 remains for the recursion-coefficient tables, the start values and the
// conversion of inputs/outputs (the ring FFTs of mixed plans run the same
// double-float arithmetic, in fft.cu).
//
// Structure, ring pairing, parity split, the separate +s / -s recursions for
// spin and the analysis reduction follow legendre_fp64.cu; only the arithmetic
// type differs.  The enhanced exponent uses steps of 2^104: pairs above 2^52
// are scaled down every 8 steps; values at scale 0 and -1 are accumulated (the
// latter times 2^-104), anything smaller is negligible.  A mixed plan hands the
// items of small m near the poles to the FP64 kernels (sht_plan_s::fp64_m_below).
#include <type_traits>

#include "dual.cuh"
#include "mix_ana.cuh"

namespace sht {

// ---------------------------------------------------------------------------
// alpha_l a_lm (a_lm: FP64, user layout) -> double-float table indexed like the coefficients
// ---------------------------------------------------------------------------
__global__ void alm_to_f2(int lmax, int spin, int nm, int narr, int astride, const int *__restrict__ mval,
                          const int64_t *__restrict__ mstart, const int64_t *__restrict__ coef_off, int64_t ncoef,
                          const double *__restrict__ alpha, DevPtrs alm, float4 *__restrict__ out, int mode) {
  const int mi = blockIdx.x;
  const int deriv = mode & kAlmDeriv, real = (mode & kAlmReal) && mval[mi] > 0;
  const int j = blockIdx.y;
  const int m = mval[mi];
  const double hf = ((mode & kAlmHalf) && m > 0) ? 0.5 : 1.0;
  const int as = spin < 0 ? -spin : spin;
  const int l0 = m > as ? m : as;
  const double *__restrict__ al = alpha + coef_off[mi] - l0;
  if (spin == 0) {
    const double2 *src = reinterpret_cast<const double2 *>(alm.p[j]) + mstart[mi];
    float4 *dst = out + (int64_t)j * ncoef + coef_off[mi] - l0;
    for (int l = l0 + threadIdx.x; l <= lmax; l += blockDim.x) {
      double2 v = src[(int64_t)l * astride];
      if (real) v = real_to_complex(v);
      const double f = hf * al[l];
      const f2 re = f2_of(f * v.x), im = f2_of(f * v.y);
      dst[l] = make_float4(re.h, re.l, im.h, im.l);
    }
    return;
  }
  // spin: P = E + iB and M = E - iB of job j (Im of m = 0 coefficients ignored);
  // deriv (Sect. 4.3): E = sqrt(l(l+1)) a_lm of the spin-0 array j, B = 0
  const double2 *E = reinterpret_cast<const double2 *>(alm.p[deriv ? j : 2 * j]) + mstart[mi];
  const double2 *B = reinterpret_cast<const double2 *>(alm.p[deriv ? j : 2 * j + 1]) + mstart[mi];
  float4 *P = out + (int64_t)(2 * j) * ncoef + coef_off[mi] - l0;
  float4 *M = out + (int64_t)(2 * j + 1) * ncoef + coef_off[mi] - l0;
  for (int l = l0 + threadIdx.x; l <= lmax; l += blockDim.x) {
    double2 e = E[(int64_t)l * astride], b = B[(int64_t)l * astride];
    if (real) {
      e = real_to_complex(e);
      b = real_to_complex(b);
    }
    double f = hf * al[l];
    if (deriv) {
      f *= sqrt((double)l * (double)(l + 1));
      b = make_double2(0.0, 0.0);
    }
    if (m == 0) e.y = b.y = 0.0;
    const f2 pr = f2_of(f * (e.x - b.y)), pi = f2_of(f * (e.y + b.x));
    const f2 mr = f2_of(f * (e.x + b.y)), mi_ = f2_of(f * (e.y - b.x));
    P[l] = make_float4(pr.h, pr.l, pi.h, pi.l);
    M[l] = make_float4(mr.h, mr.l, mi_.h, mi_.l);
  }
}

// ---------------------------------------------------------------------------
// synthesis, spin 0
//
// Loop bodies hold two steps (static even/odd parity) and are not unrolled
// further: the double-float step is ~170 instructions, and longer unrolled
// bodies stalled the issue on instruction fetch.
// ---------------------------------------------------------------------------
template <int NJ, PolarForm PF>
__device__ __forceinline__ void mix_syn_s0_body(const MixArgs &a, const int2 item) {
  const int mi = item.x;
  const int p = item.y + threadIdx.x;
  const bool valid = p < a.npairs;
  const int m = a.mval[mi];
  const int l0 = m, lmax = a.lmax;
  const int64_t co = a.coef_off[mi] - l0;
  const float4 *__restrict__ cf = a.coef32 + co;
  const PairDev pd = a.pairs[valid ? p : 0];
  // zero until the pair joins at its join record's block (no terms, a recursion of zeros)
  f2 lc = {0.f, 0.f}, lp = {0.f, 0.f};
  int scale = 0;
  const float4 *jrec = a.join + ((size_t)mi * a.npairs + (valid ? p : 0)) * 3;
  const int lj = valid ? __float_as_int(__ldg(jrec + 2).z) : lmax + 1;
  const bool polar = PF == kPolarAll || (PF == kPolarCopy && __any_sync(0xffffffffu, near_pole(pd.x, valid)));
  const f3 x = node_of(pd.x, polar);
  f2 acc[2][NJ][2];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[q][j][0] = acc[q][j][1] = f2{0.f, 0.f};

  auto step = [&](const bool pol, int l, int par, bool act) {
    const f2 w = act ? lc : weight(lc, scale);
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float4 v = __ldg(a.alm32 + (int64_t)j * a.ncoef + co + l);
      acc_mul(acc[par][j][0], w, v.x, v.y);
      acc_mul(acc[par][j][1], w, v.z, v.w);
    }
    step_s0(ld_coef32(cf + l), x, pol, lc, lp);
  };
  auto recur = [&](const bool pol, int l) {  // recursion only (every lane's term negligible)
    step_s0(ld_coef32(cf + l), x, pol, lc, lp);
  };
  auto renorm_all = [&]() {
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        renorm(acc[q][j][0]);
        renorm(acc[q][j][1]);
      }
  };

  // the warp starts at its lanes' earliest join block and walks carefully (scale
  // checks, negligible terms skipped) while a lane is below scale 0 or yet to join
  auto walk = [&](const bool pol) __attribute__((always_inline)) {
    int l = __reduce_min_sync(0xffffffffu, lj);
    while (l <= lmax && __any_sync(0xffffffffu, scale < 0 || (lj <= lmax && lj >= l))) {
      if (lj == l) {
        const JoinRec r = ld_join(jrec, polar);
        lc = r.lpc;
        lp = r.lpp;
        scale = r.scp;
      }
#pragma unroll 1
      for (int k = 0; k < 4 && l <= lmax; ++k, l += 2) {
        if (__all_sync(0xffffffffu, negligible(lc, scale))) {
          recur(pol, l);
          if (l + 1 <= lmax) recur(pol, l + 1);
        } else {
          step(pol, l, 0, false);
          if (l + 1 <= lmax) step(pol, l + 1, 1, false);
        }
      }
      if (scale < 0 && fabsf(lc.h) > kScaleUp32) {
        lc = {lc.h * kScaleFactor32, lc.l * kScaleFactor32};
        lp = {lp.h * kScaleFactor32, lp.l * kScaleFactor32};
        ++scale;
      }
      renorm_all();
    }
    int since = 0;
#pragma unroll 1
    for (; l + 1 <= lmax; l += 2) {
      step(pol, l, 0, true);
      step(pol, l + 1, 1, true);
      if (++since == 8) {
        renorm_all();
        since = 0;
      }
    }
    if (l <= lmax) step(pol, l, 0, true);
  };
  if (PF == kPolarAll || (PF == kPolarCopy && polar)) walk(true);
  if (PF == kPolarNone || (PF == kPolarCopy && !polar)) walk(false);
  if (!valid) return;
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const double e0 = f2_val(acc[0][j][0]), e1 = f2_val(acc[0][j][1]);
    const double o0 = f2_val(acc[1][j][0]), o1 = f2_val(acc[1][j][1]);
    double2 fn = make_double2(e0 + o0, e1 + o1), fs = make_double2(e0 - o0, e1 - o1);
    if (m == 0) fn.y = fs.y = 0.0;
    double2 *o = a.phase + (((size_t)j * a.nm + mi) * a.npairs + p) * 2;
    o[0] = fn;
    o[1] = fs;
  }
}
template <int NJ, PolarForm PF = kPolarCopy>
__global__ void __launch_bounds__(kSynTile) mix_syn_s0(MixArgs a) {
  mix_syn_s0_body<NJ, PF>(a, a.syn_items[blockIdx.x]);
}
template <int NJ, PolarForm PF = kPolarCopy>
__global__ void __launch_bounds__(kSynTile) mix_syn_s0_batch(const MixArgs *__restrict__ args,
    const int4 *__restrict__ items) {
  const int4 it = items[blockIdx.x];
  const MixArgs &a = args[it.w];
  mix_syn_s0_body<NJ, PF>(a, make_int2(it.x, it.y));
}

// ---------------------------------------------------------------------------
// synthesis, spin s: separate +s / -s recursions (see legendre_fp64.cu)
// ---------------------------------------------------------------------------
template <int NJ, PolarForm PF>
__device__ __forceinline__ void mix_syn_spin_body(const MixArgs &a, const int2 item) {
  const int mi = item.x;
  const int p = item.y + threadIdx.x;
  const bool valid = p < a.npairs;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax;
  const int64_t co = a.coef_off[mi] - l0;
  const float4 *__restrict__ cf = a.coef32 + co;
  const PairDev pd = a.pairs[valid ? p : 0];
  // zero until the pair joins at its join record's block (no terms, a recursion of zeros)
  f2 lpc = {0.f, 0.f}, lmc = {0.f, 0.f}, lpp = {0.f, 0.f}, lmp = {0.f, 0.f};
  int scp = 0, scm = 0;
  const float4 *jrec = a.join + ((size_t)mi * a.npairs + (valid ? p : 0)) * 3;
  const int lj = valid ? __float_as_int(__ldg(jrec + 2).z) : lmax + 1;
  const bool polar = PF == kPolarAll || (PF == kPolarCopy && __any_sync(0xffffffffu, near_pole(pd.x, valid)));
  const f3 x = node_of(pd.x, polar);
  // N1 = sum P l+, N2 = sum M l-, S3 = sum (-1)^(l-l0) P l-, S4 = sum (-1)^(l-l0) M l+
  f2 r[NJ][4][2];
#pragma unroll
  for (int j = 0; j < NJ; ++j)
#pragma unroll
    for (int k = 0; k < 4; ++k) r[j][k][0] = r[j][k][1] = f2{0.f, 0.f};

  auto step = [&](const bool pol, int l, int par, bool act) {
    const f2 wp = act ? lpc : weight(lpc, scp), wm = act ? lmc : weight(lmc, scm);
    const f2 sp = par ? neg(wp) : wp, sm = par ? neg(wm) : wm;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const float4 P = __ldg(a.alm32 + (int64_t)(2 * j) * a.ncoef + co + l);
      const float4 M = __ldg(a.alm32 + (int64_t)(2 * j + 1) * a.ncoef + co + l);
      acc_mul(r[j][0][0], wp, P.x, P.y);
      acc_mul(r[j][0][1], wp, P.z, P.w);
      acc_mul(r[j][1][0], wm, M.x, M.y);
      acc_mul(r[j][1][1], wm, M.z, M.w);
      acc_mul(r[j][2][0], sm, P.x, P.y);
      acc_mul(r[j][2][1], sm, P.z, P.w);
      acc_mul(r[j][3][0], sp, M.x, M.y);
      acc_mul(r[j][3][1], sp, M.z, M.w);
    }
    step_spin(ld_coef32(cf + l), x, pol, lpc, lpp, lmc, lmp);
  };
  auto recur = [&](const bool pol, int l) {  // recursion only (every lane's terms negligible)
    step_spin(ld_coef32(cf + l), x, pol, lpc, lpp, lmc, lmp);
  };
  auto renorm_all = [&]() {
#pragma unroll
    for (int j = 0; j < NJ; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        renorm(r[j][k][0]);
        renorm(r[j][k][1]);
      }
  };

  // the warp starts at its lanes' earliest join block and walks carefully (scale
  // checks, negligible terms skipped) while a lane is below scale 0 or yet to join
  auto walk = [&](const bool pol) __attribute__((always_inline)) {
    int l = __reduce_min_sync(0xffffffffu, lj);
    while (l <= lmax && __any_sync(0xffffffffu, scp < 0 || scm < 0 || (lj <= lmax && lj >= l))) {
      if (lj == l) {
        const JoinRec r = ld_join(jrec, polar);
        lpc = r.lpc;
        lpp = r.lpp;
        lmc = r.lmc;
        lmp = r.lmp;
        scp = r.scp;
        scm = r.scm;
      }
#pragma unroll 1
      for (int k = 0; k < 4 && l <= lmax; ++k, l += 2) {
        if (__all_sync(0xffffffffu, negligible(lpc, scp) && negligible(lmc, scm))) {
          recur(pol, l);
          if (l + 1 <= lmax) recur(pol, l + 1);
        } else {
          step(pol, l, 0, false);
          if (l + 1 <= lmax) step(pol, l + 1, 1, false);
        }
      }
      if (scp < 0 && fabsf(lpc.h) > kScaleUp32) {
        lpc = {lpc.h * kScaleFactor32, lpc.l * kScaleFactor32};
        lpp = {lpp.h * kScaleFactor32, lpp.l * kScaleFactor32};
        ++scp;
      }
      if (scm < 0 && fabsf(lmc.h) > kScaleUp32) {
        lmc = {lmc.h * kScaleFactor32, lmc.l * kScaleFactor32};
        lmp = {lmp.h * kScaleFactor32, lmp.l * kScaleFactor32};
        ++scm;
      }
      renorm_all();
    }
    int since = 0;
#pragma unroll 1
    for (; l + 1 <= lmax; l += 2) {
      step(pol, l, 0, true);
      step(pol, l + 1, 1, true);
      if (++since == 8) {
        renorm_all();
        since = 0;
      }
    }
    if (l <= lmax) step(pol, l, 0, true);
  };
  if (PF == kPolarAll || (PF == kPolarCopy && polar)) walk(true);
  if (PF == kPolarNone || (PF == kPolarCopy && !polar)) walk(false);
  if (!valid) return;

  const double sig = (as & 1) ? -1.0 : 1.0;
  const double h0 = ((l0 + m) & 1) ? -0.5 : 0.5;
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const double n1r = f2_val(r[j][0][0]), n1i = f2_val(r[j][0][1]);
    const double n2r = f2_val(r[j][1][0]), n2i = f2_val(r[j][1][1]);
    const double s3r = f2_val(r[j][2][0]), s3i = f2_val(r[j][2][1]);
    const double s4r = f2_val(r[j][3][0]), s4i = f2_val(r[j][3][1]);
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
}
template <int NJ, PolarForm PF = kPolarCopy>
__global__ void __launch_bounds__(kSynTile) mix_syn_spin(MixArgs a) {
  mix_syn_spin_body<NJ, PF>(a, a.syn_items[blockIdx.x]);
}
template <int NJ, PolarForm PF = kPolarCopy>
__global__ void __launch_bounds__(kSynTile) mix_syn_spin_batch(const MixArgs *__restrict__ args,
    const int4 *__restrict__ items) {
  const int4 it = items[blockIdx.x];
  const MixArgs &a = args[it.w];
  mix_syn_spin_body<NJ, PF>(a, make_int2(it.x, it.y));
}

// ---------------------------------------------------------------------------
// Spin 0, two ring pairs per thread: the same tiles, chunks and slots with the packed
// FP32 instructions of dual.cuh -- the two pairs' recursions as two lanes, the real and
// imaginary sums of a product as two lanes, and of a warp's 32 columns two at a time in
// the reduction, whose slot table holds high and low words in planes of their own (so
// that two columns' words load as a pair) -- and one CTA barrier per two chunks, after
// which warps 0 and 1 add one chunk each.
// Bound by the FP32 pipe (a packed instruction holds it twice as long) and by warps
// waiting for one another at the barrier (1.7 stalls per issue each, 68% issue at 24 warps
// per SM).  One map, lmax 4095 22.7 -> 21.6 ms (packed lanes 22.6, one barrier per two
// chunks 21.9, the products' multiplies scalar again, without the moves that doubled an
// operand, 21.6); HEALPix 1535 1.89 -> 1.78 ms; lmax 511 147 -> 133 us.  4, 5, 7 or 8 CTAs
// per SM instead of six were slower (24.0, 23.8, 23.0, 22.8 against 22.7 before).
// ---------------------------------------------------------------------------
template <int NJ>
__device__ __forceinline__ void mix_ana_pair_body(const MixArgs &a, const int4 item) {
  constexpr int V = 2 * NJ, LC = 32 / V, TH = kAnaThreads, NP = 2;
  constexpr int ROW = TH + 2;  // 16 rows' pairs of words fall into different banks
  static_assert(LC % 2 == 0 && ROW % 2 == 0, "two degrees at a time; pairs of words");
  __shared__ __align__(8) float sloth[32][ROW], slotl[32][ROW];
  __shared__ f2 quart[2][2][TH / 32][32];  // by parity of the chunk pair, chunk
  __shared__ int tstart[2][TH / 32];     // per tile (parity): the warps' earliest join degree
  const int mi = item.x, ng = item.z & 255;
  const int m = a.mval[mi], l0 = m, lmax = a.lmax, nl = lmax - l0 + 1;
  const float4 *__restrict__ cf = a.coef32 + (a.coef_off[mi] - l0);
  double *const outp = a.part + a.part_off[mi] + (int64_t)(item.z >> 8) * nl * V;
  const int tid = threadIdx.x;

#pragma unroll 1
  for (int gi = 0; gi < ng; ++gi) {
    const int tile = item.y + gi;
    Dual<false, kScalar> rec;
    rec.p = rec.q = d2{both(0.f), both(0.f)};
    int sc[NP] = {0, 0}, lj[NP];
    // G_N + G_S and G_N - G_S of each pair: high and low words, (re, im) as lanes
    float2 gh[NP][NJ][2], gl[NP][NJ][2];
    double xd[NP];
    bool near = false;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
      const int p = tile * (TH * NP) + tid + k * TH;
      const bool valid = p < a.npairs;
      const PairDev pd = a.pairs[valid ? p : 0];
      xd[k] = pd.x;
      lj[k] = valid ? __float_as_int(__ldg(a.join + ((size_t)mi * a.npairs + p) * 3 + 2).z) : lmax + 1;
      near = near || near_pole(pd.x, valid);
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        double2 gn = make_double2(0, 0), gs = make_double2(0, 0);
        if (valid) {
          const double2 *gp = a.phase + (((size_t)j * a.nm + mi) * a.npairs + p) * 2;
          gn = gp[0];
          if (pd.south) gs = gp[1];
        }
        const f2 er = f2_of(gn.x + gs.x), ei = f2_of(gn.y + gs.y);
        const f2 orr = f2_of(gn.x - gs.x), oi = f2_of(gn.y - gs.y);
        gh[k][j][0] = make_float2(er.h, ei.h);
        gl[k][j][0] = make_float2(er.l, ei.l);
        gh[k][j][1] = make_float2(orr.h, oi.h);
        gl[k][j][1] = make_float2(orr.l, oi.l);
      }
    }
    const int jmin = min(lj[0], lj[1]);
    const bool polar = __any_sync(0xffffffffu, near);
#pragma unroll
    for (int k = 0; k < NP; ++k) rec.x[k] = node_of(xd[k], polar);

    // the tile's earliest join block; the first tile zeroes the slot's degrees before it
    {
      const int wmin = __reduce_min_sync(0xffffffffu, jmin);
      if ((tid & 31) == 0) tstart[gi & 1][tid >> 5] = wmin;
    }
    __syncthreads();
    int lstart = tstart[gi & 1][0];
#pragma unroll
    for (int w = 1; w < TH / 32; ++w) lstart = min(lstart, tstart[gi & 1][w]);
    if (gi == 0)
      for (int i = tid; i < (min(lstart, lmax + 1) - l0) * V; i += TH) outp[i] = 0.0;

    float2 wf = both(1.f);  // the lanes' accumulation weights
    // degree l into row q of the chunk (past lmax lmax's coefficients stand in: finite
    // values, never stored); ODD: the sums over G_N - G_S
    auto step = [&](const StepMode mode, int l, int q, const int odd, const bool act) __attribute__((always_inline)) {
      const float4 cc = __ldg(cf + (l <= lmax ? l : lmax));
      float2 h = rec.p.h, lo = rec.p.l;
      if (!act) {
        h = mul2(h, wf);
        lo = mul2(lo, wf);
      }
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        // each pair's exact product (one multiply, three FMAs a part), then their sum
        const float2 A = gh[0][j][odd], a1 = gl[0][j][odd], B = gh[1][j][odd], b1 = gl[1][j][odd];
        const float2 p = make_float2(__fmul_rn(h.x, A.x), __fmul_rn(h.x, A.y));
        const float2 r = make_float2(__fmul_rn(h.y, B.x), __fmul_rn(h.y, B.y));
        float2 e, f;
        e.x = __fmaf_rn(lo.x, A.x, __fmaf_rn(h.x, a1.x, __fmaf_rn(h.x, A.x, -p.x)));
        e.y = __fmaf_rn(lo.x, A.y, __fmaf_rn(h.x, a1.y, __fmaf_rn(h.x, A.y, -p.y)));
        f.x = __fmaf_rn(lo.y, B.x, __fmaf_rn(h.y, b1.x, __fmaf_rn(h.y, B.x, -r.x)));
        f.y = __fmaf_rn(lo.y, B.y, __fmaf_rn(h.y, b1.y, __fmaf_rn(h.y, B.y, -r.y)));
        const d2 t = two_sum(p, r);
        const float2 tl = add2(e, add2(t.l, f));
        sloth[q * V + 2 * j][tid] = t.h.x;
        sloth[q * V + 2 * j + 1][tid] = t.h.y;
        slotl[q * V + 2 * j][tid] = tl.x;
        slotl[q * V + 2 * j + 1][tid] = tl.y;
      }
      rec.step(mode, cc);
    };
    auto skip = [&](const StepMode mode, int l, int q) __attribute__((always_inline)) {  // no terms
#pragma unroll
      for (int v = 0; v < V; ++v) sloth[q * V + v][tid] = slotl[q * V + v][tid] = 0.f;
      rec.step(mode, __ldg(cf + (l <= lmax ? l : lmax)));
    };

    int since = 0;         // steps since the last exponent check
    bool settled = false;  // every lane's values at scale 0: they stay there (warp-uniform)
    int cb = 0;            // parity of the chunk pair: the quart buffer
    for (int lb2 = lstart; lb2 <= lmax; lb2 += 2 * LC) {
      // the slot entry that this lane adds to (warps 0 and 1: one chunk each), from the
      // previous tiles: read early, added at the end
      const int ch = tid >> 5, ll = lb2 + ch * LC + (tid & 31) / V;
      const bool mine = ch < 2 && ll <= lmax;
      double *const o = outp + (int64_t)(lb2 + ch * LC - l0) * V + (tid & 31);
      const double prev = (gi > 0 && mine) ? *o : 0.0;
#pragma unroll 1
      for (int c2 = 0; c2 < 2; ++c2) {
        const int lb = lb2 + c2 * LC;
        bool joins = false;
#pragma unroll
        for (int k = 0; k < NP; ++k)
          if (lj[k] == lb) {
            const int p = tile * (TH * NP) + tid + k * TH;
            const JoinRec r = ld_join(a.join + ((size_t)mi * a.npairs + p) * 3, polar);
            rec.start(k, r.lpc, r.lpp, 1.f);
            sc[k] = r.scp;
            joins = true;
          }
        if (joins) wf = make_float2(scale_weight(sc[0]), scale_weight(sc[1]));
        if (__any_sync(0xffffffffu, joins)) settled = false;
        // a warp none of whose lanes has joined skips this chunk's steps
        const bool wlive = lb <= lmax && __any_sync(0xffffffffu, jmin <= lb);
        auto chunk = [&](const StepMode mode) __attribute__((always_inline)) {
#pragma unroll 1
          for (int q = 0; q < LC; q += 2) {
            const int l = lb + q;
            if (l > lmax) break;
            if (!settled) settled = __all_sync(0xffffffffu, sc[0] == 0 && sc[1] == 0);
            if (settled) {
              step(mode, l, q, 0, true);
              step(mode, l + 1, q + 1, 1, true);
            } else {
              if (__all_sync(0xffffffffu, negligible(lane0(rec.p), sc[0]) && negligible(lane1(rec.p), sc[1]))) {
                skip(mode, l, q);
                skip(mode, l + 1, q + 1);
              } else {
                step(mode, l, q, 0, false);
                step(mode, l + 1, q + 1, 1, false);
              }
              since += 2;
              if (since >= 8) {
                rec.rescale(sc[0], sc[1]);
                wf = make_float2(scale_weight(sc[0]), scale_weight(sc[1]));
                since = 0;
              }
            }
          }
        };
        if (wlive) {
          if (polar) chunk(kPolar);
          else chunk(kCareful);
        }
        // a warp's slot columns are written and read by that warp only: warp-level sync
        __syncwarp();
        // each warp sums its own 32 columns of its lane's row
        const int sl = tid & 31, part = tid >> 5;
        f2 t = {0.f, 0.f};
        if (wlive) {
          const float2 *rh = reinterpret_cast<const float2 *>(&sloth[sl][part * 32]);
          const float2 *rl = reinterpret_cast<const float2 *>(&slotl[sl][part * 32]);
          d2 c = {rh[0], rl[0]};
#pragma unroll
          for (int i = 1; i < 16; ++i) {
            const d2 u = two_sum(c.h, rh[i]);
            c = {u.h, add2(add2(c.l, rl[i]), u.l)};
          }
          t = f2_add_lazy(lane0(c), lane1(c));
        }
        quart[cb][c2][part][sl] = t;
        __syncwarp();
      }
      // one barrier per two chunks: quart is double-buffered, so warps 0 and 1 read these
      // partials while the others fill the other buffer, and they have read them before
      // they reach the next barrier, after which this buffer is written again
      __syncthreads();
      if (ch < 2) {
        f2 t = quart[cb][ch][0][tid & 31];
#pragma unroll
        for (int w = 1; w < TH / 32; ++w) t = f2_add(t, quart[cb][ch][w][tid & 31]);
        if (mine) *o = prev + f2_val(t);
      }
      cb ^= 1;
    }
  }
}

// one-job shapes of up to two pairs a thread are held to 80 registers: six CTAs
// per SM instead of five (their shared slot table allows six); measured at one
// E/B pair, lmax 4095: 84.1 ms against 85.0 (two pairs) and 84.0 against 86.8 (one)
template <int NJ, int PPT, bool SPIN>
constexpr int mix_ana_min_blocks() {
  return (NJ == 1 && PPT <= 2) ? 6 : ((!SPIN && NJ == 1 && PPT == 4) ? 5 : 1);  // spin 0, 4 pairs: 96 registers
}
template <int NJ, int PPT, bool SPIN>
__global__ void __launch_bounds__(kAnaThreads, (mix_ana_min_blocks<NJ, PPT, SPIN>())) mix_ana(MixArgs a) {
  if constexpr (!SPIN && PPT == 2) {
    mix_ana_pair_body<NJ>(a, a.ana_items[blockIdx.x]);
  } else {
    __shared__ MixAnaShared sh;
    mix_ana_body<NJ, PPT, SPIN>(a, a.ana_items[blockIdx.x], sh, 0, (SPIN ? 4 : 2) * NJ, false);
  }
}
template <int NJ, int PPT, bool SPIN>
__global__ void __launch_bounds__(kAnaThreads, (mix_ana_min_blocks<NJ, PPT, SPIN>())) mix_ana_batch(const MixArgs *__restrict__ args,
    const int4 *__restrict__ items) {
  const int4 it = items[blockIdx.x];
  const MixArgs &a = args[it.w];
  if constexpr (!SPIN && PPT == 2) {
    mix_ana_pair_body<NJ>(a, make_int4(it.x, it.y, it.z, 0));
  } else {
    __shared__ MixAnaShared sh;
    mix_ana_body<NJ, PPT, SPIN>(a, make_int4(it.x, it.y, it.z, 0), sh, 0, (SPIN ? 4 : 2) * NJ, false);
  }
}

// ---------------------------------------------------------------------------
static MixArgs make_mix(const sht_plan_s *P, int polar) {
  MixArgs a;
  a.lmax = P->lmax;
  a.spin = P->spin;
  a.npairs = P->npairs;
  a.nm = P->nm;
  a.nj = P->njobs_pad;
  a.mval = P->d_mval;
  a.coef_off = P->d_coef_off;
  a.coef32 = P->d_coef32;
  a.alm32 = P->d_alm32;
  a.ncoef = P->ncoef;
  a.mpre = P->d_mpre;
  a.pairs = P->d_pairs;
  a.phase = P->d_phase;
  a.syn_items = syn_items(P, polar);
  a.ana_items = P->d_ana_items[polar];
  a.part_off = P->d_ana_part_off[polar];
  a.part = P->d_part;
  a.join = P->d_join;
  return a;
}

// ---------------------------------------------------------------------------
// Join records (see JoinRec in mixed_common.cuh), once per plan: each thread runs
// its ring pair's recursion from l0 with the steps and rescale checks of the
// double-float kernels, records the state at every block of 16 degrees up to the
// first degree pair whose values are not negligible, then walks on to lmax + 1 for
// the bound on the values' true size.
// ---------------------------------------------------------------------------
template <bool SPIN>
__global__ void __launch_bounds__(128) join_kernel(MixArgs a, float4 *__restrict__ out, int min_exp) {
  const int mi = blockIdx.y, p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= a.npairs) return;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax;
  const float4 *__restrict__ cf = a.coef32 + (a.coef_off[mi] - l0);
  const PairDev pd = a.pairs[p];
  const f3 x = f3_of(pd.x);
  f2 lpc, lmc = {0.f, 0.f}, lpp = {0.f, 0.f}, lmp = {0.f, 0.f};
  int scp, scm = 0;
  if (SPIN) {
    start_s(m, s, pd, a.mpre[mi], &lpc, &scp);
    start_s(m, -s, pd, a.mpre[mi], &lmc, &scm);
  } else {
    start_s0(m, pd, a.mpre[mi], &lpc, &scp);
  }
  // one recursion step at degree l (its row's coefficients; lmax's past lmax)
  auto step = [&](int l) {
    const Coef32 cc = ld_coef32(cf + (l <= lmax ? l : lmax));
    if (SPIN) step_spin(cc, x, false, lpc, lpp, lmc, lmp);
    else step_s0(cc, x, false, lpc, lpp);
  };
  // the kernels' exponent check, made after every eight degrees from l0
  auto rescale = [&]() {
    if (scp < 0 && fabsf(lpc.h) > kScaleUp32) {
      lpc = {lpc.h * kScaleFactor32, lpc.l * kScaleFactor32};
      lpp = {lpp.h * kScaleFactor32, lpp.l * kScaleFactor32};
      ++scp;
    }
    if (SPIN && scm < 0 && fabsf(lmc.h) > kScaleUp32) {
      lmc = {lmc.h * kScaleFactor32, lmc.l * kScaleFactor32};
      lmp = {lmp.h * kScaleFactor32, lmp.l * kScaleFactor32};
      ++scm;
    }
  };
  JoinRec r = {lpc, lpp, lmc, lmp, scp, scm, l0, 0};
  bool live = false;
  int l = l0;
  for (; l <= lmax; l += 2) {
    const int off = l - l0;
    if (off % kJoinBlock == 0) r = {lpc, lpp, lmc, lmp, scp, scm, l, 0};
    if (!(negligible(lpc, scp) && (!SPIN || negligible(lmc, scm)))) {
      live = true;
      break;
    }
    step(l);
    step(l + 1);
    if ((off + 2) % 8 == 0) rescale();
  }
  // from the first live degree on: the largest true size (the kernels' weights:
  // scale 0 as is, scale -1 times 2^-104, below that dropped), low word included
  float vmax = 0.f;
  if (live) {
    auto size = [](f2 y, int sc) {
      const float v = fabsf(y.h) + fabsf(y.l);
      return sc == 0 ? v : (sc == -1 ? v * kScaleFactor32 : 0.f);
    };
    for (; l <= lmax + 1; ++l) {
      vmax = fmaxf(vmax, size(lpc, scp));
      if (SPIN) vmax = fmaxf(vmax, size(lmc, scm));
      if (l > lmax) break;
      step(l);
      if ((l + 1 - l0) % 8 == 0) rescale();
    }
  } else {
    r.lj = lmax + 1;
  }
  // 2^lexp >= vmax (with a margin of 2^-20 for the rounding of the bound), not
  // below 2^min_exp (the plan-wide bound / 2^16: finer grids would bring the
  // digit products near FP32's range end and add nothing)
  int e = min_exp;
  if (vmax > 0.f) {
    int ev;
    frexpf(vmax * (1.f + 0x1p-20f), &ev);  // vmax' = f 2^ev, f in [0.5, 1)
    e = max(e, ev);
  }
  r.lexp = e;
  float4 *o = out + ((size_t)mi * a.npairs + p) * 3;
  o[0] = make_float4(r.lpc.h, r.lpc.l, r.lpp.h, r.lpp.l);
  o[1] = make_float4(r.lmc.h, r.lmc.l, r.lmp.h, r.lmp.l);
  o[2] = make_float4(__int_as_float(r.scp), __int_as_float(r.scm), __int_as_float(r.lj), __int_as_float(r.lexp));
}

cudaError_t launch_join_records(const sht_plan_s *P, cudaStream_t st) {
  if (P->nm == 0 || P->npairs == 0) return cudaSuccess;
  const MixArgs a = make_mix(P, 1);
  const dim3 grid((P->npairs + 127) / 128, P->nm);
  int ub;
  frexpf(P->tc_lam_bound, &ub);  // tc_lam_bound = 2^(ub - 1)
  const int min_exp = ub - 1 - 16;
  if (P->spin) join_kernel<true><<<grid, 128, 0, st>>>(a, P->d_join, min_exp);
  else join_kernel<false><<<grid, 128, 0, st>>>(a, P->d_join, min_exp);
  return cudaGetLastError();
}

// Where the synthesis of sixteen maps or eight E/B pairs keeps the difference form.  Two
// copies of these loops in one kernel overflow the instruction cache, and the polar warp's
// CTA, the longest, waits for instructions (513 Clenshaw-Curtis rings, lmax 255, sixteen
// maps: 708 us in two copies, 416 with the form in every warp, which also has the
// smaller errors: lmax 1023 6.6e-13 -> 4.7e-13).  A step of it costs 5% more, so plans
// without such rings keep the plain form (256 Gauss-Legendre rings 221 us, 241), and from
// lmax 1200 on, where the other CTAs cover the wait, two copies are as fast or faster
// (eight pairs, lmax 1535: HEALPix 43.8 ms against 46.1, Clenshaw-Curtis 50.0, 49.5).
int mix_polar_form(const sht_plan_s *P, bool polar_rings) {
  if (P->precision != SHT_MIXED || P->njobs_pad < (P->spin ? 8 : 16)) return kPolarCopy;
  return !polar_rings ? kPolarNone : (P->lmax < 1200 ? kPolarAll : kPolarCopy);
}
template <class F>
static void polar_shape(int pf, F &&f) {
  if (pf == kPolarAll) f(std::integral_constant<PolarForm, kPolarAll>{});
  else if (pf == kPolarNone) f(std::integral_constant<PolarForm, kPolarNone>{});
  else f(std::integral_constant<PolarForm, kPolarCopy>{});
}

// Legendre stage over an explicit work list (stage 0: synthesis items int2, 1:
// analysis items int4); no a_lm conversion (launch_alm_prepare_mixed does it)
cudaError_t launch_leg_mixed_items(const sht_plan_s *P, int stage, int polar, const void *items, int n,
                                   cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  MixArgs a = make_mix(P, polar);
  const int nj = P->njobs_pad;
  if (stage == 0) {
    a.syn_items = static_cast<const int2 *>(items);
    if (P->tc_syn) return launch_leg_tc_syn(P, &a, n, st);
    if (P->spin == 0) {
      switch (nj) {
        case 1: mix_syn_s0<1><<<n, kSynTile, 0, st>>>(a); break;
        case 2: mix_syn_s0<2><<<n, kSynTile, 0, st>>>(a); break;
        case 4: mix_syn_s0<4><<<n, kSynTile, 0, st>>>(a); break;
        case 8: mix_syn_s0<8><<<n, kSynTile, 0, st>>>(a); break;
        default:
          polar_shape(P->polar_form, [&](auto f) { mix_syn_s0<16, f.value><<<n, kSynTile, 0, st>>>(a); });
          break;
      }
    } else {
      switch (nj) {
        case 1: mix_syn_spin<1><<<n, kSynTile, 0, st>>>(a); break;
        case 2: mix_syn_spin<2><<<n, kSynTile, 0, st>>>(a); break;
        case 4: mix_syn_spin<4><<<n, kSynTile, 0, st>>>(a); break;
        default:
          polar_shape(P->polar_form, [&](auto f) { mix_syn_spin<8, f.value><<<n, kSynTile, 0, st>>>(a); });
          break;
      }
    }
  } else {
    a.ana_items = static_cast<const int4 *>(items);
    if (P->tc_ana || tc_ana_quad(P)) return launch_leg_tc_ana(P, &a, n, st);
    if (P->spin == 0)
      ana_shape_s0(nj, P->ana_ppt, [&](auto sh) {
        // (more maps: tc_ana_quad)
        if constexpr (decltype(sh)::nj <= 2)
          mix_ana<decltype(sh)::nj, decltype(sh)::ppt, false><<<n, kAnaThreads, 0, st>>>(a);
      });
    else
      ana_shape_spin(nj, P->ana_ppt, [&](auto sh) {
        if constexpr (decltype(sh)::nj <= 2)
          mix_ana<decltype(sh)::nj, decltype(sh)::ppt, true><<<n, kAnaThreads, 0, st>>>(a);
      });
  }
  return cudaGetLastError();
}

cudaError_t launch_leg_syn_mixed(const sht_plan_s *P, const DevPtrs &alm, int polar, cudaStream_t st, int mode) {
  cudaError_t e = launch_alm_prepare_mixed(P, alm, st, mode);
  if (e != cudaSuccess) return e;
  return launch_leg_mixed_items(P, 0, polar, syn_items(P, polar), nsyn_items(P, polar), st);
}

cudaError_t launch_leg_ana_mixed(const sht_plan_s *P, int polar, cudaStream_t st) {
  return launch_leg_mixed_items(P, 1, polar, P->d_ana_items[polar], P->nana_items[polar], st);
}

}  // namespace sht

// ---------------------------------------------------------------------------
// batches (sht_batch_execute)
// ---------------------------------------------------------------------------
namespace sht {

size_t leg_mixed_args_size() { return sizeof(MixArgs); }

void leg_mixed_fill_args(const sht_plan_s *P, int polar, void *out) {
  MixArgs a = make_mix(P, polar);
  memcpy(out, &a, sizeof(a));
}

cudaError_t launch_alm_prepare_mixed(const sht_plan_s *P, const DevPtrs &alm, cudaStream_t st, int mode) {
  if (P->nm == 0) return cudaSuccess;
  dim3 g(P->nm, P->spin ? P->njobs_pad : P->nmaps_pad);
  alm_to_f2<<<g, 256, 0, st>>>(P->lmax, P->spin, P->nm, P->nmaps_pad, P->astride, P->d_mval, P->d_mstart,
                               P->d_coef_off, P->ncoef, P->d_alpha, alm, P->d_alm32, mode);
  return cudaGetLastError();
}

cudaError_t launch_leg_mixed_batch(int stage, int spin, int nj, int ppt, int pf, const void *args, const int4 *items,
                                   int n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const MixArgs *a = static_cast<const MixArgs *>(args);
  if (stage == 0) {
    if (spin == 0) {
      switch (nj) {
        case 1: mix_syn_s0_batch<1><<<n, kSynTile, 0, st>>>(a, items); break;
        case 2: mix_syn_s0_batch<2><<<n, kSynTile, 0, st>>>(a, items); break;
        case 4: mix_syn_s0_batch<4><<<n, kSynTile, 0, st>>>(a, items); break;
        case 8: mix_syn_s0_batch<8><<<n, kSynTile, 0, st>>>(a, items); break;
        default:
          polar_shape(pf, [&](auto f) { mix_syn_s0_batch<16, f.value><<<n, kSynTile, 0, st>>>(a, items); });
          break;
      }
    } else {
      switch (nj) {
        case 1: mix_syn_spin_batch<1><<<n, kSynTile, 0, st>>>(a, items); break;
        case 2: mix_syn_spin_batch<2><<<n, kSynTile, 0, st>>>(a, items); break;
        case 4: mix_syn_spin_batch<4><<<n, kSynTile, 0, st>>>(a, items); break;
        default:
          polar_shape(pf, [&](auto f) { mix_syn_spin_batch<8, f.value><<<n, kSynTile, 0, st>>>(a, items); });
          break;
      }
    }
  } else {
    if (spin == 0)
      ana_shape_s0(nj, ppt, [&](auto sh) {
        // (more maps: tc_ana_quad)
        if constexpr (decltype(sh)::nj <= 2)
          mix_ana_batch<decltype(sh)::nj, decltype(sh)::ppt, false><<<n, kAnaThreads, 0, st>>>(a, items);
      });
    else
      ana_shape_spin(nj, ppt, [&](auto sh) {
        if constexpr (decltype(sh)::nj <= 2)
          mix_ana_batch<decltype(sh)::nj, decltype(sh)::ppt, true><<<n, kAnaThreads, 0, st>>>(a, items);
      });
  }
  return cudaGetLastError();
}

}  // namespace sht
