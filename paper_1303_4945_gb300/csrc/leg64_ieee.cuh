// leg64_ieee.cuh -- the FP64 form's Legendre sums in IEEE double, as bodies for the kernels
// of legendre_fp64.cu and for the columns and items that the fixed-point form of
// legendre_tc64.cu does not hold.  See legendre_fp64.cu for the method.
#pragma once
#include "leg64.cuh"

namespace sht {

__device__ __forceinline__ int warp_any(bool b) { return __any_sync(0xffffffffu, b); }

// ---------------------------------------------------------------------------
// Synthesis, spin 0:  F_{m,y} = sum_l a_lm lambda_lm(theta_y)   (Eq. syn2)
// ---------------------------------------------------------------------------
template <int NJ>
__device__ __forceinline__ void leg_syn_s0_body(const LegArgs &a, const int2 item) {
  const int mi = item.x;
  const int p = item.y + threadIdx.x;
  const bool valid = p < a.npairs;
  const int m = a.mval[mi];
  const int l0 = m, lmax = a.lmax;
  const int64_t co = a.coef_off[mi] - l0;
  const double2 *__restrict__ cf = a.coef + co;
  const double2 *__restrict__ al = a.pm + co;  // array j at al + j ncoef

  const PairDev pd = a.pairs[valid ? p : 0];
  const double x = pd.x;
  double mant;
  int E, scale;
  start_value(m, 0, pd, a.mpre[mi], &mant, &E);
  double lc = valid ? to_scaled(mant, E, &scale) : 0.0;
  if (!valid) scale = 0;
  double lp = 0.0;
  double acc[2][NJ][2];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[q][j][0] = acc[q][j][1] = 0.0;

  int l = l0;
  // growth phase: 8 steps per check, terms accumulate only at scale 0
  // (values at scale < 0 are below 2^-250); blocks in which no lane of the
  // warp has reached scale 0 run the recursion alone
  while (l <= lmax && warp_any(scale < 0)) {
    if (!warp_any(scale == 0)) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (l <= lmax) {
          const double ln = fma(__ldg(&cf[l].x) * x, lc, -lp);
          lp = lc;
          lc = ln;
          ++l;
        }
      }
      if (scale < 0 && fabs(lc) > kScaleUp) {
        lc *= kScaleFactor;
        lp *= kScaleFactor;
        ++scale;
      }
      continue;
    }
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
#pragma unroll
      for (int par = 0; par < 2; ++par) {
        if (l <= lmax) {
          const double w = (scale == 0) ? lc : 0.0;
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const double2 av = __ldg(al + j * a.ncoef + l);
            acc[par][j][0] = fma(av.x, w, acc[par][j][0]);
            acc[par][j][1] = fma(av.y, w, acc[par][j][1]);
          }
          const double ln = fma(__ldg(&cf[l].x) * x, lc, -lp);
          lp = lc;
          lc = ln;
          ++l;
        }
      }
    }
    if (scale < 0 && fabs(lc) > kScaleUp) {
      lc *= kScaleFactor;
      lp *= kScaleFactor;
      ++scale;
    }
  }
  // all lanes of the warp active: plain fused loop (offset l - l0 is even here)
  for (; l + 1 <= lmax; l += 2) {
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      const int ll = l + par;
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const double2 av = __ldg(al + j * a.ncoef + ll);
        acc[par][j][0] = fma(av.x, lc, acc[par][j][0]);
        acc[par][j][1] = fma(av.y, lc, acc[par][j][1]);
      }
      const double ln = fma(__ldg(&cf[ll].x) * x, lc, -lp);
      lp = lc;
      lc = ln;
    }
  }
  if (l <= lmax) {
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const double2 av = __ldg(al + j * a.ncoef + l);
      acc[0][j][0] = fma(av.x, lc, acc[0][j][0]);
      acc[0][j][1] = fma(av.y, lc, acc[0][j][1]);
    }
  }
  if (!valid) return;
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    double2 fn = make_double2(acc[0][j][0] + acc[1][j][0], acc[0][j][1] + acc[1][j][1]);
    double2 fs = make_double2(acc[0][j][0] - acc[1][j][0], acc[0][j][1] - acc[1][j][1]);
    if (m == 0) fn.y = fs.y = 0.0;  // Im a_l0 is ignored: the field is real
    double2 *o = a.phase + (((size_t)j * a.nm + mi) * a.npairs + p) * 2;
    o[0] = fn;
    o[1] = fs;
  }
}
// ---------------------------------------------------------------------------
// Synthesis, spin s.  The +s and -s recursions run separately, each with its
// own exponent (near the poles one is smaller than the other by
// tan^{2s}(theta/2); mixing them in one variable would lose the small one).
// With P = E + iB and M = E - iB (tabulated per (m, l) before the launch):
//   north:  q = -(N1 + sig N2)/2,  u = -(-i N1 + i sig N2)/2,   N1 = sum P l+, N2 = sum M l-
//   south:  q = -(S3 + sig S4)/2,  u = -(-i S3 + i sig S4)/2,   S3 = sum (-1)^(l+m) P l-,
//                                                              S4 = sum (-1)^(l+m) M l+
// with sig = (-1)^s, from sLambda(pi - t) = (-1)^(l+m) (-s)Lambda(t).
// ---------------------------------------------------------------------------
template <int NJ>
__device__ __forceinline__ void leg_syn_spin_body(const LegArgs &a, const int2 item) {
  const int mi = item.x;
  const int p = item.y + threadIdx.x;
  const bool valid = p < a.npairs;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax;
  const int64_t co = a.coef_off[mi] - l0;
  const double2 *__restrict__ cf = a.coef + co;
  const PairDev pd = a.pairs[valid ? p : 0];
  const double x = pd.x;
  double m1, m2;
  int e1, e2, scp, scm;
  start_value(m, s, pd, a.mpre[mi], &m1, &e1);
  start_value(m, -s, pd, a.mpre[mi], &m2, &e2);
  double lpc = valid ? to_scaled(m1, e1, &scp) : 0.0, lpp = 0.0;
  double lmc = valid ? to_scaled(m2, e2, &scm) : 0.0, lmp = 0.0;
  if (!valid) scp = scm = 0;
  double n1[NJ][2], n2[NJ][2], s3[NJ][2], s4[NJ][2];
#pragma unroll
  for (int j = 0; j < NJ; ++j) n1[j][0] = n1[j][1] = n2[j][0] = n2[j][1] = s3[j][0] = s3[j][1] = s4[j][0] = s4[j][1] = 0.0;

  auto step = [&](int l, int par, bool act) {
    const double wp = (act || scp == 0) ? lpc : 0.0;
    const double wm = (act || scm == 0) ? lmc : 0.0;
    const double sp = par ? -wp : wp, sm = par ? -wm : wm;  // (-1)^(l - l0) for the south ring
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const double2 P = __ldg(a.pm + (int64_t)(2 * j) * a.ncoef + co + l);
      const double2 M = __ldg(a.pm + (int64_t)(2 * j + 1) * a.ncoef + co + l);
      n1[j][0] = fma(P.x, wp, n1[j][0]);
      n1[j][1] = fma(P.y, wp, n1[j][1]);
      n2[j][0] = fma(M.x, wm, n2[j][0]);
      n2[j][1] = fma(M.y, wm, n2[j][1]);
      s3[j][0] = fma(P.x, sm, s3[j][0]);
      s3[j][1] = fma(P.y, sm, s3[j][1]);
      s4[j][0] = fma(M.x, sp, s4[j][0]);
      s4[j][1] = fma(M.y, sp, s4[j][1]);
    }
    const double2 c = __ldg(cf + l);
    const double u = fma(c.x, x, c.y), v = fma(c.x, x, -c.y);  // a x +- b, one rounding each
    const double np_ = fma(u, lpc, -lpp);
    const double nm_ = fma(v, lmc, -lmp);
    lpp = lpc;
    lpc = np_;
    lmp = lmc;
    lmc = nm_;
  };

  int l = l0;
  while (l <= lmax && warp_any(scp < 0 || scm < 0)) {
    if (!warp_any(scp == 0 || scm == 0)) {  // every term of the warp below 2^-250
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (l <= lmax) {
          const double2 c = __ldg(cf + l);
          const double np_ = fma(fma(c.x, x, c.y), lpc, -lpp);
          const double nm_ = fma(fma(c.x, x, -c.y), lmc, -lmp);
          lpp = lpc;
          lpc = np_;
          lmp = lmc;
          lmc = nm_;
          ++l;
        }
      }
    } else {
#pragma unroll
      for (int k = 0; k < 8; k += 2) {
#pragma unroll
        for (int par = 0; par < 2; ++par) {
          if (l <= lmax) {
            step(l, par, false);
            ++l;
          }
        }
      }
    }
    if (scp < 0 && fabs(lpc) > kScaleUp) {
      lpc *= kScaleFactor;
      lpp *= kScaleFactor;
      ++scp;
    }
    if (scm < 0 && fabs(lmc) > kScaleUp) {
      lmc *= kScaleFactor;
      lmp *= kScaleFactor;
      ++scm;
    }
  }
  for (; l + 1 <= lmax; l += 2) {
    step(l, 0, true);
    step(l + 1, 1, true);
  }
  if (l <= lmax) step(l, 0, true);
  if (!valid) return;

  const double sig = (as & 1) ? -1.0 : 1.0;
  const double h0 = ((l0 + m) & 1) ? -0.5 : 0.5;  // (-1)^(l0+m) / 2
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    // z1 = N1 + sig N2 (q), z2 = sig N2 - N1 (u = -(i/2) z2)
    const double ar = n1[j][0] + sig * n2[j][0], ai = n1[j][1] + sig * n2[j][1];
    const double br = sig * n2[j][0] - n1[j][0], bi = sig * n2[j][1] - n1[j][1];
    const double cr = s3[j][0] + sig * s4[j][0], ci = s3[j][1] + sig * s4[j][1];
    const double dr = sig * s4[j][0] - s3[j][0], di = sig * s4[j][1] - s3[j][1];
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
// ---------------------------------------------------------------------------
// Analysis (Eq. ana1): a_lm = sum_y G_{m,y} lambda_lm(theta_y), of tile item.y + gi into
// the item's slot (gi > 0: added to it).
// A CTA handles one m and a tile of kAnaThreads * PPT ring pairs; each thread
// walks PPT pairs in lockstep.  Per chunk of LC = 32 / V degrees every thread
// holds 32 partial sums (V values per l); a warp reduce-scatter leaves the
// warp total of value v in lane v, the 4 warps are added through shared
// memory and the tile's sum goes to the partial buffer.  A second kernel
// adds the tiles in a fixed order (deterministic result).
// ---------------------------------------------------------------------------

// 32 values per lane -> lane v holds sum over the warp of value v
__device__ __forceinline__ double warp_reduce_scatter32(double (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const bool up = lane & 16;
    const double send = up ? v[i] : v[i + 16];
    const double keep = up ? v[i + 16] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool up = lane & 8;
    const double send = up ? v[i] : v[i + 8];
    const double keep = up ? v[i + 8] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool up = lane & 4;
    const double send = up ? v[i] : v[i + 4];
    const double keep = up ? v[i + 4] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool up = lane & 2;
    const double send = up ? v[i] : v[i + 2];
    const double keep = up ? v[i + 2] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  }
  {
    const bool up = lane & 1;
    const double send = up ? v[0] : v[1];
    const double keep = up ? v[1] : v[0];
    v[0] = keep + __shfl_xor_sync(0xffffffffu, send, 1);
  }
  return v[0];
}

template <int NJ, int PPT>
__device__ __forceinline__ void leg_ana_s0_body(const LegArgs &a, const int4 item, const int gi,
                                                double (*red)[32]) {
  constexpr int V = 2 * NJ, LC = 32 / V;
  const int mi = item.x, tile = item.y + gi;
  const int m = a.mval[mi];
  const int l0 = m, lmax = a.lmax, nl = lmax - l0 + 1;
  const double2 *__restrict__ cf = a.coef + a.coef_off[mi] - l0;
  double *outp = a.part + a.part_off[mi] + (int64_t)(item.z >> 8) * nl * V;  // this item's slot

  double x[PPT], lc[PPT], lp[PPT];
  int scale[PPT];
  double ge[PPT][NJ][2], go[PPT][NJ][2];  // G_N + G_S, G_N - G_S
#pragma unroll
  for (int k = 0; k < PPT; ++k) {
    const int p = tile * (kAnaThreads * PPT) + threadIdx.x + k * kAnaThreads;
    const bool valid = p < a.npairs;
    const PairDev pd = a.pairs[valid ? p : 0];
    x[k] = pd.x;
    double mant;
    int E;
    start_value(m, 0, pd, a.mpre[mi], &mant, &E);
    lc[k] = valid ? to_scaled(mant, E, &scale[k]) : 0.0;
    if (!valid) scale[k] = 0;
    lp[k] = 0.0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      double2 gn = make_double2(0, 0), gs = make_double2(0, 0);
      if (valid) {
        const double2 *g = a.phase + (((size_t)j * a.nm + mi) * a.npairs + p) * 2;
        gn = g[0];
        if (pd.south) gs = g[1];
      }
      ge[k][j][0] = gn.x + gs.x;
      ge[k][j][1] = gn.y + gs.y;
      go[k][j][0] = gn.x - gs.x;
      go[k][j][1] = gn.y - gs.y;
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int lb = l0; lb <= lmax; lb += LC) {
    bool mine = false;
#pragma unroll
    for (int k = 0; k < PPT; ++k) mine = mine || scale[k] == 0;
    if (!__syncthreads_or(mine)) {  // no term of this tile above 2^-250 yet: recursion only
#pragma unroll
      for (int q = 0; q < LC; ++q) {
        const int l = lb + q;
        if (l <= lmax) {
          const double ca = __ldg(&cf[l].x);
#pragma unroll
          for (int k = 0; k < PPT; ++k) {
            const double ln = fma(ca * x[k], lc[k], -lp[k]);
            lp[k] = lc[k];
            lc[k] = ln;
          }
        }
      }
#pragma unroll
      for (int k = 0; k < PPT; ++k) {
        if (scale[k] < 0 && fabs(lc[k]) > kScaleUp) {
          lc[k] *= kScaleFactor;
          lp[k] *= kScaleFactor;
          ++scale[k];
        }
      }
      if (gi == 0 && warp == 0 && lb + lane / V <= lmax) outp[(int64_t)(lb - l0) * V + lane] = 0.0;
      continue;
    }
    double v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = 0.0;
#pragma unroll
    for (int q = 0; q < LC; ++q) {
      const int l = lb + q;
      if (l <= lmax) {
        const double ca = __ldg(&cf[l].x);
        const bool even = ((l - l0) & 1) == 0;
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
          const double w = (scale[k] == 0) ? lc[k] : 0.0;
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const double gr = even ? ge[k][j][0] : go[k][j][0];
            const double gi = even ? ge[k][j][1] : go[k][j][1];
            v[q * V + 2 * j] = fma(w, gr, v[q * V + 2 * j]);
            v[q * V + 2 * j + 1] = fma(w, gi, v[q * V + 2 * j + 1]);
          }
          const double ln = fma(ca * x[k], lc[k], -lp[k]);
          lp[k] = lc[k];
          lc[k] = ln;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
      if (scale[k] < 0 && fabs(lc[k]) > kScaleUp) {
        lc[k] *= kScaleFactor;
        lp[k] *= kScaleFactor;
        ++scale[k];
      }
    }
    const double wsum = warp_reduce_scatter32(v);
    red[warp][lane] = wsum;
    __syncthreads();
    if (warp == 0) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < kAnaThreads / 32; ++w) t += red[w][lane];
      const int q = lane / V;
      double *const o = outp + (int64_t)(lb - l0) * V + lane;
      if (lb + q <= lmax) *o = gi == 0 ? t : *o + t;
    }
    __syncthreads();
  }
}
// Spin analysis with separate +s / -s recursions.  Per ring W+ = GQ + i GU,
// W- = GQ - i GU; per degree l the pair contributes
//   T1 = W+_N l+ + (-1)^(l+m) W+_S l-,   T2 = W-_N l- + (-1)^(l+m) W-_S l+,
// and the reduction kernel forms E = -(T1 + sig T2)/2, B = -(i/2)(sig T2 - T1).
template <int NJ, int PPT>
__device__ __forceinline__ void leg_ana_spin_body(const LegArgs &a, const int4 item, const int gi,
                                                  double (*red)[32]) {
  constexpr int V = 4 * NJ, LC = 32 / V;
  const int mi = item.x, tile = item.y + gi;
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax, nl = lmax - l0 + 1;
  const double2 *__restrict__ cf = a.coef + a.coef_off[mi] - l0;
  double *outp = a.part + a.part_off[mi] + (int64_t)(item.z >> 8) * nl * V;  // this item's slot
  const double sg0 = ((l0 + m) & 1) ? -1.0 : 1.0;

  double x[PPT], lpc[PPT], lmc[PPT], lpp[PPT], lmp[PPT];
  int scp[PPT], scm[PPT];
  double wpn[PPT][NJ][2], wmn[PPT][NJ][2], wps[PPT][NJ][2], wms[PPT][NJ][2];
#pragma unroll
  for (int k = 0; k < PPT; ++k) {
    const int p = tile * (kAnaThreads * PPT) + threadIdx.x + k * kAnaThreads;
    const bool valid = p < a.npairs;
    const PairDev pd = a.pairs[valid ? p : 0];
    x[k] = pd.x;
    double m1, m2;
    int e1, e2;
    start_value(m, s, pd, a.mpre[mi], &m1, &e1);
    start_value(m, -s, pd, a.mpre[mi], &m2, &e2);
    lpc[k] = valid ? to_scaled(m1, e1, &scp[k]) : 0.0;
    lmc[k] = valid ? to_scaled(m2, e2, &scm[k]) : 0.0;
    if (!valid) scp[k] = scm[k] = 0;
    lpp[k] = lmp[k] = 0.0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      double2 qn = make_double2(0, 0), qs = make_double2(0, 0), un = make_double2(0, 0), us = make_double2(0, 0);
      if (valid) {
        const double2 *gq = a.phase + (((size_t)(2 * j) * a.nm + mi) * a.npairs + p) * 2;
        const double2 *gu = a.phase + (((size_t)(2 * j + 1) * a.nm + mi) * a.npairs + p) * 2;
        qn = gq[0];
        un = gu[0];
        if (pd.south) {
          qs = gq[1];
          us = gu[1];
        }
      }
      // W+ = GQ + i GU, W- = GQ - i GU; the south ones carry (-1)^(l0+m)
      wpn[k][j][0] = qn.x - un.y;
      wpn[k][j][1] = qn.y + un.x;
      wmn[k][j][0] = qn.x + un.y;
      wmn[k][j][1] = qn.y - un.x;
      wps[k][j][0] = sg0 * (qs.x - us.y);
      wps[k][j][1] = sg0 * (qs.y + us.x);
      wms[k][j][0] = sg0 * (qs.x + us.y);
      wms[k][j][1] = sg0 * (qs.y - us.x);
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int lb = l0; lb <= lmax; lb += LC) {
    bool mine = false;
#pragma unroll
    for (int k = 0; k < PPT; ++k) mine = mine || scp[k] == 0 || scm[k] == 0;
    if (!__syncthreads_or(mine)) {  // no term of this tile above 2^-250 yet: recursion only
#pragma unroll
      for (int q = 0; q < LC; ++q) {
        const int l = lb + q;
        if (l <= lmax) {
          const double2 c = __ldg(cf + l);
#pragma unroll
          for (int k = 0; k < PPT; ++k) {
            const double np_ = fma(fma(c.x, x[k], c.y), lpc[k], -lpp[k]);
            const double nm_ = fma(fma(c.x, x[k], -c.y), lmc[k], -lmp[k]);
            lpp[k] = lpc[k];
            lpc[k] = np_;
            lmp[k] = lmc[k];
            lmc[k] = nm_;
          }
        }
      }
#pragma unroll
      for (int k = 0; k < PPT; ++k) {
        if (scp[k] < 0 && fabs(lpc[k]) > kScaleUp) {
          lpc[k] *= kScaleFactor;
          lpp[k] *= kScaleFactor;
          ++scp[k];
        }
        if (scm[k] < 0 && fabs(lmc[k]) > kScaleUp) {
          lmc[k] *= kScaleFactor;
          lmp[k] *= kScaleFactor;
          ++scm[k];
        }
      }
      if (gi == 0 && warp == 0 && lb + lane / V <= lmax) outp[(int64_t)(lb - l0) * V + lane] = 0.0;
      continue;
    }
    double v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = 0.0;
#pragma unroll
    for (int q = 0; q < LC; ++q) {
      const int l = lb + q;
      if (l <= lmax) {
        const double2 c = __ldg(cf + l);
        const bool even = ((l - l0) & 1) == 0;
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
          const double wp = (scp[k] == 0) ? lpc[k] : 0.0;
          const double wm = (scm[k] == 0) ? lmc[k] : 0.0;
          const double sp = even ? wp : -wp, sm = even ? wm : -wm;
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const int o = q * V + 4 * j;
            v[o + 0] = fma(wp, wpn[k][j][0], fma(sm, wps[k][j][0], v[o + 0]));
            v[o + 1] = fma(wp, wpn[k][j][1], fma(sm, wps[k][j][1], v[o + 1]));
            v[o + 2] = fma(wm, wmn[k][j][0], fma(sp, wms[k][j][0], v[o + 2]));
            v[o + 3] = fma(wm, wmn[k][j][1], fma(sp, wms[k][j][1], v[o + 3]));
          }
          const double u = fma(c.x, x[k], c.y), w = fma(c.x, x[k], -c.y);  // a x +- b, one rounding each
          const double np_ = fma(u, lpc[k], -lpp[k]);
          const double nm_ = fma(w, lmc[k], -lmp[k]);
          lpp[k] = lpc[k];
          lpc[k] = np_;
          lmp[k] = lmc[k];
          lmc[k] = nm_;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
      if (scp[k] < 0 && fabs(lpc[k]) > kScaleUp) {
        lpc[k] *= kScaleFactor;
        lpp[k] *= kScaleFactor;
        ++scp[k];
      }
      if (scm[k] < 0 && fabs(lmc[k]) > kScaleUp) {
        lmc[k] *= kScaleFactor;
        lmp[k] *= kScaleFactor;
        ++scm[k];
      }
    }
    const double wsum = warp_reduce_scatter32(v);
    red[warp][lane] = wsum;
    __syncthreads();
    if (warp == 0) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < kAnaThreads / 32; ++w) t += red[w][lane];
      const int q = lane / V;
      double *const o = outp + (int64_t)(lb - l0) * V + lane;
      if (lb + q <= lmax) *o = gi == 0 ? t : *o + t;
    }
    __syncthreads();
  }
}
}  // namespace sht
