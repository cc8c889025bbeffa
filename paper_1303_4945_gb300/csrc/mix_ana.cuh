// mix_ana.cuh -- the double-float analysis body, for the kernels of legendre_mixed.cu and for
// the items that the digits of legendre_tc_ana.cu do not hold.
#pragma once
#include <math_constants.h>

#include "mixed_common.cuh"

namespace sht {

// ---------------------------------------------------------------------------
// analysis (tiles and partial sums as in legendre_fp64.cu).
//
// Each thread walks PPT ring pairs.  For every degree l it sums its pairs'
// V contributions in registers and stores them to a shared-memory slot
// table [32 slots = LC degrees x V values][threads]; after LC degrees each warp
// sums its own 32 columns of the table (a warp's columns are written and read by
// that warp only: warp-level synchronisation), and after one CTA barrier warp 0
// adds the four warps' partials (double-buffered by chunk parity) to the item's
// slot of partial sums.  An
// item walks a group of consecutive tiles of one m tile after tile into one
// slot (the host sizes the groups), so the partials shrink by the group size.
// Degrees are walked two at a time so the even/odd parity is static.
//
// The body takes NJ of the plan's jobs, from j0 on; vtot: the plan's partial sums per
// degree.  A value that is not finite makes all degrees of its output NaN where the
// caller asks for it (poison).
// ---------------------------------------------------------------------------
struct MixAnaShared {
  f2 slot[32][kAnaThreads + 1];
  f2 quart[2][kAnaThreads / 32][32];  // by chunk parity
  int tstart[2][kAnaThreads / 32];    // per tile (parity): the warps' earliest join degree
  unsigned bad;                       // outputs that are not finite
};

template <int NJ, int PPT, bool SPIN>
__device__ __forceinline__ void mix_ana_body(const MixArgs &a, const int4 item, MixAnaShared &sh, const int j0,
                                             const int vtot, const bool poison) {
  constexpr int V = (SPIN ? 4 : 2) * NJ, LC = 32 / V;
  constexpr bool OUT = PPT >= 2;  // the polar steps (step_spin)
  static_assert(V * LC == 32 && LC >= 2, "32 slots per chunk, two degrees at a time");
  auto &slot = sh.slot;
  auto &quart = sh.quart;
  auto &tstart = sh.tstart;
  const int mi = item.x, ng = item.z & 255;  // ng tiles from tile item.y on, one slot of partial sums
  const int m = a.mval[mi];
  const int s = a.spin, as = s < 0 ? -s : s;
  const int l0 = m > as ? m : as, lmax = a.lmax, nl = lmax - l0 + 1;
  const float4 *__restrict__ cf = a.coef32 + (a.coef_off[mi] - l0);
  double *const outp = a.part + a.part_off[mi] + (int64_t)(item.z >> 8) * nl * vtot + (SPIN ? 4 : 2) * j0;
  const double sg0 = ((l0 + m) & 1) ? -1.0 : 1.0;
  const int tid = threadIdx.x;
  if (poison && tid == 0) sh.bad = 0u;
  unsigned bad = 0u;

  // the group's tiles one after another; each adds its sums to the slot (the first
  // overwrites it), in a fixed order
#pragma unroll 1
  for (int gi = 0; gi < ng; ++gi) {
    const int tile = item.y + gi;
    f3 x[PPT];
    f2 lpc[PPT], lmc[PPT], lpp[PPT], lmp[PPT];
    int scp[PPT], scm[PPT];
    // the degree at which each pair's terms start (join record; zero state until then)
    int lj[PPT];
    // spin 0: g[k][j][0..1] = G_N + G_S, G_N - G_S (complex);
    // spin:   g[k][j][0..3] = W+_N, W-_N, (-1)^(l0+m) W+_S, (-1)^(l0+m) W-_S (complex)
    f2 g[PPT][NJ][SPIN ? 4 : 2][2];
    int jmin = lmax + 1;
    double xd[PPT];
    bool near[PPT];
  #pragma unroll
    for (int k = 0; k < PPT; ++k) {
      const int p = tile * (kAnaThreads * PPT) + tid + k * kAnaThreads;
      const bool valid = p < a.npairs;
      const PairDev pd = a.pairs[valid ? p : 0];
      xd[k] = pd.x;
      lj[k] = valid ? __float_as_int(__ldg(a.join + ((size_t)mi * a.npairs + p) * 3 + 2).z) : lmax + 1;
      near[k] = near_pole(pd.x, valid);
      jmin = min(jmin, lj[k]);
      lpc[k] = lmc[k] = lpp[k] = lmp[k] = f2{0.f, 0.f};
      scp[k] = scm[k] = 0;
  #pragma unroll
      for (int j = 0; j < NJ; ++j) {
        if (!SPIN) {
          double2 gn = make_double2(0, 0), gs = make_double2(0, 0);
          if (valid) {
            const double2 *gp = a.phase + (((size_t)(j0 + j) * a.nm + mi) * a.npairs + p) * 2;
            gn = gp[0];
            if (pd.south) gs = gp[1];
          }
          g[k][j][0][0] = f2_of(gn.x + gs.x);
          g[k][j][0][1] = f2_of(gn.y + gs.y);
          g[k][j][1][0] = f2_of(gn.x - gs.x);
          g[k][j][1][1] = f2_of(gn.y - gs.y);
          if (poison) bad |= (isfinite(gn.x + gs.x) ? 0u : 1u << (2 * j)) | (isfinite(gn.y + gs.y) ? 0u : 2u << (2 * j));
        } else {
          double2 qn = make_double2(0, 0), qs = make_double2(0, 0), un = make_double2(0, 0), us = make_double2(0, 0);
          if (valid) {
            const double2 *gq = a.phase + (((size_t)(2 * (j0 + j)) * a.nm + mi) * a.npairs + p) * 2;
            const double2 *gu = a.phase + (((size_t)(2 * (j0 + j) + 1) * a.nm + mi) * a.npairs + p) * 2;
            qn = gq[0];
            un = gu[0];
            if (pd.south) {
              qs = gq[1];
              us = gu[1];
            }
          }
          g[k][j][0][0] = f2_of(qn.x - un.y);
          g[k][j][0][1] = f2_of(qn.y + un.x);
          g[k][j][1][0] = f2_of(qn.x + un.y);
          g[k][j][1][1] = f2_of(qn.y - un.x);
          g[k][j][2][0] = f2_of(sg0 * (qs.x - us.y));
          g[k][j][2][1] = f2_of(sg0 * (qs.y + us.x));
          g[k][j][3][0] = f2_of(sg0 * (qs.x + us.y));
          g[k][j][3][1] = f2_of(sg0 * (qs.y - us.x));
          if (poison)  // T1 = W+_N l+ + (+-) W+_S l-, T2 = W-_N l- + (+-) W-_S l+
            bad |= (isfinite(qn.x - un.y + (qs.x - us.y)) ? 0u : 1u << (4 * j)) | (isfinite(qn.y + un.x + (qs.y + us.x)) ? 0u : 2u << (4 * j)) |
                   (isfinite(qn.x + un.y + (qs.x + us.y)) ? 0u : 4u << (4 * j)) | (isfinite(qn.y - un.x + (qs.y - us.x)) ? 0u : 8u << (4 * j));
        }
      }
    }

    // which of the warp's pairs run the difference form: of a tile's pairs the first
    // 128 at most hold the rings that need it, and a CTA waits for its slowest warp
    unsigned polar = 0u;
  #pragma unroll
    for (int k = 0; k < PPT; ++k) {
      if (__any_sync(0xffffffffu, near[k])) polar |= 1u << k;
      x[k] = node_of(xd[k], (polar >> k) & 1u);
    }

    // the tile starts at its pairs' earliest join block; the first tile of the group
    // zeroes the slot's degrees before it (the others leave their sums there)
    {
      const int wmin = __reduce_min_sync(0xffffffffu, jmin);
      if ((tid & 31) == 0) tstart[gi & 1][tid >> 5] = wmin;
    }
    __syncthreads();
    int lstart = tstart[gi & 1][0];
  #pragma unroll
    for (int w = 1; w < kAnaThreads / 32; ++w) lstart = min(lstart, tstart[gi & 1][w]);
    if (gi == 0)
      for (int i = tid; i < (min(lstart, lmax + 1) - l0) * V; i += kAnaThreads) outp[(int64_t)(i / V) * vtot + i % V] = 0.0;

    // one degree: this thread's V contributions (summed over its pairs) into c[];
    // the first term of each output is its exact product (no sum with zero)
    auto step = [&](const bool pol, int l, bool odd, bool act, f2 (&c)[V]) {
      // past lmax (second half of the last pair of degrees) the coefficients of
      // lmax stand in: the values are finite, never stored, and no table entry
      // outside this m is read
      const Coef32 cc = ld_coef32(cf + (l <= lmax ? l : lmax));
  #pragma unroll
      for (int k = 0; k < PPT; ++k) {
        const f2 wp = act ? lpc[k] : weight(lpc[k], scp[k]);
        if (!SPIN) {
  #pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const f2 gr = odd ? g[k][j][1][0] : g[k][j][0][0];
            const f2 gi = odd ? g[k][j][1][1] : g[k][j][0][1];
            if (k == 0) {
              c[2 * j] = mul(wp, gr);
              c[2 * j + 1] = mul(wp, gi);
            } else {
              acc_mul(c[2 * j], wp, gr.h, gr.l);
              acc_mul(c[2 * j + 1], wp, gi.h, gi.l);
            }
          }
          step_s0<OUT>(cc, x[k], OUT ? (polar >> k) & 1u : pol, lpc[k], lpp[k]);
        } else {
          const f2 wm = act ? lmc[k] : weight(lmc[k], scm[k]);
          const f2 sp = odd ? neg(wp) : wp, sm = odd ? neg(wm) : wm;
  #pragma unroll
          for (int j = 0; j < NJ; ++j) {
            // T1 = W+_N l+ + (+-) W+_S l-,  T2 = W-_N l- + (+-) W-_S l+
            if (k == 0) {
              c[4 * j + 0] = mul(wp, g[k][j][0][0]);
              c[4 * j + 1] = mul(wp, g[k][j][0][1]);
              c[4 * j + 2] = mul(wm, g[k][j][1][0]);
              c[4 * j + 3] = mul(wm, g[k][j][1][1]);
            } else {
              acc_mul(c[4 * j + 0], wp, g[k][j][0][0].h, g[k][j][0][0].l);
              acc_mul(c[4 * j + 1], wp, g[k][j][0][1].h, g[k][j][0][1].l);
              acc_mul(c[4 * j + 2], wm, g[k][j][1][0].h, g[k][j][1][0].l);
              acc_mul(c[4 * j + 3], wm, g[k][j][1][1].h, g[k][j][1][1].l);
            }
            acc_mul(c[4 * j + 0], sm, g[k][j][2][0].h, g[k][j][2][0].l);
            acc_mul(c[4 * j + 1], sm, g[k][j][2][1].h, g[k][j][2][1].l);
            acc_mul(c[4 * j + 2], sp, g[k][j][3][0].h, g[k][j][3][0].l);
            acc_mul(c[4 * j + 3], sp, g[k][j][3][1].h, g[k][j][3][1].l);
          }
          step_spin<OUT>(cc, x[k], OUT ? (polar >> k) & 1u : pol, lpc[k], lpp[k], lmc[k], lmp[k]);
        }
      }
    };
    auto rescale_all = [&]() {
  #pragma unroll
      for (int k = 0; k < PPT; ++k) {
        if (scp[k] < 0 && fabsf(lpc[k].h) > kScaleUp32) {
          lpc[k] = {lpc[k].h * kScaleFactor32, lpc[k].l * kScaleFactor32};
          lpp[k] = {lpp[k].h * kScaleFactor32, lpp[k].l * kScaleFactor32};
          ++scp[k];
        }
        if (scm[k] < 0 && fabsf(lmc[k].h) > kScaleUp32) {
          lmc[k] = {lmc[k].h * kScaleFactor32, lmc[k].l * kScaleFactor32};
          lmp[k] = {lmp[k].h * kScaleFactor32, lmp[k].l * kScaleFactor32};
          ++scm[k];
        }
      }
    };
    auto put = [&](int q, const f2 (&c)[V]) {
  #pragma unroll
      for (int v = 0; v < V; ++v) slot[q * V + v][tid] = c[v];
    };

    auto recur = [&](const bool pol, int l) {  // recursion only
      const Coef32 cc = ld_coef32(cf + (l <= lmax ? l : lmax));
  #pragma unroll
      for (int k = 0; k < PPT; ++k) {
        const bool pk = OUT ? (polar >> k) & 1u : pol;
        if (!SPIN) step_s0<OUT>(cc, x[k], pk, lpc[k], lpp[k]);
        else step_spin<OUT>(cc, x[k], pk, lpc[k], lpp[k], lmc[k], lmp[k]);
      }
    };
    auto mode = [&]() {  // 0: all terms at scale 0, 2: all negligible, 1: weighted
      bool ok = true, dead = true;
  #pragma unroll
      for (int k = 0; k < PPT; ++k) {
        ok = ok && scp[k] == 0 && scm[k] == 0;
        dead = dead && negligible(lpc[k], scp[k]) && (!SPIN || negligible(lmc[k], scm[k]));
      }
      return __all_sync(0xffffffffu, ok) ? 0 : (__all_sync(0xffffffffu, dead) ? 2 : 1);
    };
    const f2 zero[V] = {};

    int since = 0;         // steps since the last exponent check
    bool settled = false;  // every lane's values at scale 0: they stay there (warp-uniform)
    int cb = 0;            // chunk parity: the quart buffer
    for (int lb = lstart; lb <= lmax; lb += LC) {
      // pairs joining at this degree take the recursion state where their terms start
      bool joins = false;
  #pragma unroll
      for (int k = 0; k < PPT; ++k)
        if (lj[k] == lb) {
          const int p = tile * (kAnaThreads * PPT) + tid + k * kAnaThreads;
          const JoinRec r = ld_join(a.join + ((size_t)mi * a.npairs + p) * 3, (polar >> k) & 1u);
          lpc[k] = r.lpc;
          lpp[k] = r.lpp;
          lmc[k] = r.lmc;
          lmp[k] = r.lmp;
          scp[k] = r.scp;
          scm[k] = r.scm;
          joins = true;
        }
      if (__any_sync(0xffffffffu, joins)) settled = false;
      // a warp none of whose lanes has joined holds zeros: it skips this chunk's
      // steps and adds zeros to the reduction
      const bool wlive = __any_sync(0xffffffffu, jmin <= lb);
      // this chunk's slot entry from the previous tiles (read early, added at the end)
      const bool mine = tid < 32 && lb + tid / V <= lmax;
      double *const o = outp + (int64_t)(lb - l0 + tid / V) * vtot + tid % V;
      const double prev = (gi > 0 && mine) ? *o : 0.0;
      auto chunk = [&](const bool pol) __attribute__((always_inline)) {
  #pragma unroll 1
        for (int q = 0; q < LC; q += 2) {
          const int l = lb + q;
          if (l > lmax) break;
          const int md = settled ? 0 : mode();
          settled = md == 0;
          if (md == 2) {
            recur(pol, l);
            recur(pol, l + 1);
            put(q, zero);
            put(q + 1, zero);
          } else {
            f2 c0[V], c1[V];
            if (md == 0) {
              step(pol, l, false, true, c0);
              step(pol, l + 1, true, true, c1);
            } else {
              step(pol, l, false, false, c0);
              step(pol, l + 1, true, false, c1);
            }
            put(q, c0);
            put(q + 1, c1);
          }
          since += 2;
          if (!settled && since >= 8) {
            rescale_all();
            since = 0;
          }
        }
      };
      if (wlive) {
        if (OUT) chunk(false);
        else if (polar) chunk(true);
        else chunk(false);
      }
      // a warp's slot columns are written and read by that warp only: warp-level sync
      __syncwarp();
      {  // 32 slots x kAnaThreads values: each warp sums its own 32 columns, then 4 partials per slot
        const int sl = tid & 31, part = tid >> 5;
        f2 t = {0.f, 0.f};
        if (wlive) {
          const f2 *row = &slot[sl][part * 32];
          t = row[0];
  #pragma unroll 8
          for (int i = 1; i < 32; ++i) t = f2_add_lazy(t, row[i]);
        }
        quart[cb][part][sl] = t;
      }
      __syncwarp();
      // one barrier per chunk: quart is double-buffered, so warp 0 reads this chunk's
      // partials while the others fill the other buffer, and it has read them before
      // it reaches the next barrier, after which this buffer is written again
      __syncthreads();
      if (tid < 32) {
        f2 t = quart[cb][0][tid];
  #pragma unroll
        for (int w = 1; w < kAnaThreads / 32; ++w) t = f2_add(t, quart[cb][w][tid]);
        if (mine) *o = prev + f2_val(t);
      }
      cb ^= 1;
    }
  }
  if (poison) {
    if (bad) atomicOr(&sh.bad, bad);
    __syncthreads();
    bad = sh.bad;
    for (int i = tid; bad && i < nl * V; i += kAnaThreads)
      if ((bad >> (i % V)) & 1u) outp[(int64_t)(i / V) * vtot + i % V] = CUDART_NAN;
  }
}

}  // namespace sht
