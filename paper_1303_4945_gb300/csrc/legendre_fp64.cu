// legendre_fp64.cu -- Legendre stage (Eqs. syn2 and ana1) in IEEE double.
//
// One thread owns one north/south ring pair and walks l upwards from
// l0 = max(m, |s|), generating sLambda_lm on the fly by the three-term recursion
// of Sect. 4.1 and applying each value as soon as it exists (the fused loop of
// Sect. 3.2, Figs. 1-2).  The southern ring of a pair comes for free from
//   sLambda_lm(pi - t) = (-1)^(l+m) (-s)Lambda_lm(t):
// even and odd (l+m) terms are kept apart and combined at the end.
//
// Spin s != 0 runs the +s and -s recursions side by side, each with its own
// exponent, and contracts them with P = E + iB and M = E - iB:
//   Q + iU = sum_m e^{im phi} [ -(1/2) sum_l (P (s)Lambda + (-1)^s M (-s)Lambda) ] + c.c. terms,
// see leg_syn_spin; the analysis uses W+- = G_Q +- i G_U the same way.
// Blocks of the growth phase in which no lane has reached scale 0 run the
// recursion alone.
//
// The recursion runs on p_l = Lambda_l / alpha_l (tables.cu), whose three-term form
// has a unit coefficient: 2 FP64 instructions a step (4 at spin s) where the form with
// three coefficients takes 3 (6).  The a_lm tables hold alpha_l a_lm, and the
// reduction of an analysis multiplies by alpha_l.  The FP64 pipe issues one warp
// instruction in 16 cycles per SM, so these kernels are bound by that count.
//
// Enhanced exponent range (Sect. 4.1): the recursion pair is held as
// y * 2^(600 scale); while scale < 0 the terms are below ~2^-300 and are not
// accumulated; every 8 steps values above 2^300 are scaled down by 2^-600.
#include "leg64_ieee.cuh"

namespace sht {

template <int NJ>
__global__ void __launch_bounds__(kSynTile) leg_syn_s0(LegArgs a) {
  leg_syn_s0_body<NJ>(a, a.syn_items[blockIdx.x]);
}
template <int NJ>
__global__ void __launch_bounds__(kSynTile) leg_syn_s0_batch(const LegArgs *__restrict__ args,
    const int4 *__restrict__ items) {
  const int4 it = items[blockIdx.x];
  const LegArgs &a = args[it.w];
  leg_syn_s0_body<NJ>(a, make_int2(it.x, it.y));
}

template <int NJ>
__global__ void __launch_bounds__(kSynTile) leg_syn_spin(LegArgs a) {
  leg_syn_spin_body<NJ>(a, a.syn_items[blockIdx.x]);
}
template <int NJ>
__global__ void __launch_bounds__(kSynTile) leg_syn_spin_batch(const LegArgs *__restrict__ args,
    const int4 *__restrict__ items) {
  const int4 it = items[blockIdx.x];
  const LegArgs &a = args[it.w];
  leg_syn_spin_body<NJ>(a, make_int2(it.x, it.y));
}
template <int NJ, int PPT>
__global__ void __launch_bounds__(kAnaThreads) leg_ana_s0(LegArgs a) {
  __shared__ double red[kAnaThreads / 32][32];
  leg_ana_s0_body<NJ, PPT>(a, a.ana_items[blockIdx.x], 0, red);
}
template <int NJ, int PPT>
__global__ void __launch_bounds__(kAnaThreads) leg_ana_s0_batch(const LegArgs *__restrict__ args,
    const int4 *__restrict__ items) {
  const int4 it = items[blockIdx.x];
  const LegArgs &a = args[it.w];
  __shared__ double red[kAnaThreads / 32][32];
  leg_ana_s0_body<NJ, PPT>(a, make_int4(it.x, it.y, it.z, 0), 0, red);
}

template <int NJ, int PPT>
__global__ void __launch_bounds__(kAnaThreads) leg_ana_spin(LegArgs a) {
  __shared__ double red[kAnaThreads / 32][32];
  leg_ana_spin_body<NJ, PPT>(a, a.ana_items[blockIdx.x], 0, red);
}
template <int NJ, int PPT>
__global__ void __launch_bounds__(kAnaThreads) leg_ana_spin_batch(const LegArgs *__restrict__ args,
    const int4 *__restrict__ items) {
  const int4 it = items[blockIdx.x];
  const LegArgs &a = args[it.w];
  __shared__ double red[kAnaThreads / 32][32];
  leg_ana_spin_body<NJ, PPT>(a, make_int4(it.x, it.y, it.z, 0), 0, red);
}

// Adds the tiles of every (m, l) in tile order, multiplies by alpha_l (the kernels
// sum G_m p_l = G_m Lambda_lm / alpha_l) and writes a_lm.
// spin 0: V = 2 njobs values (re, im per job).
// spin s: V = 4 njobs values (T1, T2 per job): E = -(T1 + sig T2)/2, B = -(i/2)(sig T2 - T1).
__global__ void ana_reduce(int lmax, int spin, int nm, int njobs_pad, int ncomp, int astride, int add,
                           int real, int grad,
                           const int *__restrict__ mval, const int64_t *__restrict__ mstart,
                           const int64_t *__restrict__ coef_off, const double *__restrict__ alpha,
                           const int64_t *__restrict__ part_off, const int *__restrict__ nslot,
                           const double *__restrict__ part, DevPtrs alm) {
  const int mi = blockIdx.y;
  const int m = mval[mi];
  const int as = spin < 0 ? -spin : spin;
  const int l0 = m > as ? m : as;
  const int nl = lmax - l0 + 1;
  const int V = (spin ? 4 : 2) * njobs_pad;
  const int l = l0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (l > lmax) return;
  const int nt = nslot[mi];
  const double al = alpha[coef_off[mi] + (l - l0)];
  const double *pb = part + part_off[mi] + (int64_t)(l - l0) * V;
  const int64_t idx = mstart[mi] + (int64_t)l * astride;
  const int vper = spin ? 4 : 2;
  for (int j = 0; j < ncomp; ++j) {
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int tt = 0; tt < nt; ++tt)
      for (int k = 0; k < vper; ++k) t[k] += pb[(int64_t)tt * nl * V + vper * j + k];
    for (int k = 0; k < vper; ++k) t[k] *= al;
    double2 out[2];
    int nout;
    if (spin == 0) {
      out[0] = make_double2(t[0], m == 0 ? 0.0 : t[1]);
      nout = 1;
    } else {
      const double sig = (as & 1) ? -1.0 : 1.0;
      out[0] = make_double2(-0.5 * (t[0] + sig * t[2]), -0.5 * (t[1] + sig * t[3]));
      const double zr = sig * t[2] - t[0], zi = sig * t[3] - t[1];
      out[1] = make_double2(0.5 * zi, -0.5 * zr);
      if (m == 0) out[0].y = out[1].y = 0.0;
      nout = 2;
    }
    for (int c = 0; c < nout; ++c) {
      double2 *o = reinterpret_cast<double2 *>(alm.p[nout * j + c]) + idx;
      double2 r = (real && m > 0) ? complex_to_real(out[c]) : out[c];
      if (grad && m > 0) r = make_double2(2.0 * r.x, 2.0 * r.y);  // the stored a_lm also stands for a_{l,-m}
      if (add) {
        const double2 old = *o;
        r.x += old.x;
        r.y += old.y;
      }
      *o = r;
    }
  }
  // spin: entries l < |s| (outside the recursion) are zero for l >= m
  if (spin && l == l0 && !add) {
    for (int ll = m; ll < l0; ++ll) {
      const int64_t i2 = mstart[mi] + (int64_t)ll * astride;
      for (int j = 0; j < 2 * ncomp; ++j) reinterpret_cast<double2 *>(alm.p[j])[i2] = make_double2(0.0, 0.0);
    }
  }
}

// alpha_l times the a_lm of every (m, l), indexed like the coefficient table: array j
// at spin 0; P = E + iB and M = E - iB (arrays 2j, 2j + 1) at spin s.
//
// wide (plans whose synthesis contracts in fixed point): byte 4 mi + j says whether the
// column's values range too far for it.  On a ring where only the degrees from some l on
// have Lambda near its bound (below, it falls away exponentially) the result comes from
// those alone, so of every four neighbouring degrees, and of the last two, one has to lie
// within 2^kWideRange of the largest of the column.  Spectra like 1/(l + 1) do (lmax 1023: a
// factor of some 2^10 in a column, and 2^2 to 2^3 of chance); a column of zeros does; a band
// limit below lmax or an infinity does not.
constexpr int kPmThreads = 256;
__global__ void __launch_bounds__(kPmThreads)
    alm_to_pm(int lmax, int spin, int nm, int astride, const int *__restrict__ mval, const int64_t *__restrict__ mstart,
              const int64_t *__restrict__ coef_off, int64_t ncoef, const double *__restrict__ alpha, DevPtrs alm,
              double2 *__restrict__ out, int mode, unsigned char *__restrict__ wide) {
  __shared__ int smax[4], smin[4], stail[4];
  const int mi = blockIdx.x, j = blockIdx.y, tid = threadIdx.x;
  const int64_t co = coef_off[mi];
  if (co >= ncoef) return;  // beyond the table (a mixed plan's m above its FP64 columns)
  const int deriv = mode & kAlmDeriv, real = (mode & kAlmReal) && mval[mi] > 0;
  const int m = mval[mi];
  const double hf = ((mode & kAlmHalf) && m > 0) ? 0.5 : 1.0;
  const int as = spin < 0 ? -spin : spin;
  const int l0 = m > as ? m : as;
  // deriv (Sect. 4.3): E = sqrt(l(l+1)) a_lm of the spin-0 array j, B = 0
  const int per = spin && !deriv ? 2 : 1;
  const double2 *E = reinterpret_cast<const double2 *>(alm.p[per * j]) + mstart[mi];
  const double2 *B = reinterpret_cast<const double2 *>(alm.p[per * j + per - 1]) + mstart[mi];
  double2 *P = out + (int64_t)((spin ? 2 : 1) * j) * ncoef + co - l0;
  double2 *M = P + ncoef;
  if (tid < 4) {
    smax[tid] = stail[tid] = 0;
    smin[tid] = kFieldMax;
  }
  __syncthreads();
  int vmax[4] = {0, 0, 0, 0}, vmin[4] = {kFieldMax, kFieldMax, kFieldMax, kFieldMax};
  for (int l = l0 + tid; l - (tid & 31) <= lmax; l += kPmThreads) {
    const bool in = l <= lmax;
    double2 p = make_double2(0.0, 0.0), q = p;
    if (in) {
      double2 e = E[(int64_t)l * astride], b = make_double2(0.0, 0.0);
      if (spin && !deriv) b = B[(int64_t)l * astride];
      if (real) {
        e = real_to_complex(e);
        b = real_to_complex(b);
      }
      double f = hf * alpha[co + l - l0];
      if (deriv) f *= sqrt((double)l * (double)(l + 1));
      if (!spin) {
        p = make_double2(f * e.x, f * e.y);
      } else {
        if (m == 0) e.y = b.y = 0.0;  // Im of m = 0 coefficients is ignored
        p = make_double2(f * (e.x - b.y), f * (e.y + b.x));
        q = make_double2(f * (e.x + b.y), f * (e.y - b.x));
        M[l] = q;
      }
      P[l] = p;
    }
    if (!wide) continue;
    const int z[4] = {size_field(p.x), size_field(p.y), size_field(q.x), size_field(q.y)};
    const int first = l - (tid & 3);  // of the lane's four degrees
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      int four = max(z[v], __shfl_xor_sync(0xffffffffu, z[v], 1));
      four = max(four, __shfl_xor_sync(0xffffffffu, four, 2));
      vmax[v] = max(vmax[v], z[v]);
      if (first + 3 <= lmax) vmin[v] = min(vmin[v], four);
      if (in && l >= lmax - 1) atomicMax(&stail[v], z[v]);
    }
  }
  if (!wide) return;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const int hi = __reduce_max_sync(0xffffffffu, vmax[v]), lo = __reduce_min_sync(0xffffffffu, vmin[v]);
    if ((tid & 31) == 0) {
      atomicMax(&smax[v], hi);
      atomicMin(&smin[v], lo);
    }
  }
  __syncthreads();
  if (tid == 0) {
    bool w = false;
    for (int v = 0; v < 4; ++v)
      w = w || (smax[v] > 0 && (smax[v] < kFieldMin || smax[v] >= kFieldMax ||
                                min(smin[v], stail[v]) < smax[v] - kWideRange));
    wide[4 * mi + j] = w ? 1 : 0;
  }
}
// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static LegArgs make_args(const sht_plan_s *P, int polar, bool lo = false) {
  LegArgs a;
  a.lmax = P->lmax;
  a.spin = P->spin;
  a.npairs = P->npairs;
  a.nm = P->nm;
  a.mval = P->d_mval;
  a.coef_off = P->d_coef_off;
  a.coef = P->d_coef;
  a.pm = P->d_pm64;
  a.ncoef = P->ncoef64;  // the P/M table's stride between arrays
  a.mpre = P->d_mpre;
  a.pairs = P->d_pairs;
  a.phase = P->d_phase;
  a.syn_items = lo ? P->d_syn_lo[polar] : P->d_syn_items[polar];
  a.ana_items = lo ? P->d_ana_lo[polar] : P->d_ana_items[polar];
  a.part_off = P->d_ana_part_off[polar];
  a.part = P->d_part;
  a.lexp = P->d_lexp;
  a.ref = P->d_ref;
  a.wide_syn = P->d_wide_syn;
  a.err = P->d_err;
  return a;
}

// Legendre stage over an explicit work list (stage 0: synthesis items int2, 1:
// analysis items int4); no a_lm conversion (launch_alm_prepare_fp64 does it)
cudaError_t launch_leg_fp64_items(const sht_plan_s *P, int stage, int polar, const void *items, int n,
                                  cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  LegArgs a = make_args(P, polar);
  if (stage == 0 ? P->tc64_syn : P->tc64_ana) return launch_leg_tc64_items(P, stage, &a, items, n, st);
  const int nj = P->njobs_pad;
  if (stage == 0) {
    a.syn_items = static_cast<const int2 *>(items);
    if (P->spin == 0) {
      switch (nj) {
        case 1: leg_syn_s0<1><<<n, kSynTile, 0, st>>>(a); break;
        case 2: leg_syn_s0<2><<<n, kSynTile, 0, st>>>(a); break;
        case 4: leg_syn_s0<4><<<n, kSynTile, 0, st>>>(a); break;
        case 8: leg_syn_s0<8><<<n, kSynTile, 0, st>>>(a); break;
        default: leg_syn_s0<16><<<n, kSynTile, 0, st>>>(a); break;
      }
    } else {
      switch (nj) {
        case 1: leg_syn_spin<1><<<n, kSynTile, 0, st>>>(a); break;
        case 2: leg_syn_spin<2><<<n, kSynTile, 0, st>>>(a); break;
        case 4: leg_syn_spin<4><<<n, kSynTile, 0, st>>>(a); break;
        default: leg_syn_spin<8><<<n, kSynTile, 0, st>>>(a); break;
      }
    }
  } else {
    a.ana_items = static_cast<const int4 *>(items);
    if (P->spin == 0)
      ana_shape_s0(nj, P->ana_ppt, [&](auto sh) {
        leg_ana_s0<decltype(sh)::nj, decltype(sh)::ppt><<<n, kAnaThreads, 0, st>>>(a);
      });
    else
      ana_shape_spin(nj, P->ana_ppt, [&](auto sh) {
        leg_ana_spin<decltype(sh)::nj, decltype(sh)::ppt><<<n, kAnaThreads, 0, st>>>(a);
      });
  }
  return cudaGetLastError();
}

cudaError_t launch_leg_syn_fp64(const sht_plan_s *P, const DevPtrs &alm, int polar, cudaStream_t st, bool lo,
                                int mode) {
  const int n = lo ? P->nsyn_lo[polar] : P->nsyn_items[polar];
  if (n == 0) return cudaSuccess;
  cudaError_t e = launch_alm_prepare_fp64(P, alm, st, mode);
  if (e != cudaSuccess) return e;
  return launch_leg_fp64_items(P, 0, polar, lo ? (const void *)P->d_syn_lo[polar] : P->d_syn_items[polar], n, st);
}

cudaError_t launch_leg_ana_fp64(const sht_plan_s *P, int polar, cudaStream_t st, bool lo) {
  const int n = lo ? P->nana_lo[polar] : P->nana_items[polar];
  return launch_leg_fp64_items(P, 1, polar, lo ? (const void *)P->d_ana_lo[polar] : P->d_ana_items[polar], n, st);
}

cudaError_t launch_ana_reduce(const sht_plan_s *P, const DevPtrs &alm, int polar, int add, cudaStream_t st,
                              bool real, bool grad) {
  dim3 grid((P->lmax + 1 + 127) / 128, P->nm);
  ana_reduce<<<grid, 128, 0, st>>>(P->lmax, P->spin, P->nm, P->njobs_pad, P->ncomp, P->astride, add,
                                   real ? 1 : 0, grad ? 1 : 0,
                                   P->d_mval, P->d_mstart, P->d_coef_off, P->d_alpha, P->d_ana_part_off[polar],
                                   P->d_ana_nslot[polar],
                                   P->d_part, alm);
  return cudaGetLastError();
}

}  // namespace sht

// ---------------------------------------------------------------------------
// batches (sht_batch_execute): per-plan argument records and batched launches
// ---------------------------------------------------------------------------
namespace sht {

size_t leg_fp64_args_size() { return sizeof(LegArgs); }

void leg_fp64_fill_args(const sht_plan_s *P, int polar, void *out, bool lo) {
  LegArgs a = make_args(P, polar, lo);
  memcpy(out, &a, sizeof(a));
}

cudaError_t launch_alm_prepare_fp64(const sht_plan_s *P, const DevPtrs &alm, cudaStream_t st, int mode) {
  if (P->nm == 0) return cudaSuccess;
  dim3 g(P->nm, P->njobs_pad);
  alm_to_pm<<<g, kPmThreads, 0, st>>>(P->lmax, P->spin, P->nm, P->astride, P->d_mval, P->d_mstart, P->d_coef_off,
                               P->ncoef64, P->d_alpha, alm, P->d_pm64, mode,
                               P->tc64_syn ? reinterpret_cast<unsigned char *>(P->d_wide_syn) : nullptr);
  return cudaGetLastError();
}

// stage 0: synthesis, 1: analysis; all plans of the launch share spin class, njobs_pad and tiling
cudaError_t launch_leg_fp64_batch(int stage, int spin, int nj, int ppt, const void *args, const int4 *items,
                                  int n, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const LegArgs *a = static_cast<const LegArgs *>(args);
  if (stage == 0) {
    if (spin == 0) {
      switch (nj) {
        case 1: leg_syn_s0_batch<1><<<n, kSynTile, 0, st>>>(a, items); break;
        case 2: leg_syn_s0_batch<2><<<n, kSynTile, 0, st>>>(a, items); break;
        case 4: leg_syn_s0_batch<4><<<n, kSynTile, 0, st>>>(a, items); break;
        case 8: leg_syn_s0_batch<8><<<n, kSynTile, 0, st>>>(a, items); break;
        default: leg_syn_s0_batch<16><<<n, kSynTile, 0, st>>>(a, items); break;
      }
    } else {
      switch (nj) {
        case 1: leg_syn_spin_batch<1><<<n, kSynTile, 0, st>>>(a, items); break;
        case 2: leg_syn_spin_batch<2><<<n, kSynTile, 0, st>>>(a, items); break;
        case 4: leg_syn_spin_batch<4><<<n, kSynTile, 0, st>>>(a, items); break;
        default: leg_syn_spin_batch<8><<<n, kSynTile, 0, st>>>(a, items); break;
      }
    }
  } else {
    if (spin == 0)
      ana_shape_s0(nj, ppt, [&](auto sh) {
        leg_ana_s0_batch<decltype(sh)::nj, decltype(sh)::ppt><<<n, kAnaThreads, 0, st>>>(a, items);
      });
    else
      ana_shape_spin(nj, ppt, [&](auto sh) {
        leg_ana_spin_batch<decltype(sh)::nj, decltype(sh)::ppt><<<n, kAnaThreads, 0, st>>>(a, items);
      });
  }
  return cudaGetLastError();
}

}  // namespace sht
