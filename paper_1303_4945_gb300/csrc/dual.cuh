// dual.cuh -- two double-float recursions side by side in one thread: the +s and -s
// recursions of a ring pair, or the spin-0 recursions of two ring pairs.
//
// sm_103a's packed FP32 instructions (two lanes per issue slot, the same lane rate)
// halve the issue slots of sums and plain products.  Measured on GB300, in lane
// operations per second: packed add or multiply 38 T, with another instruction of the
// integer pipe beside it 37 T, scalar adds the same way 25 T; packed FMA with three
// different operands 26 T against 36 T scalar, so FMAs stay scalar.  Every lane
// rounds as the scalar forms of df.cuh and mixed_common.cuh do.
#pragma once
#include "mixed_common.cuh"

namespace sht {

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }

struct d2 {
  float2 h, l;
};
__device__ __forceinline__ f2 lane0(const d2 &a) { return {a.h.x, a.l.x}; }
__device__ __forceinline__ f2 lane1(const d2 &a) { return {a.h.y, a.l.y}; }
__device__ __forceinline__ d2 two_sum(float2 a, float2 b) {
  const float2 s = add2(a, b), bb = sub2(s, a);
  return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ d2 fast_two_sum(float2 a, float2 b) {
  const float2 s = add2(a, b);
  return {s, sub2(b, sub2(s, a))};
}
// u p - q, normalised (mul_sub of mixed_common.cuh in both lanes)
__device__ __forceinline__ d2 mul_sub(const d2 &u, const d2 &p, const d2 &q) {
  const float2 m = mul2(u.h, p.h);
  float2 e;
  e.x = __fmaf_rn(u.l.x, p.h.x, __fmaf_rn(u.h.x, p.l.x, __fmaf_rn(u.h.x, p.h.x, -m.x)));
  e.y = __fmaf_rn(u.l.y, p.h.y, __fmaf_rn(u.h.y, p.l.y, __fmaf_rn(u.h.y, p.h.y, -m.y)));
  const d2 s = two_sum(m, neg2(q.h));
  return fast_two_sum(s.h, add2(sub2(e, q.l), s.l));
}

// How a step forms u = a x + b.  kFast: spin s, |a x| >= |b| in both lanes (a fast
// two-sum); kCareful: any order; kPolar: the difference form of a polar warp.
enum StepMode { kFast, kCareful, kPolar };

// step_polar of mixed_common.cuh in both lanes, every lane rounded as there (spin s: one
// ring, +b and -b; spin 0: two rings)
struct DualState {
  d2 p, q;
};
template <bool SPIN>
__device__ __forceinline__ DualState dual_polar_step(float4 c, f3 y0, f3 y1, d2 p, d2 q) {
  const f2 a = {c.x, c.y}, b = {c.z, c.w};
  auto lane_of = [&](const f3 &y) {  // (a - 2) - a y as a pair (spin s: the same for both lanes)
    const float m = __fmul_rn(a.h, y.h);
    float e = __fmaf_rn(a.h, y.h, -m);
    e = __fmaf_rn(a.h, y.m, e);
    e = __fmaf_rn(a.l, y.h, e);
    const f2 t = two_sum(__fsub_rn(a.h, 2.0f), -m);
    return f2{t.h, __fadd_rn(__fsub_rn(a.l, e), t.l)};
  };
  const f2 t0 = lane_of(y0), t1 = SPIN ? t0 : lane_of(y1);
  d2 v = {make_float2(t0.h, t1.h), make_float2(t0.l, t1.l)};
  if (SPIN) {
    const d2 t = two_sum(v.h, make_float2(b.h, -b.h));
    v = {t.h, add2(add2(v.l, t.l), make_float2(b.l, -b.l))};
  }
  v = fast_two_sum(v.h, v.l);
  const float2 m = mul2(v.h, p.h);
  float2 e;
  e.x = __fmaf_rn(v.l.x, p.h.x, __fmaf_rn(v.h.x, p.l.x, __fmaf_rn(v.h.x, p.h.x, -m.x)));
  e.y = __fmaf_rn(v.l.y, p.h.y, __fmaf_rn(v.h.y, p.l.y, __fmaf_rn(v.h.y, p.h.y, -m.y)));
  const d2 s = two_sum(m, q.h);
  q = fast_two_sum(s.h, add2(add2(e, q.l), s.l));
  const d2 r = two_sum(p.h, q.h);
  p = fast_two_sum(r.h, add2(add2(p.l, q.l), r.l));
  return {p, q};
}
template <bool SPIN>
static __device__ __noinline__ DualState dual_polar_step_out(float4 c, f3 y0, f3 y1, d2 p, d2 q) {
  return dual_polar_step<SPIN>(c, y0, y1, p, q);
}

// The recursions of one thread.  SPIN: lane 0 runs lambda(+s), lane 1 (-1)^(l - l0)
// lambda(-s), whose recursion is p_{l+1} = (b - a x) p_l - p_{l-1}: the sign the spin
// columns need (in a polar warp lane 1 runs lambda(-s) itself, and d2 q holds the
// differences).  Spin 0: lane t runs ring pair t.  x: cos theta, or 1 - cos theta
// in a polar warp.
//
// PS: a polar warp's step.  Packed in both lanes, in line; called, where unrolled into a
// kernel's degrees it takes registers and instruction cache from the warps that never run
// it (tensor-core synthesis of two E/B pairs, lmax 127 on 257 Clenshaw-Curtis rings: scalar 66
// us, packed 57, called 53; the analysis of one at lmax 2047: 7.20 ms, 7.11, 7.20); or two
// scalar steps, where the registers are held to 80 (double-float analysis of one map, lmax
// 2047: 3.03 ms, packed 3.09, called 3.11).
enum PolarStep { kScalar, kPacked, kCalled };
template <bool SPIN, PolarStep PS>
struct Dual {
  d2 p, q;  // current and previous values
  f3 x[SPIN ? 1 : 2];

  __device__ __forceinline__ void step(StepMode mode, const float4 &c) {
    const f2 a = {c.x, c.y}, b = {c.z, c.w};
    if (mode == kPolar) {
      const f3 &y0 = x[0], &y1 = x[SPIN ? 0 : 1];
      if (PS == kScalar) {
        f2 p0 = lane0(p), q0 = lane0(q), p1 = lane1(p), q1 = lane1(q);
        step_polar(a, b, y0, p0, q0);
        step_polar(a, neg(b), y1, p1, q1);
        p = {make_float2(p0.h, p1.h), make_float2(p0.l, p1.l)};
        q = {make_float2(q0.h, q1.h), make_float2(q0.l, q1.l)};
      } else {
        const DualState n = PS == kCalled ? dual_polar_step_out<SPIN>(c, y0, y1, p, q) : dual_polar_step<SPIN>(c, y0, y1, p, q);
        p = n.p;
        q = n.q;
      }
      return;
    }
    d2 u;
    if (SPIN) {
      const f2 t = mul(a, x[0]);
      const f2 s0 = mode == kFast ? fast_two_sum(t.h, b.h) : two_sum(t.h, b.h);
      const f2 s1 = mode == kFast ? fast_two_sum(-t.h, b.h) : two_sum(-t.h, b.h);
      u.h = make_float2(s0.h, s1.h);
      u.l = make_float2(__fadd_rn(__fadd_rn(t.l, b.l), s0.l), __fadd_rn(__fsub_rn(b.l, t.l), s1.l));
    } else {
      const f2 t0 = mul(a, x[0]), t1 = mul(a, x[SPIN ? 0 : 1]);
      u.h = make_float2(t0.h, t1.h);
      u.l = make_float2(t0.l, t1.l);
    }
    const d2 n = mul_sub(u, p, q);
    q = p;
    p = n;
  }
  // a lane's start (join record), times the power of two f
  __device__ __forceinline__ void start(int lane, f2 cur, f2 prev, float f) {
    if (lane == 0) {
      p.h.x = cur.h * f;
      p.l.x = cur.l * f;
      q.h.x = prev.h * f;
      q.l.x = prev.l * f;
    } else {
      p.h.y = cur.h * f;
      p.l.y = cur.l * f;
      q.h.y = prev.h * f;
      q.l.y = prev.l * f;
    }
  }
  // the enhanced exponent's check (mixed_common.cuh) of both lanes
  __device__ __forceinline__ void rescale(int &s0, int &s1) {
    if (s0 < 0 && fabsf(p.h.x) > kScaleUp32) {
      start(0, lane0(p), lane0(q), kScaleFactor32);
      ++s0;
    }
    if (s1 < 0 && fabsf(p.h.y) > kScaleUp32) {
      start(1, lane1(p), lane1(q), kScaleFactor32);
      ++s1;
    }
  }
};

// the accumulation weight of a value at a scale (weight() of mixed_common.cuh)
__device__ __forceinline__ float scale_weight(int sc) { return sc == 0 ? 1.f : (sc == -1 ? kScaleFactor32 : 0.f); }

// the degree from which on |a x| >= |b| for every lane of the warp: |b| <= a |s| / (l + 1)
// as m <= l (a margin of 1% covers the roundings); lmax + 1 if a ring lies on the
// equator
__device__ __forceinline__ int fast_from(int as, float x, bool valid, int lmax) {
  const float need = valid ? (x > 0.f ? 1.01f * (float)as / x : 1e9f) : 0.f;
  const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(need));  // need >= 0
  return (int)fminf(ceilf(__uint_as_float(w)), (float)(lmax + 1));
}

}  // namespace sht
