// vp_cvpair.cuh -- one contact pair of the reaction coordinate (SM,
// "Collective coordinate"): C~(r) = C(r) S(r) with the rational contact
// function C = (1 + s + s^2)/(1 + s + s^2 + s^3 + s^4), s = (r/r0)^2 (the
// printed (1 - rho^6)/(1 - rho^10) with the factor (1 - s) cancelled) and the
// quintic switch S.  Shared by the batched kernel and the adjoint kernels.
#pragma once
#include "vp_internal.cuh"

namespace vp {

struct CvConst {
  ff inv_r0sq, rs, inv_w;
  float rs2, rc2_far;
  int steep;  // a near pair may have s > 1000: its D^3 may leave the FP32 range
};

__device__ __forceinline__ CvConst cv_const(const SimConst &c) {
  return CvConst{ff{c.cv_inv_r0sq_hi, c.cv_inv_r0sq_lo}, ff{c.cv_rs_hi, c.cv_rs_lo}, ff{c.cv_inv_w_hi, c.cv_inv_w_lo},
                 c.cv_rs2, c.cv_rc2_far, c.cv_steep};
}

// Two near pairs per lane, on the packed FP32 instructions (two operations per
// issue slot): the tile kernels are bound by instruction issue (79% of the
// slots, with one pair per lane), most of it this arithmetic.
__device__ __forceinline__ float2 f2_all(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 f2_neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) { return __ffma2_rn(b, f2_all(-1.0f), a); }
__device__ __forceinline__ float2 f2_nma(float2 a, float2 b, float2 c) { return __ffma2_rn(f2_neg(a), b, c); }  // c - a b

struct ff2 { float2 hi, lo; };
__device__ __forceinline__ ff2 ff2_all(ff a) { return {f2_all(a.hi), f2_all(a.lo)}; }
__device__ __forceinline__ ff2 ff2_fast_two_sum(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b);
  return {s, f2_sub(b, f2_sub(s, a))};
}
__device__ __forceinline__ ff2 ff2_two_sum(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b), bb = f2_sub(s, a);
  return {s, __fadd2_rn(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb))};
}
__device__ __forceinline__ ff2 ff2_two_diff(float2 a, float2 b) {
  const float2 s = f2_sub(a, b), bb = f2_sub(s, a);
  return {s, f2_sub(f2_sub(a, f2_sub(s, bb)), __fadd2_rn(b, bb))};
}
__device__ __forceinline__ ff2 ff2_add(ff2 x, ff2 y) {
  const ff2 s = ff2_two_sum(x.hi, y.hi);
  return ff2_fast_two_sum(s.hi, __fadd2_rn(s.lo, __fadd2_rn(x.lo, y.lo)));
}
__device__ __forceinline__ ff2 ff2_sub(ff2 x, ff2 y) {
  const ff2 s = ff2_two_diff(x.hi, y.hi);
  return ff2_fast_two_sum(s.hi, __fadd2_rn(s.lo, f2_sub(x.lo, y.lo)));
}
__device__ __forceinline__ ff2 ff2_add_f(ff2 x, float2 y) {
  const ff2 s = ff2_two_sum(x.hi, y);
  return ff2_fast_two_sum(s.hi, __fadd2_rn(s.lo, x.lo));
}
__device__ __forceinline__ ff2 ff2_mul(ff2 x, ff2 y) {
  const float2 p = __fmul2_rn(x.hi, y.hi);
  const float2 e = __ffma2_rn(x.hi, y.hi, f2_neg(p));
  return ff2_fast_two_sum(p, __ffma2_rn(x.hi, y.lo, __ffma2_rn(x.lo, y.hi, e)));
}
__device__ __forceinline__ ff2 ff2_mul_f(ff2 x, float2 y) {
  const float2 p = __fmul2_rn(x.hi, y);
  const float2 e = __ffma2_rn(x.hi, y, f2_neg(p));
  return ff2_fast_two_sum(p, __ffma2_rn(x.lo, y, e));
}
__device__ __forceinline__ ff2 ff2_sqr(ff2 x) {
  const float2 p = __fmul2_rn(x.hi, x.hi);
  const float2 e = __ffma2_rn(x.hi, x.hi, f2_neg(p));
  return ff2_fast_two_sum(p, __ffma2_rn(__fadd2_rn(x.hi, x.hi), x.lo, e));
}
__device__ __forceinline__ ff2 ff2_div(ff2 x, ff2 y) {
  const float2 q = make_float2(__fdividef(x.hi.x, y.hi.x), __fdividef(x.hi.y, y.hi.y));
  const ff2 r = ff2_sub(x, ff2_mul_f(y, q));
  return ff2_fast_two_sum(q, make_float2(__fdividef(r.hi.x, y.hi.x), __fdividef(r.hi.y, y.hi.y)));
}

// Correctly rounded quotients and roots by Markstein's final step (IBM J. Res.
// Dev. 34, 1990): a Newton step on the hardware's approximation gives the
// correctly rounded reciprocal, and one on the quotient's (root's) remainder the
// correctly rounded result.  The hardware's approximations are not specified
// closely enough to prove that, so the tests compare every significand of
// reciprocals and roots, and quotients next to a midpoint, with the operators.  For
// numbers away from the range's ends: a denominator lies below RCP_TOP (from there
// on its reciprocal is denormal, which the approximation flushes, and an infinite
// one gives NaN), a radicand or dividend not below 2^-100 (its remainder would be
// denormal; smaller dividends occur in terms far below the sums' unit of 2^-32).
constexpr float RCP_TOP = 8.507059e37f;  // 2^126
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float2 f2_rcp(float2 b) {
  const float2 r = make_float2(rcp_approx(b.x), rcp_approx(b.y));
  return __ffma2_rn(r, f2_nma(b, r, f2_all(1.0f)), r);
}
__device__ __forceinline__ float2 f2_div(float2 a, float2 b, float2 rb) {  // rb = f2_rcp(b)
  const float2 q = __fmul2_rn(a, rb);
  return __ffma2_rn(f2_nma(b, q, a), rb, q);
}
__device__ __forceinline__ float2 f2_sqrt(float2 x) {
  const float2 y = make_float2(rsqrt_approx(x.x), rsqrt_approx(x.y));
  const float2 g = __fmul2_rn(x, y), h = __fmul2_rn(y, f2_all(0.5f));
  return __ffma2_rn(f2_nma(g, g, x), h, g);
}

struct CvPair2 {
  ff2 Ct;
  float2 dCt, d2Ct, r;
};

// C'(s) and (SECOND) C''(s) without the powers of D, whose FP32 range ends at
// r = 255 r0 (D^2) and 40 r0 (D^3): every quotient is over D itself.  Beside the
// usual form, for the pairs that need it: the usual one takes a third of the
// quotients, and its results stay what they were.
template <bool SECOND>
__device__ __forceinline__ float2 cv_far_slopes(float t) {
  const float N = 1.0f + t + t * t, D = N + t * t * t + t * t * t * t;
  const float n = N / D, n1 = (1.0f + 2.0f * t) / D, d1 = (1.0f + 2.0f * t + 3.0f * t * t + 4.0f * t * t * t) / D;
  const float Cs = n1 - n * d1;
  return make_float2(Cs, SECOND ? 2.0f / D - n * ((2.0f + 6.0f * t + 12.0f * t * t) / D) - 2.0f * d1 * Cs : 0.0f);
}

template <bool SECOND>
__device__ __forceinline__ CvPair2 cv_contact2(ff2 r2, const CvConst &k) {
  CvPair2 o;
  const ff2 s = ff2_mul(r2, ff2_all(k.inv_r0sq));
  {
    const ff2 s2 = ff2_sqr(s), s3 = ff2_mul(s2, s), s4 = ff2_sqr(s2);
    const ff2 N = ff2_add(ff2_add_f(s, f2_all(1.0f)), s2);
    o.Ct = ff2_div(N, ff2_add(ff2_add(N, s3), s4));
  }
  o.r = f2_sqrt(r2.hi);
  const float2 ds = __fmul2_rn(__fadd2_rn(o.r, o.r), f2_all(k.inv_r0sq.hi));
  // C'(s), C''(s)
  const float2 t = s.hi, t2 = __fmul2_rn(t, t), t3 = __fmul2_rn(t2, t);
  const float2 N = __fadd2_rn(__fadd2_rn(t, f2_all(1.0f)), t2);
  const float2 D = __ffma2_rn(t3, t, __fadd2_rn(N, t3));
  const float2 N1 = __ffma2_rn(t, f2_all(2.0f), f2_all(1.0f));
  const float2 D1 = __ffma2_rn(__fmul2_rn(__fmul2_rn(t, f2_all(4.0f)), t), t, __ffma2_rn(__fmul2_rn(t, f2_all(3.0f)), t, N1));
  const float2 W = __ffma2_rn(N1, D, f2_neg(__fmul2_rn(N, D1))), DD = __fmul2_rn(D, D);
  float2 Cs = f2_div(W, DD, f2_rcp(DD));
  float2 d2 = f2_all(0.0f), top = DD;  // top: the largest denominator
  if (SECOND) {
    const float2 D2 = __ffma2_rn(__fmul2_rn(t, f2_all(12.0f)), t, __ffma2_rn(t, f2_all(6.0f), f2_all(2.0f)));
    const float2 A1 = f2_nma(N, D2, __fadd2_rn(D, D));
    const float2 num = __ffma2_rn(A1, D, f2_neg(__fmul2_rn(__fadd2_rn(D1, D1), W)));
    top = __fmul2_rn(DD, D);
    d2 = f2_div(num, top, f2_rcp(top));
  }
  if (k.steep) {
    if (!(top.x < RCP_TOP)) { const float2 v = cv_far_slopes<SECOND>(t.x); Cs.x = v.x; d2.x = v.y; }
    if (!(top.y < RCP_TOP)) { const float2 v = cv_far_slopes<SECOND>(t.y); Cs.y = v.x; d2.y = v.y; }
  }
  o.dCt = __fmul2_rn(Cs, ds);
  if (SECOND)
    o.d2Ct = __ffma2_rn(__fadd2_rn(Cs, Cs), f2_all(k.inv_r0sq.hi), __fmul2_rn(__fmul2_rn(d2, ds), ds));
  const bool sx = r2.hi.x > k.rs2, sy = r2.hi.y > k.rs2;
  if (sx || sy) {
    // ff_sqrt, from the root already there
    const float2 y = o.r, yy = __fmul2_rn(y, y);
    const ff2 rem = ff2_sub(r2, ff2{yy, __ffma2_rn(y, y, f2_neg(yy))});
    const float2 y2 = __fadd2_rn(y, y);
    const ff2 r = ff2_fast_two_sum(y, make_float2(__fdividef(rem.hi.x, y2.x), __fdividef(rem.hi.y, y2.y)));
    const ff2 x = ff2_mul(ff2_add(r, ff2_all(ff_neg(k.rs))), ff2_all(k.inv_w));
    ff2 p = ff2_add_f(ff2_mul_f(x, f2_all(6.0f)), f2_all(-15.0f));
    p = ff2_add_f(ff2_mul(p, x), f2_all(10.0f));
    const ff2 m = ff2_mul(ff2_mul(ff2_sqr(x), x), p);
    // S = 1 - m
    const float2 one = f2_all(1.0f), sh = f2_sub(one, m.hi), bb = __fadd2_rn(sh, m.hi);
    const float2 se = f2_sub(f2_sub(one, bb), __fadd2_rn(m.hi, f2_sub(sh, bb)));
    const ff2 S = ff2_fast_two_sum(sh, f2_sub(se, m.lo));
    const float2 xf = x.hi, y1 = f2_sub(one, xf);
    const float2 S1 = __fmul2_rn(
        __fmul2_rn(__fmul2_rn(__fmul2_rn(__fmul2_rn(xf, f2_all(-30.0f)), xf), y1), y1), f2_all(k.inv_w.hi));
    const float2 c1 = SECOND ? __ffma2_rn(o.Ct.hi, S1, __fmul2_rn(o.dCt, S.hi))
                             : __ffma2_rn(o.dCt, S.hi, __fmul2_rn(o.Ct.hi, S1));
    const ff2 cs = ff2_mul(o.Ct, S);
    const bool zx = x.hi.x >= 1.0f, zy = x.hi.y >= 1.0f;
    if (SECOND) {
      const float2 iw = f2_all(k.inv_w.hi);
      const float2 q = __ffma2_rn(__fmul2_rn(xf, f2_all(180.0f)), xf, __fmul2_rn(xf, f2_all(-60.0f)));
      const float2 S2 = __fmul2_rn(
          __fmul2_rn(f2_nma(__fmul2_rn(__fmul2_rn(xf, f2_all(120.0f)), xf), xf, q), iw), iw);
      const float2 c2 = __ffma2_rn(o.Ct.hi, S2, __ffma2_rn(__fadd2_rn(o.dCt, o.dCt), S1, __fmul2_rn(o.d2Ct, S.hi)));
      if (sx) o.d2Ct.x = zx ? 0.f : c2.x;
      if (sy) o.d2Ct.y = zy ? 0.f : c2.y;
    }
    if (sx) { o.dCt.x = zx ? 0.f : c1.x; o.Ct.hi.x = zx ? 0.f : cs.hi.x; o.Ct.lo.x = zx ? 0.f : cs.lo.x; }
    if (sy) { o.dCt.y = zy ? 0.f : c1.y; o.Ct.hi.y = zy ? 0.f : cs.hi.y; o.Ct.lo.y = zy ? 0.f : cs.lo.y; }
  }
  return o;
}

// The squared distance below which the FP32 tests take a pair as near: they round
// a coordinate difference d by 2^-24 d before its images are taken off, so with
// atoms hundreds of boxes apart the margin in rc2_far (1e-4) does not do, and the
// limit grows with the largest d^2.  (Pairs beyond the cut-off add zeros.)
__device__ __forceinline__ float cv_near2(float rc2_far, float d2) {
  return fmaxf(rc2_far, fminf(1.1e-10f * d2 + rc2_far, 1e6f));
}

// exact minimum-image differences x_j - x_i as float-float
__device__ __forceinline__ void cv_delta2(float4 xi0, float4 xi1, float4 xj0, float4 xj1, float L, float iL, ff2 &dx,
                                          ff2 &dy, ff2 &dz) {
  dx = ff2_two_diff(make_float2(xj0.x, xj1.x), make_float2(xi0.x, xi1.x));
  dy = ff2_two_diff(make_float2(xj0.y, xj1.y), make_float2(xi0.y, xi1.y));
  dz = ff2_two_diff(make_float2(xj0.z, xj1.z), make_float2(xi0.z, xi1.z));
  // adding 1.5 2^23 and taking it away rounds to whole numbers (an image
  // number of 2^22 would leave FP32 positions without a digit below the box)
  const float2 il = f2_all(iL), m = f2_all(12582912.0f);
  const float2 nx = f2_sub(__fadd2_rn(__fmul2_rn(dx.hi, il), m), m), ny = f2_sub(__fadd2_rn(__fmul2_rn(dy.hi, il), m), m),
               nz = f2_sub(__fadd2_rn(__fmul2_rn(dz.hi, il), m), m);
  if (nx.x != 0.f || nx.y != 0.f || ny.x != 0.f || ny.y != 0.f || nz.x != 0.f || nz.y != 0.f) {
    const float2 l = f2_all(-L);
    dx = ff2_add_f(dx, __fmul2_rn(l, nx));
    dy = ff2_add_f(dy, __fmul2_rn(l, ny));
    dz = ff2_add_f(dz, __fmul2_rn(l, nz));
  }
}

}  // namespace vp
