// Double-float arithmetic on the FP32 pipe: a value is an unevaluated pair of
// floats (hi, lo) with |lo| <= ulp(hi)/2, about 48 significant bits.  The
// building blocks are the error-free transformations TwoSum (Knuth, TAOCP
// vol. 2, 4.2.2), Fast2Sum (Dekker 1971) and the FMA form of TwoProduct; the
// pair operations follow Dekker (1971) and the double-double library of
// Hida, Li and Bailey (2001) in their "sloppy" form (error ~2^-48 of the
// operands' magnitude).
//
// On top of them: sin/cos of a double-float angle by table-driven reduction
// (Tang 1990; the table holds sin, cos of k pi/256 as float pairs) with a
// three-part Cody-Waite constant (Cody & Waite 1980) and Taylor terms on the
// reduced argument |r| <= pi/512; atan2 as the FP32 atan2f refined by one
// rotation (the tangent of the residual angle, which is ~1e-7, equals the
// residual to far below double-float rounding).
//
// GB300 issues FP64 at ~1/60 of its FP32 rate: the mixed-precision
// tessellation carries its angles, normals, parameters and vertices in these
// pairs instead of FP64.
//
// Every function is host- and device-callable so that the arithmetic can be
// checked on the CPU.
#pragma once

#include <math.h>
#include <vector_types.h>

#include "ps_sincos_table.h"

#if defined(__CUDACC__)
#define PS_HD __host__ __device__ __forceinline__
#else
#define PS_HD inline
#endif

namespace ps {

struct DF {
  float hi, lo;
};
struct DF2 {
  DF x, y;
};

// The operations of the scalar pairs.  From plain operators a compiler may fuse a product into
// the sum that it goes into, and its rounding error is then counted twice.  Where results rest on
// error bounds, PS_DF_ROUNDED (defined before this header) has each rounded by itself; the
// tessellation, which is checked against 64 bits instead, keeps the operators (rounded by
// themselves they cost the rib kernel registers: 10,417 -> 10,539 us on a million near-cusp
// cubics).
#if defined(PS_DF_ROUNDED) && defined(__CUDA_ARCH__)
PS_HD float rn_mul(float a, float b) { return __fmul_rn(a, b); }
PS_HD float rn_add(float a, float b) { return __fadd_rn(a, b); }
PS_HD float rn_sub(float a, float b) { return __fsub_rn(a, b); }
#else
PS_HD float rn_mul(float a, float b) { return a * b; }
PS_HD float rn_add(float a, float b) { return a + b; }
PS_HD float rn_sub(float a, float b) { return a - b; }
#endif

PS_HD DF df_of(float a) { return DF{a, 0.f}; }
PS_HD float df_f(DF a) { return rn_add(a.hi, a.lo); }
PS_HD double df_d(DF a) { return (double)a.hi + (double)a.lo; }
PS_HD DF df_from_d(double v) {
  float h = (float)v;
  return DF{h, (float)(v - (double)h)};
}

// |a| >= |b| (or a == 0): s + e == a + b exactly
PS_HD DF fast_two_sum(float a, float b) {
  float s = rn_add(a, b);
  return DF{s, rn_sub(b, rn_sub(s, a))};
}
PS_HD DF two_sum(float a, float b) {
  float s = rn_add(a, b);
  float bb = rn_sub(s, a);
  return DF{s, rn_add(rn_sub(a, rn_sub(s, bb)), rn_sub(b, bb))};
}
PS_HD DF two_prod(float a, float b) {
  float p = rn_mul(a, b);
  return DF{p, fmaf(a, b, -p)};
}
PS_HD DF df_neg(DF a) { return DF{-a.hi, -a.lo}; }
PS_HD DF df_add(DF a, DF b) {
  DF s = two_sum(a.hi, b.hi);
  return fast_two_sum(s.hi, rn_add(s.lo, rn_add(a.lo, b.lo)));
}
PS_HD DF df_sub(DF a, DF b) { return df_add(a, df_neg(b)); }
PS_HD DF df_add_f(DF a, float b) {
  DF s = two_sum(a.hi, b);
  return fast_two_sum(s.hi, rn_add(s.lo, a.lo));
}
PS_HD DF df_mul(DF a, DF b) {
  float p = rn_mul(a.hi, b.hi);
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
  return fast_two_sum(p, e);
}
PS_HD DF df_mul_f(DF a, float b) {
  float p = rn_mul(a.hi, b);
  float e = fmaf(a.hi, b, -p);
  e = fmaf(a.lo, b, e);
  return fast_two_sum(p, e);
}
// a / b: the quotient's residual a.hi - q b is exact under an FMA
PS_HD DF df_div_f(DF a, float b) {
  float q = a.hi / b;
  float r = fmaf(-q, b, a.hi);
  return fast_two_sum(q, (r + a.lo) / b);
}
PS_HD DF df_div(DF a, DF b) {
  float q = a.hi / b.hi;
  DF r = df_sub(a, df_mul_f(b, q));
  return fast_two_sum(q, r.hi / b.hi);
}
PS_HD DF df_sqrt(DF a) {
  if (!(a.hi > 0.f)) return DF{0.f, 0.f};
  const float s = sqrtf(a.hi);
  const DF e = df_sub(a, two_prod(s, s));
  return fast_two_sum(s, e.hi / (2.f * s));
}
PS_HD bool df_lt(DF a, DF b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
PS_HD bool df_le(DF a, DF b) { return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo); }
PS_HD DF df_abs(DF a) { return (a.hi < 0.f || (a.hi == 0.f && a.lo < 0.f)) ? df_neg(a) : a; }
PS_HD bool df_is0(DF a) { return a.hi == 0.f && a.lo == 0.f; }
// b - a for floats, exactly
PS_HD DF df_diff(float b, float a) { return two_sum(b, -a); }
// a.x b.y - a.y b.x and a.x b.x + a.y b.y
PS_HD DF df_cross(DF2 a, DF2 b) { return df_sub(df_mul(a.x, b.y), df_mul(a.y, b.x)); }
PS_HD DF df_dot(DF2 a, DF2 b) { return df_add(df_mul(a.x, b.x), df_mul(a.y, b.y)); }

// A lazily normalized sum: value s + e, where e gathers the rounding errors of
// the terms added to s (|e| need not be below ulp(s)/2).  Sums of a few exact
// products of pairs reach the same ~2^-48 accuracy as normalized pair
// arithmetic with fewer operations.
struct Acc {
  float s, e;
};
// A += x y (x, y pairs)
PS_HD void acc_prod(Acc& A, DF x, DF y) {
  const DF p = two_prod(x.hi, y.hi);
  const DF t = two_sum(A.s, p.hi);
  A.e = rn_add(A.e, rn_add(t.lo, rn_add(p.lo, fmaf(x.hi, y.lo, rn_mul(x.lo, y.hi)))));
  A.s = t.hi;
}
PS_HD Acc acc_first(DF x, DF y) {
  const DF p = two_prod(x.hi, y.hi);
  return Acc{p.hi, rn_add(p.lo, fmaf(x.hi, y.lo, rn_mul(x.lo, y.hi)))};
}
PS_HD float acc_round(Acc A) { return rn_add(A.s, A.e); }

// Two pairs side by side, x and y of a point or sine and cosine of an angle: each operation is
// the scalar one above on both, one packed FP32 instruction (two lanes, each rounded as
// its scalar form) in place of two, and gives the same bits.  Where both coordinates take the
// same steps this halves the issue slots of the rib kernel's arithmetic, which is what
// bounds it (k_emit on 211 M ribs of near cusps 10.16 -> 9.10 ms, on the 43 M ribs of the bench
// workload 1,695 -> 1,603 us).
struct F2 {
  float x, y;
};
struct DFP {
  F2 hi, lo;
};
PS_HD F2 f2_fma(F2 a, F2 b, F2 c) {
#if defined(__CUDA_ARCH__)
  const float2 r = __ffma2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y), make_float2(c.x, c.y));
  return F2{r.x, r.y};
#else
  return F2{fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)};
#endif
}
PS_HD F2 f2_add(F2 a, F2 b) {
#if defined(__CUDA_ARCH__)
  const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
  return F2{r.x, r.y};
#else
  return F2{a.x + b.x, a.y + b.y};
#endif
}
PS_HD F2 f2_mul(F2 a, F2 b) {
#if defined(__CUDA_ARCH__)
  const float2 r = __fmul2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
  return F2{r.x, r.y};
#else
  return F2{a.x * b.x, a.y * b.y};
#endif
}
PS_HD F2 f2_of(float a) { return F2{a, a}; }
PS_HD F2 f2_neg(F2 a) { return F2{-a.x, -a.y}; }
PS_HD F2 f2_sub(F2 a, F2 b) { return f2_add(a, f2_neg(b)); }

PS_HD DFP two_sum2(F2 a, F2 b) {
  const F2 s = f2_add(a, b), bb = f2_sub(s, a);
  return DFP{s, f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb))};
}
// a - b exactly
PS_HD DFP two_diff2(F2 a, F2 b) {
  const F2 s = f2_sub(a, b), bb = f2_sub(s, a);
  return DFP{s, f2_sub(f2_sub(a, f2_sub(s, bb)), f2_add(b, bb))};
}
PS_HD DFP fast_two_sum2(F2 a, F2 b) {
  const F2 s = f2_add(a, b);
  return DFP{s, f2_sub(b, f2_sub(s, a))};
}
// x.hi y.lo + x.lo y.hi, the small terms of a product
PS_HD F2 cross_terms2(DFP x, DF y) {
  return f2_fma(x.hi, f2_of(y.lo), f2_mul(x.lo, f2_of(y.hi)));
}
struct Acc2 {
  F2 s, e;
};
// A += x y (y the same pair for both)
PS_HD void acc_prod2(Acc2& A, DFP x, DF y) {
  const F2 m = f2_neg(f2_mul(x.hi, f2_of(y.hi)));  // -p
  const F2 pe = f2_fma(x.hi, f2_of(y.hi), m);
  const DFP t = two_diff2(A.s, m);
  A.e = f2_add(A.e, f2_add(t.lo, f2_add(pe, cross_terms2(x, y))));
  A.s = t.hi;
}
PS_HD Acc2 acc_first2(DFP x, DF y) {
  const F2 m = f2_neg(f2_mul(x.hi, f2_of(y.hi)));
  return Acc2{f2_mul(x.hi, f2_of(y.hi)), f2_add(f2_fma(x.hi, f2_of(y.hi), m), cross_terms2(x, y))};
}
// a + g + x y rounded once (a floats; g, x, y pairs): s1 = two_sum2(a, g.hi), gl = g.lo
PS_HD F2 sum_prod_round2(DFP s1, F2 gl, DFP x, DF y) {
  const F2 m = f2_neg(f2_mul(x.hi, f2_of(y.hi)));
  const F2 pe = f2_fma(x.hi, f2_of(y.hi), m);
  const DFP s2 = two_diff2(s1.hi, m);
  return f2_add(s2.hi, f2_add(s2.lo, f2_add(f2_add(s1.lo, gl), f2_add(pe, cross_terms2(x, y)))));
}

PS_HD DF df_pi() { return DF{PS_DF_PI_HI, PS_DF_PI_LO}; }
PS_HD DF df_two_pi() { return DF{PS_DF_TWO_PI_HI, PS_DF_TWO_PI_LO}; }
PS_HD DF df_sqrt2() { return DF{PS_DF_SQRT2_HI, PS_DF_SQRT2_LO}; }

PS_HD float4 sc_tab_load(const float4* tab, int i) {
#if defined(__CUDA_ARCH__)
  return __ldg(tab + i);
#else
  return tab[i];
#endif
}

// sin and cos of x (|x| < 2^10) to ~1e-14 absolute.  tab: the 512 entries of
// ps_sincos_table.h.
//   k = nearest integer to x 256/pi, r = x - k pi/256 (|r| <= pi/512):
//   x.hi - k C1 is exact under an FMA (C1 has 24 bits, the difference is a
//   multiple of 2^-31 below 2^-7); C2 and C3 extend C1 to ~72 bits of pi/256.
//   sin r = r - r^3/6 + r^5/120 and cos r = 1 - (r^2/2 - r^4/24): the omitted
//   terms are below 1e-17 at |r| <= pi/512; the small terms are FP32 (their
//   rounding is ~2^-24 of 4e-8), the leading r and r^2/2 pairs are exact.
//   sin(a + r) = S_a - S_a c + C_a sin r, cos(a + r) = C_a - C_a c - S_a sin r
//   with c = 1 - cos r.
PS_HD void df_sincos(DF x, const float4* tab, DF& s, DF& c) {
  const float kf = rintf(x.hi * PS_256_OVER_PI);
  const int k = (int)kf;
  const float r1 = fmaf(-kf, PS_PI256_1, x.hi);
  DF r = two_sum(r1, x.lo);
  r = df_sub(r, two_prod(kf, PS_PI256_2));
  r = fast_two_sum(r.hi, fmaf(-kf, PS_PI256_3, r.lo));
  const float rh = r.hi, rl = r.lo;
  const float r2 = rh * rh;
  // sin r = rh + (rl - rh^3/6 + rh^5/120 - rl rh^2/2)
  const float st = fmaf(-rh * r2, fmaf(-r2, 1.f / 120.f, 1.f / 6.f), rl * fmaf(-0.5f, r2, 1.f));
  const DF sr = fast_two_sum(rh, st);
  // 1 - cos r = rh^2/2 - rh^4/24 + rh rl
  const DF h2 = two_prod(rh, rh);
  const DF cr = fast_two_sum(0.5f * h2.hi, fmaf(0.5f, h2.lo, fmaf(rh, rl, -r2 * r2 * (1.f / 24.f))));
  const float4 e = sc_tab_load(tab, k & 511);
  // S_a + C_a sin r - S_a c and C_a - S_a sin r - C_a c side by side, the products exact
  // in their high parts, the remaining terms gathered in FP32 (all below 2^-24 of
  // the result's ulp)
  const DFP A{F2{e.x, e.z}, F2{e.y, e.w}};    // S_a, C_a
  const DFP B{F2{e.z, -e.x}, F2{e.w, -e.y}};  // C_a, -S_a
  const F2 m1 = f2_mul(B.hi, f2_of(-sr.hi)), e1 = f2_fma(B.hi, f2_of(sr.hi), m1);
  const F2 m2 = f2_mul(A.hi, f2_of(-cr.hi)), e2 = f2_fma(A.hi, f2_of(cr.hi), m2);
  const DFP a = two_diff2(A.hi, m1), b = two_sum2(a.hi, m2);
  const F2 lo = f2_add(f2_add(f2_add(a.lo, b.lo), f2_add(A.lo, f2_sub(e1, e2))),
                       f2_sub(cross_terms2(B, sr), cross_terms2(A, cr)));
  const DFP v = fast_two_sum2(b.hi, lo);
  s = DF{v.hi.x, v.lo.x};
  c = DF{v.hi.y, v.lo.y};
}

// atan2(y, x) in (-pi, pi] to ~1e-14 (y = +0, x < 0 gives +pi).  a0 = atan2f (a few ulp); with
// (S, C) = sincos(a0), the residual angle is atan(u), u = (y C - x S)/(x C + y S),
// and |u| ~ 1e-7 makes atan(u) = u to ~1e-21.  (0, 0) gives atan2f's value.
PS_HD DF df_atan2(DF y, DF x, const float4* tab) {
  const float a0 = atan2f(y.hi, x.hi);
  if (x.hi == 0.f && y.hi == 0.f) return DF{a0, 0.f};
  // directions along an axis give the pair nearest 0, pi/2, pi, -pi/2 exactly,
  // so that exact reversals and right angles are decided as in FP64
  if (y.hi == 0.f && y.lo == 0.f) return x.hi > 0.f ? DF{0.f, 0.f} : df_pi();
  if (x.hi == 0.f && x.lo == 0.f)
    return y.hi > 0.f ? DF{PS_DF_HALF_PI_HI, PS_DF_HALF_PI_LO} : DF{-PS_DF_HALF_PI_HI, -PS_DF_HALF_PI_LO};
  DF S, C;
  df_sincos(DF{a0, 0.f}, tab, S, C);
  const DF num = df_sub(df_mul(y, C), df_mul(x, S));
  const float den = fmaf(x.hi, C.hi, y.hi * S.hi);
  return two_sum(a0, df_f(num) / den);
}

// x modulo 2 pi into [0, 2 pi) for |x| < 4 pi (one or two corrections)
PS_HD DF df_mod2pi(DF x) {
  const DF tp = df_two_pi();
  if (df_lt(x, df_of(0.f))) x = df_add(x, tp);
  if (df_lt(x, df_of(0.f))) x = df_add(x, tp);
  if (df_le(tp, x)) x = df_sub(x, tp);
  if (df_le(tp, x)) x = df_sub(x, tp);
  return x;
}

// a (-) b into (-pi, pi]: the relative angle of Sec. 3.2.2, one correction by
// 2 pi (callers map an exact reversal, -pi, to +pi)
PS_HD DF df_ominus(DF a, DF b) {
  DF d = df_sub(a, b);
  const DF pi = df_pi();
  if (df_lt(pi, d)) return df_sub(d, df_two_pi());
  if (df_lt(d, df_neg(pi))) return df_add(d, df_two_pi());
  return d;
}

}  // namespace ps
