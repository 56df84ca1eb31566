// The dash pattern and the walk of a quad over its on-stretches (Sec. 5.2): an FP32
// prefilter, the walk in double-float, and the FP64 rule that both follow.
// Every function is host- and device-callable so that the three can be compared
// on the CPU.
#pragma once

#include <math.h>
#include <stdint.h>
#include <vector_functions.h>

#include <cmath>

#if defined(PS_HD) && !defined(PS_DF_ROUNDED)
#error "ps_dash_walk.cuh comes before ps_df.cuh: its bounds need rounded operations"
#endif
#define PS_DF_ROUNDED
#include "ps_df.cuh"

namespace ps {

// FP64 operations that are not contracted
#if defined(__CUDA_ARCH__)
PS_HD double rn_mul(double a, double b) { return __dmul_rn(a, b); }
PS_HD double rn_add(double a, double b) { return __dadd_rn(a, b); }
PS_HD double rn_sub(double a, double b) { return __dsub_rn(a, b); }
PS_HD double rn_div(double a, double b) { return __ddiv_rn(a, b); }
#else
PS_HD double rn_mul(double a, double b) { return a * b; }
PS_HD double rn_add(double a, double b) { return a + b; }
PS_HD double rn_sub(double a, double b) { return a - b; }
PS_HD double rn_div(double a, double b) { return a / b; }
#endif

struct DashPattern {
  double cum[65];
  double period;
  double offset;
  float cum_f[65];             // the same in FP32, for the prefilter
  float cum_l[65];             // cum = cum_f + cum_l (+ ~2^-48 cum)
  float period_f, period_lo;   // period = period_f + period_lo (+ ~2^-48 period)
  float offset_f;
  float exact_below;           // 2^40 times the pattern's grid, or 0 (see DashWalkDF)
  uint32_t empty;              // on-stretches of no length
  int m2;
  int j_round;                 // ribs - 1 of a round cap at this dtheta
  const uint8_t* path_cap;     // cap style per path, or null: butt dash ends
  int n_path;
};

// The pattern's stretch ends, and false for a length that is negative or not a
// number, or a pattern of no length.  (An odd count is repeated.)  path_cap,
// n_path and j_round are the caller's.
inline bool dash_pattern(DashPattern& P, const float* h_pattern, int n_pattern, float offset) {
  P.m2 = (n_pattern % 2) ? 2 * n_pattern : n_pattern;
  P.cum[0] = 0.0;
  for (int i = 0; i < P.m2; ++i) {
    double d = (double)h_pattern[i % n_pattern];
    if (!(d >= 0.0)) return false;
    P.cum[i + 1] = P.cum[i] + d;
  }
  P.period = P.cum[P.m2];
  P.offset = (double)offset;
  P.empty = 0u;
  for (int i = 0; i < P.m2; i += 2)
    if (P.cum[i + 1] == P.cum[i]) P.empty |= 1u << (i >> 1);
  for (int i = 0; i <= P.m2; ++i) {
    P.cum_f[i] = (float)P.cum[i];
    P.cum_l[i] = (float)(P.cum[i] - (double)P.cum_f[i]);
  }
  P.period_f = (float)P.period;
  P.period_lo = (float)(P.period - (double)P.period_f);
  P.offset_f = offset;
  // the pattern's grid: the largest power of two that divides the offset, every
  // stretch end and the period, when all of them are FP32 numbers
  P.exact_below = 0.f;
  {
    int g = 1 << 20;  // exponent of the grid
    bool all = std::isfinite(P.period) && std::isfinite(P.offset);
    for (int i = 0; all && i <= P.m2 + 1; ++i) {
      const double v = i <= P.m2 ? P.cum[i] : P.offset;
      if (v == 0.0) continue;
      int e;
      const double m = std::frexp(std::fabs(v), &e);  // v = m 2^e, m in [1/2, 1)
      const int64_t q = (int64_t)std::ldexp(m, 53);   // v = q 2^(e - 53)
      const int z = __builtin_ctzll((unsigned long long)q);
      if (53 - z > 24) all = false;
      if (e - 53 + z < g) g = e - 53 + z;
    }
    if (all && g > -60 && g < 60) P.exact_below = (float)std::ldexp(1.0, g + 40);
  }
  return P.period > 0.0;
}

// FP32 prefilter: whether the quad [sa, sb] lies inside one interval of the
// pattern (an on-stretch or a gap) with a margin eps above the FP32 error of
// its phase.  The phase of sa is computed with error-free steps: sa + offset as
// an exact float pair (TwoSum), u - k period_f (exact but for k = -1: the result is below a
// period, and k period_f rounds to within a factor of two of u or to 0), the
// product's FMA residual and the period's low part.  What remains for k < 2^24
// is five roundings of values below two periods, at most 2^-24 of the period
// each (twice that above one period), the pattern's own FP32 rounding (2^-24) and the
// period's tail (2^-25): under 1e-6 of the period in all.  (Each operation is rounded by
// itself, rn_*: with k period_f fused into the difference its residual would count twice,
// k 2^-24 of a period.)  The FP64 rule's own
// roundings are below 2^-27 of it.  eps is 4e-6 of the period, so that few
// quads besides those that cross a boundary are left to the walk.
// 1: inside an on-stretch (the quad is emitted whole), 0: inside a gap
// (nothing), -1: crosses a boundary or lies within eps of one (see DashWalkDF).
PS_HD int dash_quick(const DashPattern& P, float sa, float sb) {
  const float per = P.period_f;
  const float eps = 4e-6f * per;
  const DF u = two_sum(sa, P.offset_f);
  const float k = floorf(u.hi / per);
  if (!(fabsf(k) < 16777216.f)) return -1;
  const DF kp = two_prod(k, per);
  // phase of sa
  const float ph = rn_sub(rn_sub(rn_add(rn_sub(u.hi, kp.hi), u.lo), kp.lo), rn_mul(k, P.period_lo));
  if (!(ph >= 0.f && ph < per)) return -1;
  const float pe = rn_add(ph, rn_sub(sb, sa));  // phase of sb, beyond the period if it wraps
  int j = 0;  // interval [cum_f[j], cum_f[j+1]) holding ph
  while (j + 1 < P.m2 && P.cum_f[j + 1] <= ph) ++j;
  if (ph - P.cum_f[j] > eps && P.cum_f[j + 1] - pe > eps) return (j & 1) ? 0 : 1;
  return -1;
}

// Walk of a quad [sa, sb] over the on-stretches of the pattern, in FP64 with
// explicitly rounded operations.  next() finds the next stretch that the quad
// keeps a piece [lo, hi] of, and whether that piece carries caps.
struct DashWalk {
  double sa, sb, k0;
  int guard, i;
  PS_HD void start(const DashPattern& P, float sa_f, float sb_f) {
    sa = (double)sa_f;
    sb = (double)sb_f;
    k0 = floor(rn_div(rn_add(sa, P.offset), P.period)) - 1.0;
    guard = 0;
    i = 0;
  }
  PS_HD bool next(const DashPattern& P, bool capped, double& lo, double& hi,
                                       bool& cap0, bool& cap1) {
    for (; guard < (1 << 20); ++guard, i = 0) {
      const double base = rn_mul(k0 + (double)guard, P.period);
      if (rn_sub(base, P.offset) > sb) {
        guard = 1 << 20;
        break;
      }
      while (i < P.m2) {
        const double a = rn_sub(rn_add(base, P.cum[i]), P.offset);
        const double b = rn_sub(rn_add(base, P.cum[i + 1]), P.offset);
        i += 2;
        if (!(b > a)) continue;
        bool keep;
        if (sb > sa) {
          lo = a > sa ? a : sa;
          hi = b < sb ? b : sb;
          keep = hi > lo;
        } else {
          lo = sa;
          hi = sb;
          keep = (sa >= a && sa < b);
        }
        if (!keep) continue;
        cap0 = capped && sb > sa && a >= sa && a < sb && a > 0.0;
        cap1 = capped && sb > sa && b > sa && b <= sb;
        return true;
      }
    }
    return false;
  }
};

// The same walk in double-float (ps_df.cuh) on the FP32 pipe.  A stretch end
// k period + cum - offset comes out within err = 2^-45 (|k| period + period +
// |offset|) of the FP64 rule's value: the roundings of the low parts sum to less
// than 2^-46 of that magnitude, the FP64 rule's own to 3 2^-53.  Every comparison of a
// stretch end with sa, sb or 0 is taken only when the two differ by more than
// err; otherwise sure is cleared and the quad goes to the FP64 walk.  err is 0 when
// the pattern is a multiple of a grid g (P.exact_below = 2^40 g; whole or
// quarter pixels, say) and the magnitude is below 2^40 g: then k period, the sums
// and the differences are exact in pairs and in FP64, and equality is decided
// too (at large s a quad often begins exactly at a stretch end, as s itself lies
// on a coarse FP32 grid).  Every operation is rounded by itself or an explicit fmaf,
// so that the counting and the writing pass walk a quad alike.  FP64 operations have a
// long latency here, and a tile waits for its slowest quad before it can publish its
// output count: with every queued quad in FP64 the kernel took 141 us on the 5,031-cubic path and
// 1,097 us on 1,000 paths with capped dashes, and 125 and 784 us this way.
struct DashWalkDF {
  float sa, sb, k0, err;
  int g, i;
  bool sure;
  PS_HD void start(const DashPattern& P, float sa_f, float sb_f) {
    sa = sa_f;
    sb = sb_f;
    const float u = rn_add(sa, P.offset_f);
    // the period that holds sa, or the one before where FP32 does not tell them apart
    k0 = floorf(u / P.period_f);
    if (!(fmaf(-k0, P.period_f, u) > fmaf(4e-6f, P.period_f, rn_mul(4e-7f, fabsf(u))))) k0 -= 1.f;
    const float n = rn_sub(sb, sa) / P.period_f;
    // (false for NaN; a period near FP32's range end has no exact products)
    sure = fabsf(k0) < 4194304.f && n < 1024.f && P.period_f > 1e-20f;
    const float mag = fmaf(fabsf(k0) + fabsf(n) + 4.f, P.period_f, fabsf(P.offset_f));
    err = mag < P.exact_below ? 0.f : rn_mul(2.8421709e-14f, mag);
    g = 0;
    i = 0;
  }
  // sign of end - x; sure is cleared when they are within err
  PS_HD int cmp(DF end, float x) {
    const float d = df_f(df_add_f(end, -x));
    if (!(err == 0.f || fabsf(d) > err)) sure = false;
    return d > 0.f ? 1 : d < 0.f ? -1 : 0;
  }
  // The next kept piece: its stretch's ends a, b; whether the piece begins at a
  // (else at sa) and ends at b (else at sb), and its caps.
  PS_HD bool next(const DashPattern& P, bool capped, DF& a, DF& b,
                                       bool& at_a, bool& at_b, bool& cap0, bool& cap1) {
    while (sure) {
      const float k = k0 + (float)g;
      const DF kp = two_prod(k, P.period_f);
      const DF base = df_add_f(
          fast_two_sum(kp.hi, fmaf(k, P.period_lo, kp.lo)), -P.offset_f);
      if (cmp(base, sb) > 0) return false;
      while (i < P.m2 && sure) {
        const DF c0{P.cum_f[i], P.cum_l[i]}, c1{P.cum_f[i + 1], P.cum_l[i + 1]};
        const bool empty = (P.empty >> (i >> 1)) & 1u;
        i += 2;
        if (empty) continue;
        if (!(rn_add(rn_sub(c1.hi, c0.hi), rn_sub(c1.lo, c0.lo)) > 2.f * err)) sure = false;
        b = df_add(base, c1);
        if (cmp(b, sa) <= 0) continue;
        a = df_add(base, c0);
        const int ca = cmp(a, sa);
        if (sb > sa) {
          if (cmp(a, sb) >= 0) continue;
          const int cb = cmp(b, sb);
          at_a = ca > 0;
          at_b = cb < 0;
          cap0 = capped && ca >= 0 && cmp(a, 0.f) > 0;
          cap1 = capped && cb <= 0;
        } else {
          if (ca > 0) continue;  // a <= sa < b is wanted
          at_a = at_b = cap0 = cap1 = false;
        }
        return sure;
      }
      ++g;
      i = 0;
    }
    return false;
  }
};

// A vertex coordinate at the fraction f (a pair, within fe) of a0 .. a1, rounded as the
// FP64 rule rounds it; ok is cleared where that rounding is not certain.
PS_HD float cut_coord(float a0, float a1, DF f, float fe, bool& ok) {
  const DF dv = df_diff(a1, a0);  // exact
  const DF v = df_add_f(df_mul(f, dv), a0);
  const float e = fmaf(fe + 5.6843419e-14f, fabsf(dv.hi),
                       rn_mul(5.6843419e-14f, fabsf(a0) + fabsf(a1)));
  ok &= v.hi + (v.lo + e) == v.hi && v.hi + (v.lo - e) == v.hi;
  return v.hi;
}
PS_HD float4 cut_rib(float4 v0, float4 v1, DF f, float fe, bool& ok) {
  return make_float4(cut_coord(v0.x, v1.x, f, fe, ok), cut_coord(v0.y, v1.y, f, fe, ok),
                     cut_coord(v0.z, v1.z, f, fe, ok), cut_coord(v0.w, v1.w, f, fe, ok));
}

}  // namespace ps
