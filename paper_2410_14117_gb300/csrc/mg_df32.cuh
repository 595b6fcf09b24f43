// Two-float arithmetic for the set-up kernels: a value is the unevaluated sum h + l of two FP32
// numbers, |l| <= ulp(h) / 2.  GB300 executes FP64 at a 64th of the FP32 rate, which made the
// domain randomisation (some 380 FP64 warp instructions per 32 envs) a quarter of a 100-sub-step
// episode of a 1,048,576-env fleet.  The sums and products below are exact or good to 2^-45, the
// elementary functions to 2^-41 (every uniform draw checked against 64-bit mantissas: radius
// 2^-41.4, sine and cosine 2^-41.8).  A result is rounded to FP32 from here only where both ends of
// its error bound round alike (round_df); the few others are left to FP64, so what is stored is
// what FP64 arithmetic stores, bit for bit.
//
// Published methods: Knuth's two-sum, Dekker's fast two-sum and the FMA two-product; the series of
// atanh, sin and cos.  Every operation is an explicit round-to-nearest intrinsic, so the compiler
// contracts and reorders nothing.
#pragma once

namespace mg {

struct df32 {
  float h, l;
};

// a + b exactly.
__device__ __forceinline__ df32 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
// a + b exactly for |a| >= |b| (or a = 0).
__device__ __forceinline__ df32 fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
// a b exactly (barring underflow).
__device__ __forceinline__ df32 two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ df32 df_mul(df32 a, df32 b) {
  const df32 p = two_prod(a.h, b.h);
  return {p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l))};
}
// c + p for |c| >= |p|, renormalised.
__device__ __forceinline__ df32 df_add_small(df32 c, df32 p) {
  const df32 s = fast_two_sum(c.h, p.h);
  return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(c.l, p.l)));
}

// A double constant in two floats.
__device__ __forceinline__ constexpr df32 df_const(double c) {
  return {(float)c, (float)(c - (double)(float)c)};
}

// q + r, |r| << |q|, rounded to FP32.  open: some number within w rel of it rounds otherwise (or it
// is not finite).
__device__ __forceinline__ float round_df(float q, float r, float w, float rel, bool &open) {
  const float f = __fadd_rn(q, __fmaf_rn(w, rel, r));
  open = !(f == __fadd_rn(q, __fmaf_rn(-w, rel, r)));
  return f;
}

// 1 / (a.h + a.l) rounded to FP32; open as in round_df.  The residual is exact but for its last
// rounding (2^-47 of the result), the neglected square of it 2^-47.
__device__ __forceinline__ float df_rcp(df32 a, bool &open) {
  const float r = __frcp_rn(a.h);
  const float e = __fmaf_rn(-a.l, r, __fmaf_rn(-a.h, r, 1.f));
  const float f = round_df(r, __fmul_rn(r, e), r, 0x1p-43f, open);
  open = open || !(a.h > 1e-20f && a.h < 1e20f);
  return f;
}

// sqrt(-2 ln u) for u in (0, 1).  u = 2^e m with m in [sqrt(1/2), sqrt(2)); with s = (m - 1) /
// (m + 1), ln m = 2 atanh s = 2 s (1 + z/3 + z^2/5 + ...), z = s^2 <= 0.0295; the terms past z^2/5
// are summed in FP32 (they are below 2^-17 of the total).
__device__ __forceinline__ df32 df_normal_radius(float u) {
  const int bits = __float_as_int(u);
  const int e = (bits - __float_as_int(0.70710677f)) >> 23;
  const float m = __int_as_float(bits - (e << 23));
  const float f = __fsub_rn(m, 1.f);        // exact
  const df32 g = fast_two_sum(m > 1.f ? m : 1.f, m > 1.f ? 1.f : m);
  const float r = __frcp_rn(g.h);
  df32 s;
  s.h = __fmul_rn(f, r);
  s.l = __fmul_rn(__fmaf_rn(-s.h, g.l, __fmaf_rn(-s.h, g.h, f)), r);
  const df32 z = df_mul(s, s);
  float q = 1.f / 17.f;
  q = __fmaf_rn(q, z.h, 1.f / 15.f);
  q = __fmaf_rn(q, z.h, 1.f / 13.f);
  q = __fmaf_rn(q, z.h, 1.f / 11.f);
  q = __fmaf_rn(q, z.h, 1.f / 9.f);
  q = __fmaf_rn(q, z.h, 1.f / 7.f);
  df32 p = two_prod(z.h, q);
  p.l = __fmaf_rn(z.l, q, p.l);
  p = df_add_small(df_const(1.0 / 5.0), p);
  p = df_add_small(df_const(1.0 / 3.0), df_mul(z, p));
  const df32 t = df_mul(z, p);
  const df32 lm = df_add_small(s, df_mul(s, t));  // atanh s
  // e ln 2 with the leading part of ln 2 in 15 bits, so that its product with e is exact
  constexpr float ln2_h = 0.693145751953125f;
  constexpr float ln2_l = (float)(0.693147180559945309417 - (double)ln2_h);
  const df32 a = two_sum(__fmul_rn((float)e, ln2_h), __fmul_rn(2.f, lm.h));
  const float lo = __fadd_rn(a.l, __fmaf_rn((float)e, ln2_l, __fmul_rn(2.f, lm.l)));
  const df32 x = fast_two_sum(__fmul_rn(-2.f, a.h), __fmul_rn(-2.f, lo));
  const float r0 = __fsqrt_rn(x.h);
  const float res = __fadd_rn(__fmaf_rn(-r0, r0, x.h), x.l);
  return {r0, __fmul_rn(res, __frcp_rn(__fadd_rn(r0, r0)))};
}

// cos(2 pi u) and sin(2 pi u) for a u in (0, 1) with 24 bits.  The argument is reduced exactly to
// t in [-1/4, 1/4] half turns; x = pi t, y = x^2 <= 0.617, and the first four coefficients of each
// series are applied in two floats, the rest in FP32.
__device__ __forceinline__ void df_cos_sin_turn(float u, df32 &c, df32 &s) {
  const float v = __fadd_rn(u, u);
  const float jf = rintf(__fadd_rn(v, v));
  const int j = (int)jf;
  const float t = __fmaf_rn(-0.5f, jf, v);  // exact
  constexpr double pi = 3.14159265358979323846;
  constexpr float pi_h = (float)pi, pi_l = (float)(pi - (double)pi_h);
  df32 x = two_prod(t, pi_h);
  x.l = __fmaf_rn(t, pi_l, x.l);
  const df32 y = df_mul(x, x);
  auto tail = [&](double c, float t) {  // c + y t
    df32 p = two_prod(y.h, t);
    p.l = __fmaf_rn(y.l, t, p.l);
    return df_add_small(df_const(c), p);
  };
  auto term = [&](double c, df32 p) { return df_add_small(df_const(c), df_mul(y, p)); };
  float ts = 1.f / 6227020800.f;
  ts = __fmaf_rn(ts, y.h, -1.f / 39916800.f);
  ts = __fmaf_rn(ts, y.h, 1.f / 362880.f);
  float tc = -1.f / 87178291200.f;
  tc = __fmaf_rn(tc, y.h, 1.f / 479001600.f);
  tc = __fmaf_rn(tc, y.h, -1.f / 3628800.f);
  tc = __fmaf_rn(tc, y.h, 1.f / 40320.f);
  const df32 ps = term(-1.0 / 6.0, term(1.0 / 120.0, tail(-1.0 / 5040.0, ts)));
  const df32 pc = term(-0.5, term(1.0 / 24.0, tail(-1.0 / 720.0, tc)));
  const df32 sn = df_add_small(x, df_mul(x, df_mul(y, ps)));
  const df32 cs = df_add_small({1.f, 0.f}, df_mul(y, pc));
  // rotate by j quarter turns
  const bool odd = j & 1, neg_c = (j + 1) & 2, neg_s = j & 2;
  c = odd ? sn : cs;
  s = odd ? cs : sn;
  if (neg_c) c = {-c.h, -c.l};
  if (neg_s) s = {-s.h, -s.l};
}

}  // namespace mg
