// kf_df.cuh -- double-float arithmetic on the FP32 pipe, for the mixed kernel
// and for the logarithm of the FP64 kernels.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "kf_device.cuh"

namespace kfgb {
namespace dev {

// ---- double-float ("df") values: an unevaluated sum hi + lo of two floats
// with |lo| <= ulp(hi) / 2, about 48 significant bits.  Error-free
// transformations: Knuth's TwoSum, Dekker's Fast2Sum and the exact product
// from one FMA; sums and products of df values as in Dekker (1971), dot
// products as Dot2 of Ogita, Rump and Oishi (2005).  The _rn intrinsics keep
// the compiler from contracting or reassociating these steps.
struct DF {
  float hi, lo;
};
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
// exact for |a| >= |b| or a = 0
__device__ __forceinline__ DF fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DF two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return {p, __fmaf_rn(a, b, -p)};
}
// x + f (the final TwoSum keeps the pair normalised under cancellation)
__device__ __forceinline__ DF df_add_f(DF x, float f) {
  const DF s = two_sum(x.hi, f);
  return two_sum(s.hi, __fadd_rn(s.lo, x.lo));
}
// x + y, with the low parts summed exactly as well
__device__ __forceinline__ DF df_add(DF x, DF y) {
  const DF s = two_sum(x.hi, y.hi);
  const DF t = two_sum(x.lo, y.lo);
  const DF u = two_sum(s.hi, __fadd_rn(s.lo, t.hi));
  return two_sum(u.hi, __fadd_rn(u.lo, t.lo));
}
__device__ __forceinline__ DF df_neg(DF x) { return {-x.hi, -x.lo}; }
// x * y (the lo * lo term is below the pair's resolution)
__device__ __forceinline__ DF df_mul(DF x, DF y) {
  const DF p = two_prod(x.hi, y.hi);
  return fast_two_sum(p.hi, __fmaf_rn(x.hi, y.lo, __fmaf_rn(x.lo, y.hi, p.lo)));
}
// float value (hi + lo rounded)
__device__ __forceinline__ float df_f(DF x) { return __fadd_rn(x.hi, x.lo); }
// conversions: to FP64 exactly, from FP64 as the nearest float and the
// nearest float to the rest
__device__ __forceinline__ double df_to_d(DF x) { return f2d(x.hi) + f2d(x.lo); }
__device__ __forceinline__ DF df_from_d(double v) {
  const float h = d2f(v);
  return {h, d2f(v - f2d(h))};
}
// from FP64 without an FP64 instruction: hi is the value cut to 24 bits, lo
// the float of the 29 bits cut off (integer pipe), so hi + lo is within 2^-48
// of the value; below 2^-96 the rest is dropped.  Zero, Inf and NaN as d2f.
__device__ __forceinline__ DF df_cut(double v) {
  const uint32_t w = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
  const uint32_t ah = w & 0x7fffffffu, sg = w & 0x80000000u;
  if (ah < 0x38100000u || ah >= 0x47e00000u) return {d2f(v), 0.0f};
  const uint32_t r = __funnelshift_l(l, ah, 3) + 0x40000000u;  // see d2f
  const float hi = __uint_as_float(r | sg);
  const uint32_t e = r >> 23;  // biased exponent of hi
  if (e < 31u) return {hi, 0.0f};
  // rest = (l mod 2^29) 2^-29 ulp(hi), ulp(hi) = 2^(e - 150)
  const float ulp = __uint_as_float(((e - 23u) << 23) | sg);
  return fast_two_sum(hi, (float)(l & 0x1fffffffu) * 0x1p-29f * ulp);
}
// acc - a * b, the sum left unnormalised: a chain of these ends with df_norm
__device__ __forceinline__ DF df_fnma_acc(DF acc, DF a, DF b) {
  const DF p = two_prod(a.hi, b.hi);
  const float c = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
  const DF s = two_sum(acc.hi, -p.hi);
  return {s.hi, __fadd_rn(s.lo, __fsub_rn(acc.lo, c))};
}
__device__ __forceinline__ DF df_norm(DF x) { return fast_two_sum(x.hi, x.lo); }
__device__ __forceinline__ DF df_fnma(DF acc, DF a, DF b) { return df_norm(df_fnma_acc(acc, a, b)); }
// x + a * b + f
__device__ __forceinline__ DF df_muladd(DF x, DF a, DF b, float f) {
  const DF p = two_prod(a.hi, b.hi);
  const float c = __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo));
  const DF s = two_sum(x.hi, p.hi);
  const DF t = two_sum(s.hi, f);
  return two_sum(t.hi, __fadd_rn(t.lo, __fadd_rn(s.lo, __fadd_rn(x.lo, c))));
}
// 1 / x: a float reciprocal and one Newton step (relative error about 2^-44)
__device__ __forceinline__ DF df_rcp(DF x) {
  const float y = __frcp_rn(x.hi);
  const DF p = two_prod(x.hi, y);
  const float e = __fmaf_rn(-x.lo, y, __fsub_rn(__fsub_rn(1.0f, p.hi), p.lo));
  return fast_two_sum(y, __fmul_rn(y, e));
}

// The library's logarithm, out of line (arguments outside the fast range).
static __device__ __noinline__ double log_call(double x) { return log(x); }

// Natural logarithm of a positive normal double for 10 FP64 instructions where
// the library's takes some 25: x = 2^e m with m in [0.7, 1.42),
// z = (m - 1) / (m + 1),
//   log m = 2 z + z w (2/3 + w (2/5 + w (2/7 + w (2/9 + w t(w))))),  w = z^2,
// the series of 2 atanh(z): z itself in FP64, the rest (at most 1 % of it) in
// pairs of floats on the FP32 pipe and its last terms t (2/11 ... 2/21) in
// float; e ln 2 is added in FP64.  |z| <= 0.172: the terms left out are below
// 1e-18, t's rounding and that of w t 2e-16 of log m; z's three roundings and
// the pairs' (2^-46 of the 1 %) bring it to at most 6e-16 of the logarithm.
// With 2/9 in t as well it is 3.7e-15; with 2/11 a full pair too, 5e-16 for
// 0.4 % of the fit with energy loss (three logarithms a state).  Against the
// library's function: FP64 fit of 100k tracks of 30 planes 5.39 -> 5.29 ms,
// energy loss at 50k tracks 2.45 -> 2.31 ms.
__device__ __forceinline__ double log_df(double x) {
  const int h = __double2hiint(x);
  if (h < 0x00100000 || h >= 0x7ff00000) return log_call(x);
  const bool up = (h & 0xfffff) > 0x6a09e;  // m > sqrt(2): halve it
  const int e = (h >> 20) - 1023 + (up ? 1 : 0);
  const double m = __hiloint2double((h & 0xfffff) | (up ? 0x3fe00000 : 0x3ff00000), __double2loint(x));
  const double zd = (m - 1.0) * rcp_nr<2>(m + 1.0);
  const DF z = df_cut(zd);
  const DF w = df_mul(z, z);
  const float f = w.hi;
  float t = fmaf(f, 2.0f / 21.0f, 2.0f / 19.0f);
  t = fmaf(f, t, 2.0f / 17.0f);
  t = fmaf(f, t, 2.0f / 15.0f);
  t = fmaf(f, t, 2.0f / 13.0f);
  t = fmaf(f, t, 2.0f / 11.0f);
  // c + w * a with a constant pair c above the product
  auto level = [&](double c, DF a) {
    const float ch = (float)c, cl = (float)(c - (double)(float)c);
    const DF b = df_mul(w, a);
    const DF s = fast_two_sum(ch, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(b.lo, cl)));
  };
  // 2/9 + w t: the product's rounding is 1e-9 of the sum
  constexpr float c9 = (float)(2.0 / 9.0), c9l = (float)(2.0 / 9.0 - (double)c9);
  DF a = fast_two_sum(c9, __fmul_rn(f, t));
  a.lo = __fadd_rn(a.lo, c9l);
  a = level(2.0 / 7.0, a);
  a = level(2.0 / 5.0, a);
  a = level(2.0 / 3.0, a);
  const DF c = df_mul(df_mul(z, w), a);
  // e as a double through the low word of 2^52 + 2^31 + e
  const double ed = __hiloint2double(0x43300000, e ^ (int)0x80000000) - 4503601774854144.0;
  return fma(ed, 0.693147180559945309, fma(2.0, zd, df_to_d(c)));
}

}  // namespace dev
}  // namespace kfgb
