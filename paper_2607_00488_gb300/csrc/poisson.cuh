// Per-bin Poisson deviance terms of -2 ln L (eq. logL).
//
// With C = 2 sum_j [n_j - n_j ln n_j + lnGamma(n_j + 1)] (theta independent,
// computed once per data set in FP64),
//   -2 ln L = C + 2 sum_j t_j,   t_j = mu_j - n_j + n_j ln(n_j / mu_j)
// which is eq. logL term by term (0 ln 0 = 0).  t_j >= 0 and is small where
// the model fits, so summing t instead of mu - n ln mu avoids the large
// cancelling magnitudes of the direct form.
#pragma once

#include <cuda_runtime.h>

#include "dfloat.cuh"

namespace srw {

// FP64 term (single-point path).  mu < 0, or mu == 0 with n > 0, gives +inf.
__device__ __forceinline__ double poisson_term_f64(double mu, double n) {
  if (mu < 0.0) return __longlong_as_double(0x7ff0000000000000LL);
  if (n == 0.0) return mu;
  if (mu == 0.0) return __longlong_as_double(0x7ff0000000000000LL);
  return mu - n + n * log(n / mu);
}

// The same term in double-float on the FP32 pipes, within 1.4e-13 (n + mu), 1e-14
// (n + mu) rms, of the exact one (each operation emulated on 16,000 pairs).  With k
// the power of two that brings n' = n 2^-k within a factor ~sqrt(2) of mu and
// v = (n' - mu)/(n' + mu),
//   ln(n/mu) = k ln 2 + 2 atanh(v) = k ln 2 + 2 v (1 + v^2 (1/3 + v^2 (1/5 + v^2 q(v^2)))),
// |v| < 0.18; q in FP32 (its part of the bracket is below 2e-4, so its rounding
// is below 1e-11 v^3), the rest in double-float (with 1/5 in FP32 as well
// 5e-12 (n + mu); a 4096-point solar-set scan 1272 us, so 1277).  False, and no term,
// outside 1e-30 < mu, n with n / mu within 2^+-96 (n = 0 with mu >= 0 is
// inside), where n', mu and their low parts are normal FP32 numbers; NaN and
// infinities are outside as well.  The caller then takes poisson_term_f64.
__device__ __forceinline__ bool poisson_term_df(dfloat mu, dfloat n, dfloat* t) {
  if (n.hi == 0.f && mu.hi >= 0.f) {
    *t = mu;
    return true;
  }
  const float r = __fdividef(n.hi, mu.hi) * 1.41421356f;
  const int k = (__float_as_int(r) >> 23) - 127;  // r > 0: n / mu in 2^k [0.707, 1.415)
  if (!(mu.hi > 1e-30f) || !(n.hi > 1e-30f) || abs(k) > 96) return false;
  const float p2 = __int_as_float((127 - k) << 23);
  const dfloat ns = {n.hi * p2, n.lo * p2};
  const dfloat d = df_add(ns, dfloat{-mu.hi, -mu.lo}), s = df_add(ns, mu);
  const float q0 = __fdividef(d.hi, s.hi);  // v to FP32, then one correction step
  const dfloat q0s = two_prod(q0, s.hi);
  const dfloat rem = df_add(d, dfloat{-q0s.hi, -fmaf(q0, s.lo, q0s.lo)});
  const dfloat v = fast_two_sum(q0, __fdividef(rem.hi, s.hi));
  const dfloat v2 = df_mul(v, v);
  float q = fmaf(v2.hi, 1.f / 19.f, 1.f / 17.f);
  q = fmaf(v2.hi, q, 1.f / 15.f);
  q = fmaf(v2.hi, q, 1.f / 13.f);
  q = fmaf(v2.hi, q, 1.f / 11.f);
  q = fmaf(v2.hi, q, 1.f / 9.f);
  q = fmaf(v2.hi, q, 1.f / 7.f);
  const dfloat third = {0.33333334f, -9.9341072e-9f}, fifth = {0.2f, -2.9802323e-9f};
  const dfloat w = df_mul(v2, df_add(third, df_mul(v2, df_add(fifth, q * v2.hi))));
  dfloat l = df_add(v, df_mul(v, w));
  l = {2.f * l.hi, 2.f * l.lo};
  const float kf = (float)k;
  const dfloat ln2 = {0.69314718f, -1.9046542e-9f};
  dfloat kl = two_prod(kf, ln2.hi);
  kl = fast_two_sum(kl.hi, fmaf(kf, ln2.lo, kl.lo));
  l = df_add(kl, l);
  *t = df_add(df_add(mu, dfloat{-n.hi, -n.lo}), df_mul(n, l));
  return true;
}

// a / b as the product with PTX's approximate reciprocal (rcp.approx.ftz: 1 ulp,
// a subnormal b counts as 0), for b that is 0, infinite, NaN or at least 1e-30 in
// magnitude.
__device__ __forceinline__ float reciprocal(float b) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
  return r;
}
__device__ __forceinline__ float quotient(float a, float b) { return __fmul_rn(a, reciprocal(b)); }

// FP32 term of the tensor-core epilogue, branch-free and without per-element
// special cases.  With v = (n - mu)/(n + mu), ln(n/mu) = 2 atanh(v), hence
//   t = (n - mu) v + 2 n (v^3/3 + v^5/5 + v^7/7 + v^9/9 + ...)
// which has no cancellation; for |v| < 0.1 the truncation after v^9 is below
// 1e-10 relative.  Larger |v| uses the direct form, whose cancellation is
// then at most a factor ~10.  Both forms are evaluated and selected, so lanes
// holding different parameter points never diverge; the quotients use the
// fast division (at most 2 ulp).  The bin constants carry n = 0 for masked
// bins (their term is then finite and the caller multiplies it by the 0/1
// mask).  The log argument is floored at 1e-30: for n = 0 the term is
// 0 * ln(1e-30) = 0, so t = mu (mu = 0 included, where n / mu is NaN and the
// floor applies); mu = 0 with n > 0 gives +inf through ln(inf).  mu < 0 is
// left to the caller (it tracks the smallest mu of the active bins).
// It is formed from dm = mu - n (and n), for callers that form mu - n
// directly: an FP32 mu of 1e5 counts carries an absolute rounding error of
// ~6e-3, while mu - n near the data is a few hundred, so its FP32 value is
// ~1e3 times more precise and the series branch then loses nothing to it.
// The log branch (far from the data) takes mu - n of the same rounded mu that
// enters the logarithm: then mu's rounding error e enters t only as
// (1 - n/mu) e, as in the exact expression (dt/dmu = 1 - n/mu); with the
// unrounded dm it would enter as -(n/mu) e, about e itself.
__device__ __forceinline__ float poisson_term_f32_dm(float dm, float n) {
  const float mu = n + dm, s = n + mu;
  const float v = __fdividef(-dm, s);
  const float v2 = v * v;
  float p = fmaf(v2, 1.f / 9.f, 1.f / 7.f);
  p = fmaf(v2, p, 1.f / 5.f);
  p = fmaf(v2, p, 1.f / 3.f);
  const float ts = fmaf(-dm, v, 2.f * n * v * v2 * p);
  const float tl = fmaf(n, logf(fmaxf(__fdividef(n, mu), 1e-30f)), mu - n);
  return fabsf(v) < 0.1f ? ts : tl;
}

}  // namespace srw
