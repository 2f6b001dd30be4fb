// Solves of the implicit form of Eq. (2.14).
//
// lam = C max(a / (2 lam + dt), gamma_min)^(n-1) with C = K / c_s^2 and
// a = 2 sqrt((Pxx^2 + 2 Pxy^2 + Pyy^2) / 2) / c_s^2, Pxx.. the second moments of
// f-hat - f^eq (Eq. 2.18 at the same lam turns them into gamma-dot(lam) =
// a / (2 lam + dt)). F(lam) = lam - C max(...)^(n-1) increases strictly, so the
// root is unique: it is the clamp value lam_c = C gamma_min^(n-1) when
// gamma-dot(lam_c) <= gamma_min, and otherwise lies in [0, lam_c] (n < 1) or
// [lam_c, C (a/dt)^(n-1)] (n > 1) with gamma-dot > gamma_min.
//
// GB300 issues one FP64 warp instruction per 64 cycles and sub-partition, and an
// FP64 Newton iteration takes ~45 with the power by log2 and exp2; so the root is
// first found in FP32 with the hardware's log2 and exp2 (lambda_approx, a few
// 1e-6), and only the last correction is made in the precision of the result.
// Six 300x260 cavities in the FP32 form: 596 -> 59 us a step (with the rows per
// task of capi.cu; 543 with those alone).
#pragma once
#include <cuda_runtime.h>

#include "d2q9.cuh"
#include "fastpow.cuh"
#include "internal.h"
#include "step64.cuh"

namespace ifd {

// The root to a few 1e-6 in FP32: Newton from lam_start, kept inside the bracket
// by bisection, until a step is below 1e-4 (the next error is its square). It
// may be poor where the values leave the range of a float; its callers check.
__device__ __forceinline__ float lambda_approx(float a, float lam_start, float C, float m, float dt,
                                               float lamc) {
  auto power = [&](float g) { return C * exp2f(m * __log2f(g)); };
  float lo = m < 0.0f ? 0.0f : lamc;
  float hi = m < 0.0f ? lamc : power(__fdividef(a, dt));
  float lam = (lam_start > lo && lam_start < hi) ? lam_start : 0.5f * (lo + hi);
  for (int it = 0; it < 10; ++it) {
    const float r = __fdividef(1.0f, 2.0f * lam + dt);
    const float P = power(a * r), F = lam - P;
    if (F > 0.0f) hi = lam; else lo = lam;
    float next = lam - __fdividef(F, 1.0f + 2.0f * m * P * r);
    if (!(next >= lo && next <= hi)) next = 0.5f * (lo + hi);
    const bool done = fabsf(next - lam) <= 1e-4f * next;
    lam = next;
    if (done) break;
  }
  return lam;
}

// The root in FP64: Newton from lambda_approx (or lam_start where the values leave
// the range of a float), inside the bracket, until a step is below 4e-15 of lam
// (F = lam - P is itself a difference of nearly equal numbers, so steps much
// smaller than that are rounding): two iterations as a rule. Kept out of line so
// that the lagged path is compiled as without it.
static __device__ __noinline__ double lambda_implicit(double a, double lam_start, const CavDev &cv,
                                                      const double *powtab, const double *powt) {
  const double C = cv.Kics2, dt = cv.dt, m = cv.nm1, lamc = cv.lam0;
  if (m == 0.0) return C;
  if (a <= cv.gmin * (2.0 * lamc + dt)) return lamc;
  double lo, hi;
  if (m < 0.0) {
    lo = 0.0;
    hi = lamc;
  } else {
    lo = lamc;
    hi = C * pow_fast((a / dt) * (a / dt), cv.half_nm1, powtab);
  }
  if (cv.impl_f32 && a > 1e-25 && a < 1e25)
    lam_start = double(lambda_approx(float(a), float(lam_start), float(C), float(m), float(dt),
                                     float(lamc)));
  double lam = (lam_start > lo && lam_start < hi) ? lam_start : 0.5 * (lo + hi);
  for (int it = 0; it < 20; ++it) {
    const double r = recip(2.0 * lam + dt);
    const double g = a * r;
    const double P = power64(g * g, cv, powtab, powt);
    const double F = lam - P;
    if (F == 0.0) break;                                   // the root itself
    if (F > 0.0) hi = lam; else lo = lam;
    double next = lam - F * recip(1.0 + 2.0 * m * P * r);
    if (!(next >= lo && next <= hi)) next = 0.5 * (lo + hi);
    const bool done = fabs(next - lam) <= 4e-15 * next;
    lam = next;
    if (done) break;
  }
  return lam;
}

// Per-cavity constants of the FP32 form's solve, whose strain rate comes from an
// FP32 value G2 = (Pxx^2 + 2 Pxy^2 + Pyy^2) / 2 in units of c (a = 6 sqrt(G2)).
struct ImplPair {
  float C, m, hm, lamc, dth, dtl;  // dt as a pair of floats
  float g2c;                       // largest float G2 that is clamped
  bool use;
};
__device__ __forceinline__ ImplPair impl_pair(const CavDev &cv) {
  const float dth = float(cv.dt);
  return {float(cv.Kics2), float(cv.nm1), float(cv.half_nm1), float(cv.lam0), dth,
          float(cv.dt - double(dth)), cv.g2c_f, cv.impl_f32 != 0};
}

// The FP64 root rounded to float: lambda_approx, then one Newton step with
// x = 2 lam + dt, 1 / x, q = 36 G2 / x^2 and P = C q^m as pairs of floats, whose errors
// are 2^-43, 2^-42 and (pow_pair) 2^-39.8: F = lam - P, whose leading difference is
// exact, is known to 2^-38 lam. With D = F' = 1 + 2 m P / x, d = F / D the step and
// F'' = -4 m (m + 1) P / x^2, |F''| <= |m (m + 1)| / lam to 2e-4, the error of lam - d is
//   E = (2^-38 lam + |m (m + 1)| d^2 / (2 lam) + 2^-19 max(1, |m|) |d|) / D,
// the last term for the roundings of D, of the quotients and of d. The float is taken
// only where lam - d - E and lam - d + E round to it (pow_pair's rounding test; E is a
// few 1e-12 lam, so that one root in 10^4 is in doubt); else, and where the table does
// not cover q, the step is large, D is near zero (n < 0.02) or a low part could
// underflow, the FP64 solve decides. (Six 300x260 cavities, without this test 56.4 us
// a step, with it 58.9.)
__device__ __forceinline__ float lambda_implicit_pair(float G2, float lam_start, const ImplPair &s,
                                                      const PowPair &pw, const CavDev &cv,
                                                      const double *powtab, const double *powt) {
  if (s.use) {
    if (G2 <= s.g2c) return s.lamc;
    const float lam = lambda_approx(6.0f * sqrtf(G2), lam_start, s.C, s.m, s.dth, s.lamc);
    const float t = 2.0f * lam, xh = t + s.dth, bb = xh - t;
    const float xl = ((t - (xh - bb)) + (s.dth - bb)) + s.dtl;
    const float rh = __fdividef(1.0f, xh), rl = rh * (fmaf(-xh, rh, 1.0f) - xl * rh);
    const float sh = rh * rh, sl = fmaf(rh, rh, -sh) + 2.0f * rh * rl;
    const float Ah = 36.0f * G2, Al = fmaf(36.0f, G2, -Ah);
    const float qh = Ah * sh, ql = fmaf(Ah, sh, -qh) + (Ah * sl + Al * sh);
    if (pow_pair_covers(qh, pw) && fminf(fminf(Ah, sh), qh) >= 0x1p-80f) {
      float Ph, Pl;
      pow_pair_parts(qh, pw, Ph, Pl);
      Pl = fmaf(Ph, s.hm * __fdividef(ql, qh), Pl);    // (q_h + q_l)^m
      const float D = fmaf(2.0f * s.m * Ph, rh, 1.0f), d = __fdividef((lam - Ph) - Pl, D);
      const float ad = fabsf(d), k = 0.55f * fabsf(s.m * (s.m + 1.0f));
      const float E = __fdividef(
          fmaf(lam, 0x1p-38f, ad * fmaf(k, __fdividef(ad, lam), 0x1p-19f * fmaxf(1.0f, fabsf(s.m)))), D);
      const float r = lam - (d + E);
      if (ad <= 1e-4f * lam && D >= 0x1p-6f && r == lam - (d - E)) return r;
    }
  }
  return float(lambda_implicit(6.0 * sqrt(double(G2)), double(lam_start), cv, powtab, powt));
}

}  // namespace ifd
