// FP64 device helpers of the staged step (staged64.cu) and of its adjoint (adjoint.cu).
//
// GB300 issues one FP64 warp instruction per SM sub-partition every 64
// cycles, so these kernels are bound by the number of FP64 instructions and
// by the warps that execute them, not by bytes or by any other instruction.
// Hence, throughout:
//  * conversions, comparisons, clamps and side selections, which would take an
//    FP64 slot each (F2F, DSETP), are done on the bits with integer
//    instructions, which are free beside it;
//  * reciprocals take three FP64 instructions after an FP32 seed (recip);
//  * threads map to nodes by a linear index over the interior and then over
//    the walls (node_of), so that no warp of a ragged row runs with a few
//    lanes (65 columns in tiles of 32 leave 32 % of the lanes idle, 257 11 %)
//    and the wall rule runs in warps of its own.
#pragma once
#include <cuda_runtime.h>

#include "fastpow.cuh"
#include "internal.h"

namespace ifd {

// An integer as a type (compile-time population index).
template <int N>
struct Const {
  static constexpr int value = N;
};

// The node of this thread: blocks [blk0, blk0 + nblk_in) of a cavity take its
// interior nodes row by row, the blocks after them its wall nodes (bottom row,
// lid row, then the two side columns in turn).
struct Node64 {
  int cav, i, j;
  bool valid, wall;  // wall is uniform over the block
};
template <int NT>
__device__ __forceinline__ Node64 node_of(const int *blk_cav, const CavDev *cavs) {
  Node64 r;
  const int b = blockIdx.x;
  r.cav = blk_cav[b];
  const CavDev &cv = cavs[r.cav];
  const int lb = b - cv.blk0;
  r.wall = lb >= cv.nblk_in;
  if (!r.wall) {
    const unsigned n = unsigned(lb) * NT + threadIdx.x;
    const unsigned w = unsigned(cv.nx - 2);
    const unsigned row = n / w;
    r.valid = row < unsigned(cv.ny - 2);
    r.i = int(n - row * w) + 1;
    r.j = int(row) + 1;
  } else {
    const int n = (lb - cv.nblk_in) * NT + int(threadIdx.x);
    const int k = n - 2 * cv.nx;
    r.valid = k < 2 * (cv.ny - 2);
    if (k < 0) {
      const bool lid = n >= cv.nx;
      r.i = lid ? n - cv.nx : n;
      r.j = lid ? cv.ny - 1 : 0;
    } else {
      r.i = (k & 1) ? cv.nx - 1 : 0;
      r.j = 1 + (k >> 1);
    }
  }
  return r;
}

// float(x) truncated and double(f), on the bits (exact for a normal float;
// a zero or subnormal float gives a value below 2^-126 in magnitude).
__device__ __forceinline__ float narrow_pos(int hi, int lo) {
  return __int_as_float(((hi - (896 << 20)) << 3) | int(unsigned(lo) >> 29));
}
__device__ __forceinline__ double widen(float f) {
  const int b = __float_as_int(f);
  return __hiloint2double((b & int(0x80000000u)) | (((b & 0x7FFFFFFF) >> 3) + (896 << 20)),
                          b << 29);
}

// 1 / x within 0.5005 ulp: an FP32 reciprocal r (relative error e0 < 2^-21: 2^-23 from
// the truncated argument, 2 ulps of __fdividef) and one step of the cubic iteration
// r (1 + e + e^2), e = 1 - x r (M. Altman, "An optimum cubically convergent iterative
// method of inverting a linear bounded operator in Hilbert space", Pacific J. Math.
// 10, 1960: the geometric series of 1 / (1 - e) after e^2), whose error is e0^3, 2^-11
// ulp, before the one rounding of the last fma; e itself is exact to 2^-74. So it
// differs from the division in about one argument in 10^3, by one ulp. Arguments
// outside [2^-100, 2^100), zero, negative ones and NaN take the division.
__device__ __forceinline__ double recip(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  if (unsigned(hi - (923 << 20)) >= unsigned(200 << 20)) return 1.0 / x;
  const double r = widen(__fdividef(1.0f, narrow_pos(hi, lo)));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// Signs from the bits; +-0 is nonpositive and nonnegative.
__device__ __forceinline__ bool negative(double x) { return __double2hiint(x) < 0; }
__device__ __forceinline__ bool zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ bool nonpositive(double x) { return negative(x) || zero(x); }
__device__ __forceinline__ bool nonnegative(double x) { return !negative(x) || zero(x); }

// K/c_s^2 q^m, m = (n-1)/2, for an FP64 argument q > 0: the table-driven binomial
// form of pow_tab (fastpow.cuh) on the full FP64 fraction f of q = 2^e f. As
// there, t = f (1/c_j) - 1 carries the rounding of 1/c_j (<= 1.2e-16 absolute) and
// one of its own below 2^-62, and the tail's coefficient c3 is FP32: with the four
// roundings of the tables and products the result is within 4.5e-16 + |m| 1.2e-16 +
// |b3| 6.7e-16 + |C(m,6)| 5.6e-17, b3 = m (m-1) (m-2) / 6: 7.2e-16 for |m| <= 1
// (n <= 3), against pow_fast's 5e-16 + 2.2e-16 |m log2 q|, with 6 FP64 instructions
// instead of ~22. Beyond, b3 grows as m^3 (5e-14 at n = 20): pow_fast, as for an
// argument whose exponent is not a normal float's, which the table does not cover,
// and for a NaN.
__device__ __forceinline__ double power64(double q, const CavDev &cv, const double *powtab,
                                          const double *__restrict__ powt) {
  const int hi = __double2hiint(q), lo = __double2loint(q);
  if (unsigned(hi - (897 << 20)) >= cv.p64_n)
    return cv.Kics2 * pow_fast(q, cv.half_nm1, powtab);
  const unsigned e = (unsigned(hi) >> 20) - 896u, j = (unsigned(hi) >> 12) & 255u;
  const int fh = (hi & 0x000FFFFF) | 0x3FF00000;
  const double2 dr = __ldg(reinterpret_cast<const double2 *>(powt) + j);
  const double t = fma(__hiloint2double(fh, lo), dr.y, -1.0);
  const float cj = __uint_as_float(0x3F804000u | (j << 15));
  const float tf = __fdividef(narrow_pos(fh, lo) - cj, cj);
  const float c3 = fmaf(tf, fmaf(tf, cv.pb5, cv.pb4), cv.pb3);
  const double w = fma(t, fma(t, widen(c3), cv.pb2), cv.half_nm1);
  const double P = __ldg(powt + 512 + e) * dr.x;
  return fma(P, t * w, P);
}
// The power law of Eq. (1.4), K/c_s^2 max(q, gmin2)^m (a NaN is clamped).
__device__ __forceinline__ double power_law64(double q, const CavDev &cv, const double *powtab,
                                              const double *__restrict__ powt) {
  const long long b = __double_as_longlong(q);
  const bool above = b > __double_as_longlong(cv.gmin2) && b <= 0x7FF0000000000000ll;
  return power64(above ? q : cv.gmin2, cv, powtab, powt);
}

// Moments of a deviation set in lattice units: m = sum e_i g_i (u = c m) and
// p = P / c_s^2 = (9 sum_{i>0} g_i - 6 |m|^2) / 5 (Eqs. 2.10-2.11 with
// c_s^2 = c^2 / 3), in which the equilibrium does not contain c.
struct Mom64 {
  double x, y, p, xx, yy;  // m, p, m_x^2, m_y^2
};
__device__ __forceinline__ Mom64 moments64(const double g[9]) {
  Mom64 m;
  const double d57 = g[5] - g[7], d68 = g[6] - g[8];
  m.x = (g[1] - g[3]) + (d57 - d68);
  m.y = (g[2] - g[4]) + (d57 + d68);
  const double s = ((g[1] + g[3]) + (g[2] + g[4])) + ((g[5] + g[7]) + (g[6] + g[8]));
  m.xx = m.x * m.x;
  m.yy = m.y * m.y;
  m.p = fma(1.8, s, -1.2 * (m.xx + m.yy));
  return m;
}

// w-weighted polynomial of Eq. (2.8) with p, m_x, m_y, m_x^2, m_y^2 and
// (m_x +- m_y)^2 given separately: E_i + w_i 3 e_i . m,
// E_i = wbar_i p + w_i (4.5 (e_i . m)^2 - 1.5 |m|^2). 24 FP64 instructions.
__device__ __forceinline__ void poly64(double p, double x, double y, double xx, double yy,
                                       double pp, double mm, double sp, double sm, double f[9]) {
  const double m2 = xx + yy;
  const double t9 = (1.0 / 9.0) * fma(-1.5, m2, p), t36 = 0.25 * t9;
  f[0] = fma(-2.0 / 3.0, m2, (-5.0 / 9.0) * p);
  const double e1 = fma(0.5, xx, t9), e2 = fma(0.5, yy, t9);
  const double e5 = fma(0.125, pp, t36), e6 = fma(0.125, mm, t36);
  f[1] = fma(1.0 / 3.0, x, e1);
  f[3] = fma(-1.0 / 3.0, x, e1);
  f[2] = fma(1.0 / 3.0, y, e2);
  f[4] = fma(-1.0 / 3.0, y, e2);
  f[5] = fma(1.0 / 12.0, sp, e5);
  f[7] = fma(-1.0 / 12.0, sp, e5);
  f[6] = fma(1.0 / 12.0, sm, e6);
  f[8] = fma(-1.0 / 12.0, sm, e6);
}
// Designed equilibrium, Eq. (2.8), minus w_i rho0.
__device__ __forceinline__ void equilibrium64(const Mom64 &m, double geq[9]) {
  const double sp = m.x + m.y, sm = m.y - m.x;
  poly64(m.p, m.x, m.y, m.xx, m.yy, sp * sp, sm * sm, sp, sm, geq);
}

// Wall-node rule (Sec. 4), F_b = f^eq(P_b, u_w) + F - f^eq(P, u) with F and m
// those of the inner neighbour, (wx, wy) = u_w / c and dp = (P_b - P) / c_s^2
// (0 at zeroth order): the difference of the two equilibria is formed at once,
// so that the pressure terms they share are not.
__device__ __forceinline__ void wall64(double F[9], const Mom64 &m, double wx, double wy,
                                       double dp) {
  const double sp = m.x + m.y, sm = m.y - m.x, wp = wx + wy, wm = wy - wx;
  double d[9];
  poly64(dp, wx - m.x, wy - m.y, wx * wx - m.xx, wy * wy - m.yy, wp * wp - sp * sp,
         wm * wm - sm * sm, wp - sp, wm - sm, d);
#pragma unroll
  for (int q = 0; q < 9; ++q) F[q] += d[q];
}

// The pair of opposite directions that population q >= 1 belongs to: (1, 3),
// (2, 4), (5, 7), (6, 8) = 0..3, and whether it is the pair's second member.
__host__ __device__ constexpr int pair_of(int q) { return q < 5 ? (q - 1) & 1 : 2 + ((q - 5) & 1); }
__host__ __device__ constexpr bool second_of(int q) { return q == 3 || q == 4 || q == 7 || q == 8; }

// Contravariant velocities of a node, per pair of opposite directions: the
// magnitude times scale / (2 d) (scale = dt/2 or dt), and whether the pair's
// first member is advected from below (c >= 0). On the trapezoid the eta
// velocity is uniform.
template <bool GEN>
struct Speeds64 {
  double xi[4], eta[GEN ? 4 : 1];
  bool xpos[4], epos[4];
};
template <bool GEN>
__device__ __forceinline__ Speeds64<GEN> speeds64(const CavDev &cv, const Geo &geo, int stage,
                                                  int i, int j, int64_t node) {
  Speeds64<GEN> s;
  if constexpr (GEN) {
    const double *gm = geo.gmet + 7 * cv.off + node;
    const double x = cv.sxi[stage] * gm[0], y = cv.sxi[stage] * gm[cv.plane];
    const double ex_ = cv.seta[stage] * gm[2 * cv.plane], ey_ = cv.seta[stage] * gm[3 * cv.plane];
    s.xi[0] = x, s.xi[1] = y, s.xi[2] = x + y, s.xi[3] = y - x;
    s.eta[0] = ex_, s.eta[1] = ey_, s.eta[2] = ex_ + ey_, s.eta[3] = ey_ - ex_;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      s.xpos[p] = !negative(s.xi[p]);
      s.epos[p] = !negative(s.eta[p]);
      s.xi[p] = fabs(s.xi[p]);
      s.eta[p] = fabs(s.eta[p]);
    }
  } else {
    // c_xi = A (e_x - e_y x_eta / H), A = c xi_x > 0 (Eqs. 3.4, 3.8.2)
    const double A = geo.ax[stage][cv.goff + j], xe = geo.xeH[cv.goff + i];
    const double m = 1.0 - xe, p = 1.0 + xe;
    s.xi[0] = A, s.xi[1] = A * fabs(xe), s.xi[2] = A * fabs(m), s.xi[3] = A * fabs(p);
    s.xpos[0] = true, s.xpos[1] = negative(xe), s.xpos[2] = !negative(m), s.xpos[3] = negative(p);
    s.eta[0] = cv.seta_H[stage];
    s.epos[0] = s.epos[1] = s.epos[2] = s.epos[3] = true;  // e_y of the first members >= 0
  }
  return s;
}

// The mixed difference's terms (Mix64) at F with stride d (signed: the upwind
// neighbour is F[-d]), summed before any speed multiplies them: with the default
// blend, whose coefficients are short, a constant F gives exactly 0.
__device__ __forceinline__ double mix64(const double *F, int d, bool edge, const Mix64 &m,
                                        double f0) {
  const double a = F[d], b = F[-d], f = F[edge ? -d : -2 * d];
  const double kb = edge ? m.wb : m.kb, k0 = edge ? m.w0 : m.k0, kf = edge ? 0.0 : m.kf;
  return fma(kf, f, fma(k0, f0, fma(kb, b, m.ka * a)));
}

// What the stencils of a node take besides the planes: its speeds, the
// coefficients, the row pitch and the walls it is next to. None of it is
// written by a step, so a kernel forms it before the one before it is done.
template <bool GEN>
struct Stencil64 {
  Speeds64<GEN> s;
  Mix64 mix;
  int pitch;
  bool clo, chi, lo, hi;
};
template <bool GEN>
__device__ __forceinline__ Stencil64<GEN> stencil64(const CavDev &cv, const Geo &geo, int stage,
                                                    int i, int j) {
  Stencil64<GEN> st;
  st.pitch = cv.pitch;
  st.s = speeds64<GEN>(cv, geo, stage, i, j, int64_t(j) * st.pitch + i);
  st.mix = cv.mix;
  st.clo = i == 1;
  st.chi = i == cv.nx - 2;
  st.lo = j == 1;
  st.hi = j == cv.ny - 2;
  return st;
}

// base - scale (c_xi D_xi + c_eta D_eta) F_q at interior node F (Eqs. 3.6-3.7):
// 10 FP64 instructions a plane (5 where e_y = 0 on the trapezoid). The eta speed of
// the trapezoid could be in the coefficients, for 9; but four roundings at the size
// of F then take the place of one, and a constant F leaves them behind (error of g
// against extended precision, 1025^2, 2 steps: 1.42e-16 of its rms against 1.24e-16
// so and 1.28e-16 with the differences formed first, for 14 instructions).
template <int Q, bool GEN>
__device__ __forceinline__ double advect64(double base, const double *F, double f0,
                                           const Stencil64<GEN> &st) {
  constexpr int p = pair_of(Q);
  const bool xpos = st.s.xpos[p] != second_of(Q);
  double out = fma(-st.s.xi[p],
                   mix64(F, xpos ? 1 : -1, xpos ? st.clo : st.chi, st.mix, f0), base);
  if constexpr (GEN) {
    const bool epos = st.s.epos[p] != second_of(Q);
    out = fma(-st.s.eta[p],
              mix64(F, epos ? st.pitch : -st.pitch, epos ? st.lo : st.hi, st.mix, f0), out);
  } else if constexpr (Q != 1 && Q != 3) {
    constexpr bool epos = Q == 2 || Q == 5 || Q == 6;
    out = fma(-st.s.eta[0],
              mix64(F, epos ? st.pitch : -st.pitch, epos ? st.lo : st.hi, st.mix, f0), out);
  }
  return out;
}

}  // namespace ifd
