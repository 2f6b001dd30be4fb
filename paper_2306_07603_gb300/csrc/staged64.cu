// Staged FP64 IFDLBM step: three launches per time step, no recomputation.
//
//   k_collide64  every node: Step (2) (moments, f^eq, power-law lam) and Step
//                (3), f-hat^+ (Eq. 2.15) and f-bar^+ (Eq. 2.16)
//   k_half64     Step (4): half step f-bar(t+dt/2) (Eq. 3.7), its moments and
//                f(t+dt/2) (Eq. 2.17); wall nodes by extrapolation
//   k_full64     Step (5): f-hat(t+dt) (Eq. 3.6); wall nodes (Step 6); residual
//                partials of Eq. (2.19) and Eq. (5.1)
//
// Bound: the FP64 pipe (step64.cuh), busy 81-85 % of the kernels' time. A node's
// step takes 102 + 139 + 76 FP64 instructions in the three kernels (105 + 139 + 128
// where the residual is formed), which is why the intermediate planes are kept
// (they stay in L2 for a cavity sweep) rather than recomputed. Ten 257^2 cavities:
// 391 us a step, 333 at the pipe's rate (133 + 173 + 95 from a cold cache, one
// launch after another). The form before, tiles of 32 x 8 nodes with both upwind
// sides evaluated, the power by log2 and exp2 and the wall rule in every edge
// warp, took 218 + 356 + 259 instructions and 1211 us. One 65^2 cavity: 20.3 us a
// step against 94; there the three launches and the latency of a warp count, so
// each kernel starts while the one before it ends (launch.cuh) and forms what the
// step does not change before waiting for it, and blocks are one warp (34.1 us
// before these three).
//
// Wall nodes follow the rule of the FP32 staged kernels (staged.cu): a wall
// node (i, j) takes the node (clamp(i, 1, nx-2), clamp(j, 1, ny-2)), which its
// thread evaluates again.
#include <cstdint>

#include "d2q9.cuh"
#include "implicit.cuh"
#include "internal.h"
#include "launch.cuh"
#include "reduce.cuh"
#include "step64.cuh"

namespace ifd {

namespace {

// Threads per block NT: 128, or 32 on small batches. The registers follow: a
// small batch has too few warps for its latencies to hide behind others, so
// its kernels may use up to 144 registers to have more loads in flight (14
// blocks of a warp still fit on an SM); four blocks of 128 threads take 128.
template <int NT>
constexpr int MIN_BLOCKS = NT == 32 ? 14 : 4;

template <int NT>
__global__ void __launch_bounds__(NT, MIN_BLOCKS<NT>) k_collide64(StepArgs a) {
  const Node64 r = node_of<NT>(a.blk_cav, a.cav);
  const CavDev &cv = a.cav[r.cav];
  const int64_t node = int64_t(r.j) * cv.pitch + r.i, plane = cv.plane, b9 = 9 * cv.off + node;
  const double dt = cv.dt;
  previous_done();
  dependents_may_start();
  if (!r.valid) return;
  const double *gin = (const double *)a.g_in + b9;
  const double lam_prev = ((const double *)a.lam_in)[cv.off + node];
  double g[9], d[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) g[q] = gin[q * plane];
  const Mom64 m = moments64(g);                  // Eqs. (2.10)-(2.11)
  equilibrium64(m, d);                           // Eq. (2.8)
#pragma unroll
  for (int q = 0; q < 9; ++q) d[q] -= g[q];      // f^eq - f-hat
  const double diag = (d[5] + d[6]) + (d[7] + d[8]);
  const double pxx = (d[1] + d[3]) + diag, pyy = (d[2] + d[4]) + diag;
  const double pxy = (d[5] - d[6]) + (d[7] - d[8]);
  const double pp = fma(pxx, pxx, fma(pyy, pyy, (pxy + pxy) * pxy));
  double lam;
  if (cv.implicit) {
    lam = lambda_implicit(2.0 * cv.c * cv.c * sqrt(0.5 * pp) * cv.inv_cs2, lam_prev, cv, a.powtab,
                          a.powt + int64_t(r.cav) * POWT_SIZE);
  } else {
    // Eqs. (2.12)-(2.13) with f = f(f-hat, lam_prev) of Eq. (2.18): |gamma-dot|^2 =
    // 2 D:D = k^2 pp c^4 / 2 with k = -2 / ((2 lam_prev + dt) c_s^2)
    const double k = recip(fma(2.0, lam_prev, dt));
    lam = power_law64(cv.strain2 * pp * (k * k), cv, a.powtab, a.powt + int64_t(r.cav) * POWT_SIZE);
  }
  ((double *)a.lam_out)[cv.off + node] = lam;    // lam(t), also next lam_prev
  const double i2 = recip(fma(2.0, lam, dt));
  const double bp = 2.0 * dt * i2;   // Eq. (2.15): (2 lam - dt)/(2 lam + dt) = 1 - bp
  const double bb = 0.75 * bp;       // Eq. (2.16): (4 lam - dt)/(4 lam + 2 dt) = 1 - bb
  double *fp = (double *)a.fp + b9, *fb = (double *)a.fb + b9;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    fp[q * plane] = fma(bp, d[q], g[q]);
    fb[q * plane] = fma(bb, d[q], g[q]);
  }
  if (a.want_residual) {
    double *m0 = a.m0 + 3 * cv.off + node;
    m0[0] = cv.c * m.x;
    m0[plane] = cv.c * m.y;
    m0[2 * plane] = cv.cs2 * m.p;
  }
}

// out = base - scale A(F) of every moving population at an interior node: base
// and F point to the node in plane 0 of their sets (SAME: base = F).
template <bool GEN, bool SAME>
__device__ __forceinline__ void advect_all64(const Stencil64<GEN> &st, int64_t plane,
                                             const double *base, const double *F, double out[9]) {
  auto one = [&](auto qc) {
    constexpr int q = decltype(qc)::value;
    const double *Fq = F + q * plane;
    const double f0 = Fq[0];
    out[q] = advect64<q, GEN>(SAME ? f0 : base[q * plane], Fq, f0, st);
  };
  one(Const<1>()), one(Const<2>()), one(Const<3>()), one(Const<4>());
  one(Const<5>()), one(Const<6>()), one(Const<7>()), one(Const<8>());
}

// f(t + dt/2) at an interior node: the half step of Eq. (3.7) from f-bar^+ (fb,
// at the node), then Eq. (2.17) with the node's lambda(t). Returns its moments,
// which are those of f-bar (Eq. 2.17 keeps u and P).
template <bool GEN>
__device__ __forceinline__ Mom64 half_at64(const Stencil64<GEN> &st, int64_t plane, double dt,
                                           const double *fb, const double *lam_at, double f[9]) {
  const double lam = *lam_at;
  f[0] = fb[0];
  advect_all64<GEN, true>(st, plane, fb, fb, f);
  const Mom64 m = moments64(f);                        // Eqs. (2.10)-(2.11) on f-bar
  double geq[9];
  equilibrium64(m, geq);
  const double bh = dt * recip(fma(4.0, lam, dt));     // Eq. (2.17): 4 lam/(4 lam + dt) = 1 - bh
#pragma unroll
  for (int q = 0; q < 9; ++q) f[q] = fma(bh, geq[q] - f[q], f[q]);
  return m;
}

// f-hat(t + dt) at an interior node: the full step of Eq. (3.6).
template <bool GEN>
__device__ __forceinline__ void full_at64(const Stencil64<GEN> &st, int64_t plane,
                                          const double *fp, const double *fh, double f[9]) {
  f[0] = fp[0];
  advect_all64<GEN, false>(st, plane, fp, fh, f);
}

// Wall node (i, j) from F and its moments at the inner neighbour; F2 the next
// node's populations where the wall pressure is extrapolated at first order
// (P_b = 2 P - P_2). The lid nodes 0 < i < nx-1 move with the lid.
__device__ __forceinline__ void wall_node64(double F[9], const Mom64 &m, double dp, int i, int j,
                                            const CavDev &cv) {
  const bool lid = j == cv.ny - 1 && i > 0 && i < cv.nx - 1;
  const double ic = 1.0 / cv.c;
  wall64(F, m, lid ? cv.lid_ux * ic : 0.0, lid ? cv.lid_uy * ic : 0.0, dp);
}

template <int NT, bool GEN>
__global__ void __launch_bounds__(NT, MIN_BLOCKS<NT>) k_half64(StepArgs a) {
  const Node64 r = node_of<NT>(a.blk_cav, a.cav);
  const CavDev &cv = a.cav[r.cav];
  const int ii = min(max(r.i, 1), cv.nx - 2), jj = min(max(r.j, 1), cv.ny - 2);
  const Stencil64<GEN> st = stencil64<GEN>(cv, a.geo, 0, ii, jj);
  const int64_t plane = cv.plane, off = cv.off;
  const double dt = cv.dt;
  previous_done();
  dependents_may_start();
  if (!r.valid) return;
  const double *fb = (const double *)a.fb + 9 * off, *lam = (const double *)a.lam_out + off;
  const int64_t node = int64_t(jj) * st.pitch + ii;
  double f[9];
  const Mom64 m = half_at64<GEN>(st, plane, dt, fb + node, lam + node, f);
  if (r.wall) {
    double dp = 0.0;
    if (cv.wallp) {
      const int i2 = 2 * ii - r.i, j2 = 2 * jj - r.j;
      const int64_t n2 = int64_t(j2) * st.pitch + i2;
      double f2[9];
      dp = m.p - half_at64<GEN>(stencil64<GEN>(cv, a.geo, 0, i2, j2), plane, dt, fb + n2, lam + n2,
                                f2).p;
    }
    wall_node64(f, m, dp, r.i, r.j, cv);
  }
  double *fh = (double *)a.fh + 9 * off + int64_t(r.j) * st.pitch + r.i;
#pragma unroll
  for (int q = 0; q < 9; ++q) fh[q * plane] = f[q];
}

template <int NT, bool GEN>
__global__ void __launch_bounds__(NT, MIN_BLOCKS<NT>) k_full64(StepArgs a) {
  const Node64 r = node_of<NT>(a.blk_cav, a.cav);
  const CavDev &cv = a.cav[r.cav];
  const int ii = min(max(r.i, 1), cv.nx - 2), jj = min(max(r.j, 1), cv.ny - 2);
  const Stencil64<GEN> st = stencil64<GEN>(cv, a.geo, 1, ii, jj);
  const int64_t plane = cv.plane;
  previous_done();
  dependents_may_start();
  Partial p = {0, 0, 0, 0, 0, 0, 0};
  if (r.valid) {
    const double *fp = (const double *)a.fp + 9 * cv.off, *fh = (const double *)a.fh + 9 * cv.off;
    const int64_t node = int64_t(jj) * st.pitch + ii;
    double f[9];
    full_at64<GEN>(st, plane, fp + node, fh + node, f);
    if (r.wall) {
      const Mom64 m = moments64(f);
      double dp = 0.0;
      if (cv.wallp) {
        const int i2 = 2 * ii - r.i, j2 = 2 * jj - r.j;
        const int64_t n2 = int64_t(j2) * st.pitch + i2;
        double f2[9];
        full_at64<GEN>(stencil64<GEN>(cv, a.geo, 1, i2, j2), plane, fp + n2, fh + n2, f2);
        dp = m.p - moments64(f2).p;
      }
      wall_node64(f, m, dp, r.i, r.j, cv);
    }
    const int64_t me = int64_t(r.j) * st.pitch + r.i;
    double *out = (double *)a.g_out + 9 * cv.off + me;
#pragma unroll
    for (int q = 0; q < 9; ++q) out[q * plane] = f[q];
    // a velocity can be non-finite only if a population is, or is above 2^1015:
    // the exponents are looked at first, the velocity formed only then
    int top = 0;
#pragma unroll
    for (int q = 1; q < 9; ++q) top = max(top, __double2hiint(f[q]) & 0x7FFFFFFF);
    if (top >= ((1015 + 1023) << 20) || a.want_residual) {
      const Mom64 m = moments64(f);
      const double u1 = cv.c * m.x, v1 = cv.c * m.y;
      if (!(isfinite(u1) && isfinite(v1))) atomicOr(a.status, 1u);
      if (a.want_residual) {
        const double *m0 = a.m0 + 3 * cv.off + me;
        const double P1 = cv.cs2 * m.p;
        const double du = u1 - m0[0], dv = v1 - m0[plane], dP = P1 - m0[2 * plane];
        p.du2 = du * du + dv * dv;
        p.u2 = u1 * u1 + v1 * v1;
        p.dP2 = dP * dP;
        const double Pfull = P1 + a.pref[r.cav];  // P of the deviations plus their reference
        p.P2 = Pfull * Pfull;
        p.du2max = p.du2;
        p.u2max = p.u2;
        const double wx = ((r.i == 0 || r.i == cv.nx - 1) ? 0.5 : 1.0) * cv.dxi;
        const double wy = ((r.j == 0 || r.j == cv.ny - 1) ? 0.5 : 1.0) * cv.deta;
        const double J = GEN ? a.geo.gmet[7 * cv.off + 6 * plane + me]
                             : a.geo.xxi[cv.goff + r.j] * cv.H;
        p.ek = 0.5 * wx * wy * J * p.u2;          // Eq. (5.1)
      }
    }
  }
  if (a.want_residual) block_partial<NT / 32>(p, a.part, blockIdx.x);
}

}  // namespace

void launch_collide64(const StepArgs &a, int nblk, int nt, cudaStream_t s) {
  launch_after(nt == 32 ? k_collide64<32> : k_collide64<128>, nblk, nt, 0, s, a);
}
void launch_half64(const StepArgs &a, int nblk, int nt, cudaStream_t s) {
  if (a.geo.gmet)
    launch_after(nt == 32 ? k_half64<32, true> : k_half64<128, true>, nblk, nt, 0, s, a);
  else
    launch_after(nt == 32 ? k_half64<32, false> : k_half64<128, false>, nblk, nt, 0, s, a);
}
void launch_full64(const StepArgs &a, int nblk, int nt, cudaStream_t s) {
  if (a.geo.gmet)
    launch_after(nt == 32 ? k_full64<32, true> : k_full64<128, true>, nblk, nt, 0, s, a);
  else
    launch_after(nt == 32 ? k_full64<32, false> : k_full64<128, false>, nblk, nt, 0, s, a);
}

}  // namespace ifd
