// Staged IFDLBM step of the FP32 storage (staged64.cu has the FP64 one): three
// launches per time step, no recomputation; and the helper kernels of both.
//
//   k_collide  every node: Step (2) (moments, f^eq, lagged power-law lam),
//              Step (3) f-hat^+ (Eq. 2.15) and f-bar^+ (Eq. 2.16)
//   k_half     every node: Step (4) half step f-bar(t+dt/2) (Eq. 3.7), its
//              moments and f(t+dt/2) (Eq. 2.17); wall nodes by
//              non-equilibrium extrapolation from their inner neighbour
//   k_full     every node: Step (5) f-hat(t+dt) (Eq. 3.6); wall nodes by
//              non-equilibrium extrapolation (Step 6); residual partials of
//              Eq. (2.19) and Eq. (5.1)
//
// A wall node (i, j) takes its neighbour (clamp(i, 1, nx-2), clamp(j, 1,
// ny-2)): the adjacent node along the grid normal on a side, the diagonal
// node at a corner. The lid nodes 0 < i < nx-1 of row ny-1 move at (U, 0);
// every other wall node, the two top corners included, is at rest.
#include <algorithm>
#include <cstdint>

#include "d2q9.cuh"
#include "implicit.cuh"
#include "internal.h"
#include "launch.cuh"
#include "reduce.cuh"

namespace ifd {

// Relaxation time of Step (2) of the FP32 staged kernels: strain rate from f^ne
// (Eqs. 2.12-2.13, with f = f(f-hat, lam_prev) of Eq. 2.18), q = |gamma-dot|^2 =
// 2 D:D, the clamped power law mu = K max(|gamma-dot|, gamma_min)^(n-1)
// evaluated as K max(q, gamma_min^2)^((n-1)/2) (Eq. 1.4), and lam = mu / c_s^2
// (Eq. 2.14). Pxx, Pxy, Pyy are sum_i c_ia c_ib (g_i - geq_i). The strain rate
// is formed in FP32, clamped at cv.gmin2_f; the power law of Eq. (1.4)
// (pow_tab, FP64 result, error within 6e-16) and the implicit form's solve are
// FP64, as the FP32-deviation form specifies. With cv.pow32 (an opt-in) they
// are FP32 instead (pow_f32, lambda_implicit_f32; the clamp at the largest
// float not above gamma_min^2). powt: the cavity's pow_tab table.
__device__ __forceinline__ double relaxation_time(float Pxx, float Pxy, float Pyy,
                                                  float lam_prev, const CavDev &cv,
                                                  const double *powtab, const double *powt) {
  if (cv.implicit) {
    const float G2 = 0.5f * (Pxx * Pxx + 2.0f * Pxy * Pxy + Pyy * Pyy);
    if (cv.pow32)
      return double(lambda_implicit_f32(2.0f * sqrtf(G2) * float(cv.inv_cs2), lam_prev, cv));
    return lambda_implicit(2.0 * sqrt(double(G2)) * cv.inv_cs2, double(lam_prev), cv, powtab,
                           powt);
  }
  // f^ne = 2 lam_prev/(2 lam_prev + dt) (f-hat - f^eq);  S = -sum c c f^ne / (lam_prev c_s^2)
  const float k = -2.0f / ((2.0f * lam_prev + float(cv.dt)) * float(cv.cs2));
  const float Sxx = k * Pxx, Sxy = k * Pxy, Syy = k * Pyy;
  const float q2 = 0.5f * (Sxx * Sxx + 2.0f * Sxy * Sxy + Syy * Syy);
  if (cv.pow32) {
    const float q = fmaxf(q2, __double2float_rd(cv.gmin2));
    return double(float(cv.Kics2) * pow_f32(q, float(cv.half_nm1)));
  }
  return pow_tab(fmaxf(q2, cv.gmin2_f), powt, cv.half_nm1, cv.pb2, cv.pb3, cv.pb4, cv.pb5);
}

struct ReduceArgs {
  const CavDev *cav;
  const double *part;
  double *resid;
};

struct NodeRef {
  int cav, i, j;
  bool valid;
};

__device__ __forceinline__ NodeRef tile_node(const int *tile_cav, const CavDev *cavs) {
  NodeRef r;
  const int t = blockIdx.x;
  r.cav = tile_cav[t];
  const CavDev &cv = cavs[r.cav];
  const int lt = t - cv.tile0;
  r.i = (lt % cv.tiles_x) * TILE_X + threadIdx.x;
  r.j = (lt / cv.tiles_x) * TILE_Y + threadIdx.y;
  r.valid = r.i < cv.nx && r.j < cv.ny;
  return r;
}

template <class T>
__device__ __forceinline__ void load9(const T *base, int64_t plane, int64_t node, T v[9]) {
#pragma unroll
  for (int q = 0; q < 9; ++q) v[q] = base[q * plane + node];
}

template <class T>
__device__ __forceinline__ void store9(T *base, int64_t plane, int64_t node, const T v[9]) {
#pragma unroll
  for (int q = 0; q < 9; ++q) base[q * plane + node] = v[q];
}

// ---------------------------------------------------------------------------
// Step (2)-(3): collision-side transforms, pointwise
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(TILE_X *TILE_Y) k_collide(StepArgs a) {
  const NodeRef r = tile_node(a.tile_cav, a.cav);
  if (!r.valid) return;
  const CavDev &cv = a.cav[r.cav];
  const int64_t node = int64_t(r.j) * cv.pitch + r.i;
  const int64_t b9 = 9 * cv.off;
  T g[9];
  load9((const T *)a.g_in + b9, cv.plane, node, g);
  const T lam_prev = ((const T *)a.lam_in)[cv.off + node];

  const T c = T(cv.c), cs2 = T(cv.cs2), ics2 = T(cv.inv_cs2);
  T ux, uy, P;
  moments(g, c, cs2, ux, uy, P);                 // Eqs. (2.10)-(2.11)
  T geq[9];
  equilibrium(P, ux, uy, c, ics2, geq);          // Eq. (2.8)
  T d[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) d[q] = g[q] - geq[q];
  T pxx, pxy, pyy;
  second_moments(d, c, pxx, pxy, pyy);
  const double lam = relaxation_time(pxx, pxy, pyy, lam_prev, cv, a.powtab,
                                     a.powt + int64_t(r.cav) * POWT_SIZE);
  const T L = T(lam), dt = T(cv.dt);
  ((T *)a.lam_out)[cv.off + node] = L;           // lam(t), also next lam_prev

  const T i2 = T(1) / (T(2) * L + dt);
  const T bp = T(2) * dt * i2;     // Eq. (2.15): (2 lam - dt)/(2 lam + dt) = 1 - bp
  const T bb = T(1.5) * dt * i2;   // Eq. (2.16): 3 dt/(4 lam + 2 dt), (4 lam - dt)/(4 lam + 2 dt) = 1 - bb
  T *fp = (T *)a.fp + b9;
  T *fb = (T *)a.fb + b9;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    fp[q * cv.plane + node] = toward(g[q], geq[q], bp);
    fb[q * cv.plane + node] = toward(g[q], geq[q], bb);
  }
  double *m0 = a.m0 + 3 * cv.off;
  m0[node] = double(ux);
  m0[cv.plane + node] = double(uy);
  m0[2 * cv.plane + node] = double(P);
}

// Advection term (c_{q xi} D_xi + c_{q eta} D_eta) F_q at interior node
// (i, j) of plane F (Eqs. 3.4-3.7 with the mixed scheme of Eq. 2.5).
template <class T>
__device__ __forceinline__ T advect(const T *F, int64_t node, int pitch, int i, int j, int nx,
                                    int ny, T cxi, T ceta, const CavDev &cv) {
  // clamped neighbour offsets: the clamped values are never used
  const int im2 = i >= 2 ? -2 : -1, ip2 = i <= nx - 3 ? 2 : 1;
  const int jm2 = j >= 2 ? -2 : -1, jp2 = j <= ny - 3 ? 2 : 1;
  const T f0 = F[node];
  const T eta_b = T(cv.eta_b);
  const T dxi = dmix2(F[node + im2], F[node - 1], f0, F[node + 1], F[node + ip2], cxi >= T(0),
                      i == 1, i == nx - 2, eta_b) * T(cv.inv2dxi);
  const int64_t p = pitch;
  const T deta = dmix2(F[node + jm2 * p], F[node - p], f0, F[node + p], F[node + jp2 * p],
                       ceta >= T(0), j == 1, j == ny - 2, eta_b) * T(cv.inv2deta);
  return cxi * dxi + ceta * deta;
}

__device__ __forceinline__ void wall_neighbour(const CavDev &cv, int i, int j, int &ii, int &jj,
                                               bool &wall, double &uwx, double &uwy) {
  wall = (i == 0) | (j == 0) | (i == cv.nx - 1) | (j == cv.ny - 1);
  ii = min(max(i, 1), cv.nx - 2);
  jj = min(max(j, 1), cv.ny - 2);
  const bool lid = j == cv.ny - 1 && i > 0 && i < cv.nx - 1;
  uwx = lid ? cv.lid_ux : 0.0;
  uwy = lid ? cv.lid_uy : 0.0;
}

// Contravariant velocities of Eq. (3.4) at a node. GEN = false: the
// separable trapezoid metrics (A = c xi_x(eta), B = A x_eta(xi)/H,
// c_eta = c e_y / H); GEN = true: the per-node metric planes of a general
// quadrilateral (a handle holds one kind only, so the kind is a template
// parameter and the trapezoid kernels carry no trace of the general one).
template <bool GEN>
struct NodeMetrics {
  double a, b, c, d;  // A, B, c/H, - (trapezoid); c xi_x, c xi_y, c eta_x, c eta_y (general)
};
template <bool GEN>
__device__ __forceinline__ NodeMetrics<GEN> node_metrics(const CavDev &cv, const Geo &geo, int ii,
                                                         int jj, int64_t node) {
  NodeMetrics<GEN> m;
  if constexpr (GEN) {
    const double *gm = geo.gmet + 7 * cv.off;
    m.a = cv.c * gm[node];
    m.b = cv.c * gm[cv.plane + node];
    m.c = cv.c * gm[2 * cv.plane + node];
    m.d = cv.c * gm[3 * cv.plane + node];
  } else {
    m.a = cv.c * geo.xix[cv.goff + jj];
    m.b = m.a * geo.xeH[cv.goff + ii];
    m.c = cv.c / cv.H;
    m.d = 0.0;
  }
  return m;
}
template <bool GEN>
__device__ __forceinline__ void contravariant(const NodeMetrics<GEN> &m, int q, double &cxi,
                                              double &ceta) {
  if constexpr (GEN) {
    cxi = ex(q) * m.a + ey(q) * m.b;
    ceta = ex(q) * m.c + ey(q) * m.d;
  } else {
    cxi = cxi_of(q, m.a, m.b);
    ceta = ey(q) * m.c;
  }
}

// ---------------------------------------------------------------------------
// Step (4): half step and f(t + dt/2)
// ---------------------------------------------------------------------------
// f(t + dt/2) at interior node (ii, jj): the half step of Eq. (3.7) from
// f-bar^+, then Eq. (2.17) with the node's lambda(t).
template <class T, bool GEN>
__device__ __forceinline__ void half_at(const StepArgs &a, const CavDev &cv, int ii, int jj,
                                        T fh[9]) {
  const T *fb = (const T *)a.fb + 9 * cv.off;
  const int64_t node = int64_t(jj) * cv.pitch + ii;
  const T lam = ((const T *)a.lam_out)[cv.off + node];
  const NodeMetrics<GEN> met = node_metrics<GEN>(cv, a.geo, ii, jj, node);
  const T hdt = T(0.5 * cv.dt);
  T fbar[9];
  fbar[0] = fb[node];
#pragma unroll
  for (int q = 1; q < 9; ++q) {
    const T *F = fb + q * cv.plane;
    double cx, ce;
    contravariant(met, q, cx, ce);
    fbar[q] = F[node] - hdt * advect(F, node, cv.pitch, ii, jj, cv.nx, cv.ny, T(cx), T(ce), cv);
  }
  const T c = T(cv.c), cs2 = T(cv.cs2), ics2 = T(cv.inv_cs2);
  T ux, uy, P;
  moments(fbar, c, cs2, ux, uy, P);              // Eqs. (2.10)-(2.11) on f-bar
  T geq[9];
  equilibrium(P, ux, uy, c, ics2, geq);
  const T L = T(lam), dt = T(cv.dt);
  const T bh = dt / (T(4) * L + dt);             // Eq. (2.17): 4 lam/(4 lam + dt) = 1 - bh
#pragma unroll
  for (int q = 0; q < 9; ++q) fh[q] = toward(fbar[q], geq[q], bh);
}

// Pressure of a deviation set (Eq. 2.11).
template <class T>
__device__ __forceinline__ T pressure_of(const T g[9], const CavDev &cv) {
  T ux, uy, P;
  moments(g, T(cv.c), T(cv.cs2), ux, uy, P);
  return P;
}

// Wall value from the inner neighbour's F (in F on entry). Zeroth-order wall
// pressure: P_b = P_nb. First order (cv.wallp): P_b = 2 P_nb - P_nnb with
// F2 the same quantity at the next node beyond the neighbour.
template <class T>
__device__ __forceinline__ void wall_rule(T F[9], const T F2[9], bool first, double uwx,
                                          double uwy, const CavDev &cv) {
  if (!first) {
    nee(F, T(uwx), T(uwy), cv);
    return;
  }
  const T Pb = T(2) * pressure_of(F, cv) - pressure_of(F2, cv);
  nee_p(F, T(uwx), T(uwy), Pb, T(cv.c), T(cv.cs2), T(cv.inv_cs2));
}

template <class T, bool GEN>
__global__ void __launch_bounds__(TILE_X *TILE_Y) k_half(StepArgs a) {
  const NodeRef r = tile_node(a.tile_cav, a.cav);
  if (!r.valid) return;
  const CavDev &cv = a.cav[r.cav];
  int ii, jj;
  bool wall;
  double uwx, uwy;
  wall_neighbour(cv, r.i, r.j, ii, jj, wall, uwx, uwy);
  T fh[9];
  half_at<T, GEN>(a, cv, ii, jj, fh);
  if (wall) {
    T f2[9];
    if (cv.wallp) half_at<T, GEN>(a, cv, 2 * ii - r.i, 2 * jj - r.j, f2);
    wall_rule(fh, f2, cv.wallp != 0, uwx, GEN ? uwy : 0.0, cv);
  }
  store9((T *)a.fh + 9 * cv.off, cv.plane, int64_t(r.j) * cv.pitch + r.i, fh);
}

// ---------------------------------------------------------------------------
// Steps (5)-(6): full step, wall nodes, residual partials
// ---------------------------------------------------------------------------
// f-hat(t + dt) at interior node (ii, jj): the full step of Eq. (3.6).
template <class T, bool GEN>
__device__ __forceinline__ void full_at(const StepArgs &a, const CavDev &cv, int ii, int jj,
                                        T gn[9]) {
  const int64_t b9 = 9 * cv.off;
  const T *fh = (const T *)a.fh + b9;
  const T *fp = (const T *)a.fp + b9;
  const int64_t node = int64_t(jj) * cv.pitch + ii;
  const NodeMetrics<GEN> met = node_metrics<GEN>(cv, a.geo, ii, jj, node);
  const T dt = T(cv.dt);
  gn[0] = fp[node];
#pragma unroll
  for (int q = 1; q < 9; ++q) {
    const T *F = fh + q * cv.plane;
    double cx, ce;
    contravariant(met, q, cx, ce);
    gn[q] = fp[q * cv.plane + node] -
            dt * advect(F, node, cv.pitch, ii, jj, cv.nx, cv.ny, T(cx), T(ce), cv);  // Eq. (3.6)
  }
}

template <class T, bool GEN>
__global__ void __launch_bounds__(TILE_X *TILE_Y) k_full(StepArgs a) {
  const NodeRef r = tile_node(a.tile_cav, a.cav);
  const CavDev &cv = a.cav[r.cav];
  Partial p = {0, 0, 0, 0, 0, 0, 0};
  if (r.valid) {
    int ii, jj;
    bool wall;
    double uwx, uwy;
    wall_neighbour(cv, r.i, r.j, ii, jj, wall, uwx, uwy);
    const int64_t b9 = 9 * cv.off;
    T gn[9];
    full_at<T, GEN>(a, cv, ii, jj, gn);
    if (wall) {
      T g2[9];
      if (cv.wallp) full_at<T, GEN>(a, cv, 2 * ii - r.i, 2 * jj - r.j, g2);
      wall_rule(gn, g2, cv.wallp != 0, uwx, GEN ? uwy : 0.0, cv);
    }
    const int64_t me = int64_t(r.j) * cv.pitch + r.i;
    store9((T *)a.g_out + b9, cv.plane, me, gn);

    T ux, uy, P;
    moments(gn, T(cv.c), T(cv.cs2), ux, uy, P);
    const double u1 = double(ux), v1 = double(uy), P1 = double(P);
    if (!(isfinite(u1) && isfinite(v1))) atomicOr(a.status, 1u);
    if (a.want_residual) {
      const double *m0 = a.m0 + 3 * cv.off;
      const double du = u1 - m0[me], dv = v1 - m0[cv.plane + me], dP = P1 - m0[2 * cv.plane + me];
      p.du2 = du * du + dv * dv;
      p.u2 = u1 * u1 + v1 * v1;
      p.dP2 = dP * dP;
      const double Pfull = P1 + a.pref[r.cav];   // P of the deviations plus their reference
      p.P2 = Pfull * Pfull;
      p.du2max = p.du2;
      p.u2max = p.u2;
      const double wx = ((r.i == 0 || r.i == cv.nx - 1) ? 0.5 : 1.0) * cv.dxi;
      const double wy = ((r.j == 0 || r.j == cv.ny - 1) ? 0.5 : 1.0) * cv.deta;
      double J;
      if constexpr (GEN)
        J = a.geo.gmet[7 * cv.off + 6 * cv.plane + me];
      else
        J = a.geo.xxi[cv.goff + r.j] * cv.H;
      p.ek = 0.5 * wx * wy * J * p.u2;  // Eq. (5.1)
    }
  }
  if (a.want_residual) block_partial<TILE_X * TILE_Y / 32>(p, a.part, blockIdx.x);
}

// A cluster of CS blocks per cavity: fixed-order reduction of that cavity's
// partials, each block over a contiguous share of the slots, the last sums in
// the first block's shared memory. One block takes 2.5 us of FP64 additions
// alone for the 2065 slots of a 257^2 cavity (12 us in all); eight take an eighth.
template <int CS>
__global__ void __launch_bounds__(256) k_residual_reduce(ReduceArgs a) {
  __shared__ double all[CS][7];
  const int k = blockIdx.x / CS, r = blockIdx.x % CS;
  const CavDev &cv = a.cav[k];
  const int s0 = int(int64_t(cv.nparts) * r / CS), s1 = int(int64_t(cv.nparts) * (r + 1) / CS);
  cluster_arrive<CS>();
  previous_done();
  dependents_may_start();
  const Partial p = sum_slots(a.part + int64_t(cv.part0 + s0) * NPART, threadIdx.x, 256, s1 - s0);
  cluster_running<CS>();
  block_reduce<8>(p, cluster_at<CS>(&all[r][0]));
  cluster_done<CS>();
  if (r == 0 && threadIdx.x == 0) {
    double v[7];
#pragma unroll
    for (int q = 0; q < 7; ++q) v[q] = all[0][q];
    for (int b = 1; b < CS; ++b)
#pragma unroll
      for (int q = 0; q < 7; ++q) v[q] = q < 5 ? v[q] + all[b][q] : fmax(v[q], all[b][q]);
    residual_of(v, a.resid + 4 * k);
  }
}

// ---------------------------------------------------------------------------
// Initial state (Step 1), macros / stream function, state import and export
// ---------------------------------------------------------------------------
template <class T>
__global__ void __launch_bounds__(TILE_X *TILE_Y) k_init(const CavDev *cavs, const int *tile_cav,
                                                          T *g, T *lam) {
  const NodeRef r = tile_node(tile_cav, cavs);
  if (!r.valid) return;
  const CavDev &cv = cavs[r.cav];
  const int64_t node = int64_t(r.j) * cv.pitch + r.i;
  const bool lid = r.j == cv.ny - 1 && r.i > 0 && r.i < cv.nx - 1;
  T geq[9];
  equilibrium(T(0), lid ? T(cv.lid_ux) : T(0), lid ? T(cv.lid_uy) : T(0), T(cv.c),
              T(cv.inv_cs2), geq);
  store9(g + 9 * cv.off, cv.plane, node, geq);
  lam[cv.off + node] = T(cv.lam0);
}

// double(x) by integer instructions (the conversion would take the FP64 pipe):
// normal arguments by widen, infinities and NaNs with the largest exponent, zeros
// and subnormals scaled by 2^64 first.
__device__ __forceinline__ double to_double(float x) {
  const int b = __float_as_int(x), s = b & int(0x80000000u), m = b & 0x7FFFFFFF;
  const int t = __float_as_int(x * 0x1p64f) & 0x7FFFFFFF;
  const bool small = m < 0x00800000, large = m >= 0x7F800000;
  const int f = small ? t : m;
  const int e = large ? (2047 - 255) << 20 : (small ? (896 - 64) << 20 : 896 << 20);
  const int hi = f == 0 ? 0 : (f >> 3) + e;
  return __hiloint2double(s | hi, f << 29);
}
__device__ __forceinline__ double to_double(double x) { return x; }

struct MacrosArgs {
  const CavDev *cav;
  Geo geo;
  int cavity;
  const double *pref;
  const void *g;
  double *rho, *u, *v, *psi;
};

// Macros at every node and the stream function psi_j = deta (sum_{k <= j} I_k -
// (I_0 + I_j) / 2), I = u y_eta - v x_eta (trapezoidal rule, psi = 0 on the bottom
// wall). A cluster of CS blocks holds 32 xi = const lines, each block a share of
// the rows in MSEG segments. Pass 1: rho, u, v and I at every node (I parked in
// psi), and the segment's sum of I. The sums of the segments below, in the block
// and in the cluster's blocks before it, give each segment its offset, and pass
// 2 writes psi. One block per 32 lines left 119 of the 152 SMs idle (1025^2: 157
// us, now 71, both from a cold cache). Bound now by latency: the FP64 pipe (11
// instructions a node) has 19 us of work in it and the bytes take 13, but 264
// blocks at one per SM are 1.7 rounds, each thread taking its rows one by one.
constexpr int MSEG = 32;
constexpr int MACROS_CS = 8;

template <class T, int CS, bool GEN>
__global__ void __launch_bounds__(32 * MSEG) k_macros(MacrosArgs a) {
  const CavDev &cv = a.cav[a.cavity];
  const int i = int(blockIdx.x / CS) * 32 + threadIdx.x, r = blockIdx.x % CS;
  const int w = threadIdx.y;
  const int seg = (cv.ny + CS * MSEG - 1) / (CS * MSEG);
  const int j0 = min(cv.ny, (r * MSEG + w) * seg), j1 = min(cv.ny, j0 + seg);
  const bool col = i < cv.nx;
  const int64_t plane = cv.plane, pitch = cv.pitch, nx = cv.nx;
  const double rho0 = cv.rho0, ics2 = cv.inv_cs2, H = cv.H, deta = cv.deta;
  const T c = T(cv.c), cs2 = T(cv.cs2);
  const double xeta = col && !GEN ? a.geo.xeta[cv.goff + i] : 0.0;
  const double *gm = GEN ? a.geo.gmet + 7 * cv.off : nullptr;
  __shared__ double part[MSEG][33];  // (a line's sums are read along it too)
  __shared__ double below[CS][32];   // (first block's: the blocks' totals)
  if (a.psi) cluster_arrive<CS>();   // (psi: uniform over the launch)
  previous_done();
  dependents_may_start();
  const double p0 = a.pref[a.cavity];
  const T *gb = (const T *)a.g + 9 * cv.off;
  double sum = 0.0;
  for (int j = j0; col && j < j1; ++j) {
    T gg[9];
    const int64_t nd = j * pitch + i, o = j * nx + i;
    load9(gb, plane, nd, gg);
    T ux, uy, P;
    moments(gg, c, cs2, ux, uy, P);
    const double ud = to_double(ux), vd = to_double(uy);
    if (a.rho) a.rho[o] = rho0 + (p0 + to_double(P)) * ics2;
    if (a.u) a.u[o] = ud;
    if (a.v) a.v[o] = vd;
    if (a.psi) {
      double I;
      if constexpr (GEN)
        I = ud * gm[5 * plane + nd] - vd * gm[4 * plane + nd];
      else
        I = ud * H - vd * xeta;
      a.psi[o] = I;
      sum += I;
    }
  }
  if (!a.psi) return;  // uniform over the launch
  double acc = 0.0;
  if (r == 0 && w == 0 && col) acc = -0.5 * a.psi[i];  // I_0 counts half
  part[w][threadIdx.x] = sum + acc;
  __syncthreads();
  {  // sums of the segments up to each, along every line: warp w takes line w
    double v = part[threadIdx.x][w];
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const double b = __shfl_up_sync(0xffffffffu, v, o);
      if (int(threadIdx.x) >= o) v += b;
    }
    part[threadIdx.x][w] = v;
  }
  __syncthreads();
  if (w > 0) acc = part[w - 1][threadIdx.x];
  if constexpr (CS > 1) {
    cluster_running<CS>();
    if (w == MSEG - 1) cluster_at<CS>(&below[r][0])[threadIdx.x] = part[w][threadIdx.x];
    cluster_done<CS>();
    const double *all = cluster_at<CS>(&below[0][0]);
    for (int b = 0; b < r; ++b) acc += all[b * 32 + threadIdx.x];
    cluster_done<CS>();   // the first block's memory is there until all have read it
  }
  for (int j = j0; col && j < j1; ++j) {
    const int64_t o = j * nx + i;
    const double I = a.psi[o];
    acc += I;
    a.psi[o] = deta * (acc - 0.5 * I);
  }
}

// Probes: u, v, P (Eqs. 2.10-2.11, P including the reference pressure of the
// stored deviations) at n nodes given as (cavity, i, j); a probe outside its
// cavity (or naming no cavity) gets NaN.
template <class T>
__global__ void k_probe(const CavDev *cavs, int ncav, const double *pref, const T *g, int n,
                        const int *probes, double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int c = probes[3 * k], i = probes[3 * k + 1], j = probes[3 * k + 2];
  if (c < 0 || c >= ncav || i < 0 || j < 0 || i >= cavs[c].nx || j >= cavs[c].ny) {
    out[3 * k] = out[3 * k + 1] = out[3 * k + 2] = nan("");
    return;
  }
  const CavDev &cv = cavs[c];
  T gg[9];
  load9(g + 9 * cv.off, cv.plane, int64_t(j) * cv.pitch + i, gg);
  T ux, uy, P;
  moments(gg, T(cv.c), T(cv.cs2), ux, uy, P);
  out[3 * k] = double(ux);
  out[3 * k + 1] = double(uy);
  out[3 * k + 2] = pref[c] + double(P);
}

template <class T>
__global__ void k_export(const CavDev *cavs, int cavity, const double *pref, const T *g,
                         const T *lam, double *fhat, double *lamo) {
  const CavDev &cv = cavs[cavity];
  const double pt = pref[cavity] * cv.inv_cs2;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= cv.nx) return;
  const int64_t node = int64_t(j) * cv.pitch + i, o = int64_t(j) * cv.nx + i;
  const int64_t n2 = int64_t(cv.nx) * cv.ny;
  if (fhat)
#pragma unroll
    for (int q = 0; q < 9; ++q)
      fhat[q * n2 + o] = double(g[9 * cv.off + q * cv.plane + node]) + wgt(q) * cv.rho0 +
                         wbar(q) * pt;
  if (lamo) lamo[o] = double(lam[cv.off + node]);
}

template <class T>
__global__ void k_import(const CavDev *cavs, int cavity, const double *pref, T *g, T *lam,
                         const double *fhat, const double *lami) {
  const CavDev &cv = cavs[cavity];
  const double pt = pref[cavity] * cv.inv_cs2;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
  if (i >= cv.nx) return;
  const int64_t node = int64_t(j) * cv.pitch + i, o = int64_t(j) * cv.nx + i;
  const int64_t n2 = int64_t(cv.nx) * cv.ny;
#pragma unroll
  for (int q = 0; q < 9; ++q)
    g[9 * cv.off + q * cv.plane + node] = T(fhat[q * n2 + o] - wgt(q) * cv.rho0 - wbar(q) * pt);
  lam[cv.off + node] = T(lami[o]);
}

// Copies up to three segments of device memory (ifdlbm_save_state_dev and the
// like), 16 bytes per thread and turn. Bound by the launch at the sizes it is
// used for: the state of a 257^2 cavity 2.9 us (16.5 as three copies of the
// copy engine), its step's intermediates 4.1 us (24.7).
__global__ void __launch_bounds__(256) k_copy(CopyArgs a) {
  previous_done();
  dependents_may_start();
  const int64_t t0 = int64_t(blockIdx.x) * 256 + threadIdx.x, step = int64_t(gridDim.x) * 256;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int4 *src = static_cast<const int4 *>(a.src[k]);
    int4 *dst = static_cast<int4 *>(a.dst[k]);
    const int64_t n = a.bytes[k] / 16;
    int64_t t = t0;
    for (; t + 3 * step < n; t += 4 * step) {
      const int4 v0 = src[t], v1 = src[t + step], v2 = src[t + 2 * step], v3 = src[t + 3 * step];
      dst[t] = v0;
      dst[t + step] = v1;
      dst[t + 2 * step] = v2;
      dst[t + 3 * step] = v3;
    }
    for (; t < n; t += step) dst[t] = src[t];
    if (t0 < (a.bytes[k] & 15) / 8)   // a last double
      reinterpret_cast<double *>(dst + n)[t0] = reinterpret_cast<const double *>(src + n)[t0];
  }
}

// Re-basing of the stored deviations on the mean pressure (FP32 storage):
// a uniform pressure offset is a neutral mode of the scheme that drifts, and
// carrying it in every g_i would make the FP32 rounding of g grow with it.
// k_psum: per tile, sum of P(g) in FP64; k_pshift: per cavity, the mean
// (fixed-order sum over its tiles) into ptile[ntiles + k], pref += mean;
// k_rebase: g_i -= wbar_i mean / c_s^2 at every node (one rounding).
template <class T>
__global__ void __launch_bounds__(TILE_X *TILE_Y) k_psum(const CavDev *cavs, const int *tile_cav,
                                                          const T *g, double *ptile) {
  const NodeRef r = tile_node(tile_cav, cavs);
  const CavDev &cv = cavs[r.cav];
  double v = 0.0;
  if (r.valid) {
    T gg[9];
    load9(g + 9 * cv.off, cv.plane, int64_t(r.j) * cv.pitch + r.i, gg);
    T ux, uy, P;
    moments(gg, T(cv.c), T(cv.cs2), ux, uy, P);
    v = double(P);
  }
  __shared__ double sh[TILE_X * TILE_Y];
  const int t = threadIdx.y * TILE_X + threadIdx.x;
  sh[t] = v;
  __syncthreads();
  for (int w = TILE_X * TILE_Y / 2; w > 0; w >>= 1) {
    if (t < w) sh[t] += sh[t + w];
    __syncthreads();
  }
  if (t == 0) ptile[blockIdx.x] = sh[0];
}

__global__ void k_pshift(const CavDev *cavs, int ntiles, double *ptile, double *pref) {
  const CavDev &cv = cavs[blockIdx.x];
  const int n = cv.tiles_x * cv.tiles_y;
  __shared__ double sh[256];
  double v = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) v += ptile[cv.tile0 + k];
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double mean = sh[0] / (double(cv.nx) * cv.ny);
    ptile[ntiles + blockIdx.x] = mean;
    pref[blockIdx.x] += mean;
  }
}

template <class T>
__global__ void __launch_bounds__(TILE_X *TILE_Y) k_rebase(const CavDev *cavs, const int *tile_cav,
                                                            T *g, const double *ptile, int ntiles) {
  const NodeRef r = tile_node(tile_cav, cavs);
  if (!r.valid) return;
  const CavDev &cv = cavs[r.cav];
  const double pt = ptile[ntiles + r.cav] * cv.inv_cs2;
  T *gb = g + 9 * cv.off;
  const int64_t node = int64_t(r.j) * cv.pitch + r.i;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    T &x = gb[q * cv.plane + node];
    x = T(double(x) - wbar(q) * pt);
  }
}

__global__ void k_pow_selftest(int n, const double *x, double m, const double *tab, double *fast,
                               double *ref) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  fast[k] = pow_fast(x[k], m, tab);
  ref[k] = pow(x[k], m);
}

void launch_pow_selftest(int n, const double *x, double m, const double *tab, double *fast,
                         double *ref, cudaStream_t s) {
  k_pow_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, x, m, tab, fast, ref);
}

// pow_tab on the FP32 roundings of x (tab: a cavity table of exponent m and
// factor C); out[k] = pow_tab(float(x[k])) and out[n + k] = C * CUDA's
// pow(double(float(x[k])), m).
__global__ void k_pow_tab_selftest(int n, const double *x, double m, double C, const double *tab,
                                   double b2, float b3, float b4, float b5, double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float xf = float(x[k]);
  out[k] = pow_tab(xf, tab, m, b2, b3, b4, b5);
  out[n + k] = C * pow(double(xf), m);
}

void launch_pow_tab_selftest(int n, const double *x, double m, double C, const double *tab,
                             double b2, float b3, float b4, float b5, double *out, cudaStream_t s) {
  k_pow_tab_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, x, m, C, tab, b2, b3, b4, b5, out);
}

// The FP32 form's power of Eq. (1.4) as the fused kernel evaluates it (pow_pair
// where its table covers the argument and the float is not in doubt, else
// pow_tab): out[k] of the FP32 rounding of x[k], and out[n + k] = pow_tab's value
// rounded to FP32.
__global__ void k_pow_pair_selftest(int n, const double *x, const CavDev *cavs, int cavity,
                                    const double *powt, const float *powp, double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const CavDev &cv = cavs[cavity];
  const PowPair pw = {powp, cv.pb1h, cv.pb1l, cv.pb2f, cv.pb3, cv.pb4, cv.pe_lo, cv.pe_n};
  const float xf = float(x[k]);
  const float t = float(pow_tab(xf, powt, cv.half_nm1, cv.pb2, cv.pb3, cv.pb4, cv.pb5));
  float r;
  out[k] = double(pow_pair_covers(xf, pw) && pow_pair(xf, pw, r) ? r : t);
  out[n + k] = double(t);
}
void launch_pow_pair_selftest(int n, const double *x, const CavDev *cav, int cavity,
                              const double *powt, const float *powp, double *out, cudaStream_t s) {
  k_pow_pair_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, x, cav, cavity, powt, powp, out);
}

// The implicit form's root as the fused kernel forms it (lambda_implicit_pair):
// out[k] at G2 = x[k] (a float, in units of c) from the lagged value x[n + k], and
// out[n + k] = the FP64 solve rounded to FP32.
__global__ void k_implicit_selftest(int n, const double *x, const CavDev *cavs, int cavity,
                                    const double *powtab, const double *powt, const float *powp,
                                    double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const CavDev &cv = cavs[cavity];
  const PowPair pw = {powp, cv.pb1h, cv.pb1l, cv.pb2f, cv.pb3, cv.pb4, cv.pe_lo, cv.pe_n};
  const float G2 = float(x[k]), start = float(x[n + k]);
  out[k] = double(lambda_implicit_pair(G2, start, impl_pair(cv), pw, cv, powtab, powt));
  out[n + k] =
      double(float(lambda_implicit(6.0 * sqrt(double(G2)), double(start), cv, powtab, powt)));
}
void launch_implicit_selftest(int n, const double *x, const CavDev *cav, int cavity,
                              const double *powtab, const double *powt, const float *powp,
                              double *out, cudaStream_t s) {
  k_implicit_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, x, cav, cavity, powtab, powt, powp, out);
}

__global__ void k_recip_selftest(int n, const double *x, double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = recip(x[k]);
}
void launch_recip_selftest(int n, const double *x, double *out, cudaStream_t s) {
  k_recip_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, x, out);
}

__global__ void k_power64_selftest(int n, const double *x, const CavDev *cavs, int cavity,
                                   const double *powtab, const double *powt, double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = power64(x[k], cavs[cavity], powtab, powt);
}
void launch_power64_selftest(int n, const double *x, const CavDev *cav, int cavity,
                             const double *powtab, const double *powt, double *out,
                             cudaStream_t s) {
  k_power64_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, x, cav, cavity, powtab, powt, out);
}

__global__ void k_pow_f32_selftest(int n, const double *x, double m, double *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  out[k] = double(pow_f32(float(x[k]), float(m)));
}

// Per-node metric planes of the general quadrilaterals, one thread per node
// (blockIdx.y = cavity).
__global__ void k_quad_metrics(const CavDev *cavs, const double *corners, double *gmet) {
  const CavDev &cv = cavs[blockIdx.y];
  const int64_t n = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (n >= int64_t(cv.nx) * cv.ny) return;
  const int j = int(n / cv.nx), i = int(n - int64_t(j) * cv.nx);
  double m[7];
  quad_node_metrics(corners + 8 * blockIdx.y, double(i) / (cv.nx - 1), double(j) / (cv.ny - 1), m);
  double *gm = gmet + 7 * cv.off;
  const int64_t node = int64_t(j) * cv.pitch + i;
#pragma unroll
  for (int t = 0; t < 7; ++t) gm[t * cv.plane + node] = m[t];
}

// FP32 roundings of c xi_x, c xi_y, c eta_x, c eta_y and J (formed in FP64 by
// k_quad_metrics), one thread per node (blockIdx.y = cavity).
__global__ void k_quad_metrics_f32(const CavDev *cavs, const double *gmet, float *qmet_f) {
  const CavDev &cv = cavs[blockIdx.y];
  const int64_t n = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (n >= int64_t(cv.nx) * cv.ny) return;
  const int j = int(n / cv.nx), i = int(n - int64_t(j) * cv.nx);
  const int64_t node = int64_t(j) * cv.pitch + i;
  const double *gm = gmet + 7 * cv.off;
  float *qm = qmet_f + 5 * cv.off;
#pragma unroll
  for (int t = 0; t < 4; ++t) qm[t * cv.plane + node] = float(cv.c * gm[t * cv.plane + node]);
  qm[4 * cv.plane + node] = float(gm[6 * cv.plane + node]);
}

void launch_quad_metrics_f32(const CavDev *cav, int ncav, int64_t max_n2, const double *gmet,
                             float *qmet_f, cudaStream_t s) {
  const dim3 grid(unsigned((max_n2 + 255) / 256), unsigned(ncav));
  k_quad_metrics_f32<<<grid, 256, 0, s>>>(cav, gmet, qmet_f);
}

void launch_quad_metrics(const CavDev *cav, int ncav, int64_t max_n2, const double *corners,
                         double *gmet, cudaStream_t s) {
  const dim3 grid(unsigned((max_n2 + 255) / 256), unsigned(ncav));
  k_quad_metrics<<<grid, 256, 0, s>>>(cav, corners, gmet);
}

void launch_pow_f32_selftest(int n, const double *x, double m, double *out, cudaStream_t s) {
  k_pow_f32_selftest<<<(n + 255) / 256, 256, 0, s>>>(n, x, m, out);
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
static const dim3 kTile(TILE_X, TILE_Y);

void launch_collide(const StepArgs &a, int ntiles, cudaStream_t s) {
  k_collide<float><<<ntiles, kTile, 0, s>>>(a);
}
void launch_half(const StepArgs &a, int ntiles, cudaStream_t s) {
  if (a.geo.gmet)
    k_half<float, true><<<ntiles, kTile, 0, s>>>(a);
  else
    k_half<float, false><<<ntiles, kTile, 0, s>>>(a);
}
void launch_full(const StepArgs &a, int ntiles, cudaStream_t s) {
  if (a.geo.gmet)
    k_full<float, true><<<ntiles, kTile, 0, s>>>(a);
  else
    k_full<float, false><<<ntiles, kTile, 0, s>>>(a);
}
void launch_residual_reduce(const CavDev *cav, const double *part, double *resid, int ncav,
                            int most, cudaStream_t s) {
  const ReduceArgs a{cav, part, resid};
  if (most > REDUCE_ONE)
    launch_after(k_residual_reduce<REDUCE_CS>, ncav * REDUCE_CS, 256, 0, s, a, REDUCE_CS);
  else
    launch_after(k_residual_reduce<1>, ncav, 256, 0, s, a);
}
cudaError_t launch_copy(const CopyArgs &a, const void *mine, int device, cudaStream_t s) {
  cudaPointerAttributes at = {};
  const bool here = cudaPointerGetAttributes(&at, mine) == cudaSuccess &&
                    at.type == cudaMemoryTypeDevice && at.device == device;
  // (an address CUDA does not know: the copies below say so; and an error left by
  // earlier, unrelated work is not this call's)
  (void)cudaGetLastError();
  if (copy_by_kernel(a, here)) {
    const int64_t blocks = ((a.bytes[0] + a.bytes[1] + a.bytes[2]) / 16 + 255) / 256;
    launch_after(k_copy, int(std::max<int64_t>(1, std::min<int64_t>(blocks, 152 * 8))), 256, 0, s,
                 a);
    count_launches(1);
    return cudaGetLastError();
  }
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < 3 && e == cudaSuccess; ++k)
    if (a.bytes[k])
      e = cudaMemcpyAsync(a.dst[k], a.src[k], size_t(a.bytes[k]), cudaMemcpyDeviceToDevice, s);
  return e;
}
template <class T> void launch_init(const CavDev *cav, const int *tile_cav, void *g, void *lam,
                                    int ntiles, cudaStream_t s) {
  k_init<T><<<ntiles, kTile, 0, s>>>(cav, tile_cav, (T *)g, (T *)lam);
}
template <class T> void launch_macros(const CavDev *cav, Geo geo, int cavity, const double *pref,
                                      const void *g, double *rho, double *u, double *v,
                                      double *psi, int nx, int ny, cudaStream_t s) {
  // (a cluster's blocks get a row per thread from 8 x 32 rows on)
  const MacrosArgs a{cav, geo, cavity, pref, g, rho, u, v, psi};
  const int lines = (nx + 31) / 32;
  const dim3 block(32, MSEG);
  if (ny >= MACROS_CS * MSEG)
    launch_after(geo.gmet ? k_macros<T, MACROS_CS, true> : k_macros<T, MACROS_CS, false>,
                 lines * MACROS_CS, block, 0, s, a, MACROS_CS);
  else
    launch_after(geo.gmet ? k_macros<T, 1, true> : k_macros<T, 1, false>, lines, block, 0, s, a);
}
template <class T> void launch_export(const CavDev *cav, int cavity, const double *pref,
                                      const void *g, const void *lam, double *fhat,
                                      double *lamo, int nx, int ny, cudaStream_t s) {
  k_export<T><<<dim3((nx + 127) / 128, ny), 128, 0, s>>>(cav, cavity, pref, (const T *)g,
                                                          (const T *)lam, fhat, lamo);
}
template <class T> void launch_import(const CavDev *cav, int cavity, const double *pref, void *g,
                                      void *lam, const double *fhat, const double *lami,
                                      int nx, int ny, cudaStream_t s) {
  k_import<T><<<dim3((nx + 127) / 128, ny), 128, 0, s>>>(cav, cavity, pref, (T *)g, (T *)lam,
                                                          fhat, lami);
}
template <class T> void launch_probe(const CavDev *cav, int ncav, const double *pref, const void *g,
                                     int n, const int *probes, double *out, cudaStream_t s) {
  k_probe<T><<<(n + 127) / 128, 128, 0, s>>>(cav, ncav, pref, (const T *)g, n, probes, out);
}
template <class T> void launch_rebase(const CavDev *cav, const int *tile_cav, void *g,
                                      double *pref, double *ptile, int ntiles, int ncav,
                                      cudaStream_t s) {
  k_psum<T><<<ntiles, kTile, 0, s>>>(cav, tile_cav, (const T *)g, ptile);
  k_pshift<<<ncav, 256, 0, s>>>(cav, ntiles, ptile, pref);
  k_rebase<T><<<ntiles, kTile, 0, s>>>(cav, tile_cav, (T *)g, ptile, ntiles);
}

#define IFD_INSTANTIATE(T)                                                                     \
  template void launch_init<T>(const CavDev *, const int *, void *, void *, int,              \
                               cudaStream_t);                                                  \
  template void launch_macros<T>(const CavDev *, Geo, int, const double *, const void *,      \
                                 double *, double *, double *, double *, int, int,            \
                                 cudaStream_t);                                               \
  template void launch_export<T>(const CavDev *, int, const double *, const void *,           \
                                 const void *, double *, double *, int, int, cudaStream_t);   \
  template void launch_import<T>(const CavDev *, int, const double *, void *, void *,         \
                                 const double *, const double *, int, int, cudaStream_t);     \
  template void launch_probe<T>(const CavDev *, int, const double *, const void *, int,       \
                                const int *, double *, cudaStream_t);                         \
  template void launch_rebase<T>(const CavDev *, const int *, void *, double *, double *, int, \
                                 int, cudaStream_t);
IFD_INSTANTIATE(double)
IFD_INSTANTIATE(float)

}  // namespace ifd
