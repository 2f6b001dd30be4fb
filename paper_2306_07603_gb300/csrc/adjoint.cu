// Discrete adjoint (reverse mode) of one staged FP64 IFDLBM step.
//
// Forward step n (staged kernels; per node, deviation variables g):
//   K1  (u, v, P) = M(g), geq = E(u, v, P), Pi = sum c c (g - geq),
//       q = k^2 (Pxx^2 + 2 Pxy^2 + Pyy^2)/2, k = -2/((2 lam_p + dt) c_s^2),
//       lam = K/c_s^2 max(q, gmin^2)^((n-1)/2)                (Eqs. 1.4, 2.12-2.14)
//       FP = ap g + bp geq, FB = ab g + bb geq                (Eqs. 2.15-2.16)
//   K2  FBAR = FB - dt/2 A(FB), FH = ah FBAR + bh E(M(FBAR)) (Eqs. 3.7, 2.17)
//       wall b: FH(b) = X(FH(nb))                             (extrapolation)
//   K3  GN = FP - dt A(FH); wall b: GN(b) = X(GN(nb))         (Eq. 3.6, Step 6)
// with A_q = c_xi D_xi + c_eta D_eta the mixed scheme (Eqs. 2.5-2.7, 3.4) and
// X(F) = E(u_w, P(F)) + F - E(u(F), P(F)). Since dE/dP does not depend on u,
// X^T(G) = G - c (e_x ubar + e_y vbar) with (ubar, vbar) = (dE/du)^T G at u(F).
//
// The reverse sweep of a step takes three launches and a reduction:
//
//   k_adj_ring   G' = Gbar + X^T(walls) at the interior nodes next to a wall, in
//                place (each wall node has one source, so no two threads meet)
//   k_adj_full   FHbar = -dt A^T(G'), its wall terms by evaluating the gather
//                again at the wall nodes of a ring node, and the half step's
//                pointwise adjoint: FBARbar = ah FHbar + M^T E^T (bh FHbar)
//   k_adj_half   FBbar = FBARbar - dt/2 A^T(FBARbar) and the collision's adjoint,
//                that of (g_n, lambda_n)
//
// Parameters: n (through K = U^(2-n) H^n / Re and the exponent), Re (through K)
// and theta in degrees (through c_xi of Eq. 3.4 via cot theta, and the
// Jacobian of the kinetic-energy objective of Eq. 5.1); their partials are
// summed per block and then per cavity, in a fixed order.
//
// Bound: the FP64 pipe, as the forward step (step64.cuh). The gathers take four
// terms per axis with the coefficients and sides selected by integer
// instructions, the transposed moments and equilibrium are summed by pairs of
// opposite directions, and no pass re-forms what another has in registers.
// FP64 instructions per warp: k_adj_full 305, k_adj_half 412, the ring a small
// extra; a reverse step at 257^2 takes 126 us, at 65^2 53 us (there the latency
// of a warp). The nine launches before (wall transposes and additions as
// kernels of their own, gathers of both upwind sides) took 1980 and 400 us.
#include <cstdint>

#include "d2q9.cuh"
#include "internal.h"
#include "launch.cuh"
#include "reduce.cuh"
#include "step64.cuh"

namespace ifd {

namespace {

struct Ref {
  int cav, i, j;
  bool valid;
};

__device__ __forceinline__ Ref tile_ref(const int *tile_cav, const CavDev *cavs) {
  Ref r;
  const int t = blockIdx.x;
  r.cav = tile_cav[t];
  const CavDev &cv = cavs[r.cav];
  const int lt = t - cv.tile0;
  r.i = (lt % cv.tiles_x) * TILE_X + threadIdx.x;
  r.j = (lt / cv.tiles_x) * TILE_Y + threadIdx.y;
  r.valid = r.i < cv.nx && r.j < cv.ny;
  return r;
}

// Sum over the block of the N <= 8 values v, written by its first N threads to
// part[slot * N ..] (fixed order).
template <int N, int NWARPS>
__device__ __forceinline__ void block_sum(const double (&v)[N], double *part, int64_t slot) {
  __shared__ double sh[NWARPS][N];
  const int lane = threadIdx.x + threadIdx.y * blockDim.x;
  const int w = lane >> 5, l = lane & 31;
  double v8[8] = {};
#pragma unroll
  for (int k = 0; k < N; ++k) v8[k] = v[k];
  const double s = warp_sums8(v8);
  if ((l & 3) == 0 && l < 4 * N) sh[w][l >> 2] = s;
  __syncthreads();
  if (lane < N) {
    double acc = 0.0;
    for (int k = 0; k < NWARPS; ++k) acc += sh[k][lane];
    part[slot * N + lane] = acc;
  }
}

// The interior node of this thread: blocks [0, nblk_core) of a cavity take the
// nodes away from the walls row by row, the blocks after them the ring of
// nodes next to a wall (rows 1 and ny-2, then columns 1 and nx-2 in turn).
template <int NT>
__device__ __forceinline__ Node64 interior_node(const int *blk_cav, const CavDev *cavs,
                                                bool ring_only) {
  Node64 r;
  r.cav = blk_cav[blockIdx.x];
  const CavDev &cv = cavs[r.cav];
  const int lb = int(blockIdx.x) - (ring_only ? cv.ring0 : cv.adj0);
  const int core = ring_only ? 0 : cv.nblk_core;
  r.wall = lb >= core;  // a ring node
  if (!r.wall) {
    const unsigned n = unsigned(lb) * NT + threadIdx.x, w = unsigned(cv.nx - 4), row = n / w;
    r.valid = row < unsigned(cv.ny - 4);
    r.i = int(n - row * w) + 2;
    r.j = int(row) + 2;
  } else {
    const int n = (lb - core) * NT + int(threadIdx.x), w = cv.nx - 2, k = n - 2 * w;
    r.valid = k < 2 * (cv.ny - 4);
    if (k < 0) {
      const bool top = n >= w;
      r.i = 1 + (top ? n - w : n);
      r.j = top ? cv.ny - 2 : 1;
    } else {
      r.i = (k & 1) ? cv.nx - 2 : 1;
      r.j = 2 + (k >> 1);
    }
  }
  return r;
}

// (dE / d(m_x, m_y, p))^T h at m, E the equilibrium in lattice units
// (equilibrium64): x, y, p.
struct Adj64 {
  double x, y, p;
};
__device__ __forceinline__ Adj64 equilibrium_T(const double h[9], double mx, double my) {
  const double s13 = h[1] + h[3], d13 = h[1] - h[3], s24 = h[2] + h[4], d24 = h[2] - h[4];
  const double s57 = h[5] + h[7], d57 = h[5] - h[7], s68 = h[6] + h[8], d68 = h[6] - h[8];
  const double t9 = (1.0 / 9.0) * fma(0.25, s57 + s68, s13 + s24);
  const double w3 = -3.0 * fma(4.0 / 9.0, h[0], t9);  // -3 sum w_i h_i
  const double a = (mx + my) * s57, b = (my - mx) * s68;
  Adj64 r;
  r.p = fma(-5.0 / 9.0, h[0], t9);
  r.x = fma(1.0 / 3.0, d13, fma(1.0 / 12.0, d57 - d68, fma(0.25, a - b, mx * (s13 + w3))));
  r.y = fma(1.0 / 3.0, d24, fma(1.0 / 12.0, d57 + d68, fma(0.25, a + b, my * (s24 + w3))));
  return r;
}

// out[i] = k h[i] + (dM/dg)^T (x, y, p), M the moments of moments64 at m.
__device__ __forceinline__ void moments_T(const Adj64 &b, double mx, double my, double k,
                                          const double h[9], double out[9]) {
  const double p2 = -2.4 * b.p, X = fma(p2, mx, b.x), Y = fma(p2, my, b.y), Z = 1.8 * b.p;
  const double s = X + Y, d = Y - X;
  out[0] = k * h[0];
  out[1] = fma(k, h[1], Z + X);
  out[3] = fma(k, h[3], Z - X);
  out[2] = fma(k, h[2], Z + Y);
  out[4] = fma(k, h[4], Z - Y);
  out[5] = fma(k, h[5], Z + s);
  out[7] = fma(k, h[7], Z - s);
  out[6] = fma(k, h[6], Z + d);
  out[8] = fma(k, h[8], Z - d);
}

// h += X^T(w), X the wall rule (Sec. 4) at the populations F of the inner
// neighbour: X^T(w) = w - e (dE/dm)^T w.
__device__ __forceinline__ void wall_T(double h[9], const double w[9], double mx, double my) {
  const Adj64 b = equilibrium_T(w, mx, my);
  const double s = b.x + b.y, d = b.y - b.x;
  h[0] += w[0];
  h[1] += w[1] - b.x;
  h[3] += w[3] + b.x;
  h[2] += w[2] - b.y;
  h[4] += w[4] + b.y;
  h[5] += w[5] - s;
  h[7] += w[7] + s;
  h[6] += w[6] - d;
  h[8] += w[8] + d;
}

// The wall nodes whose extrapolation source is ring node (i, j), at most three:
// the node across the side wall, the one across the bottom or lid, and at a
// corner the diagonal one. `k` in 0..2; false if there is no such node.
__device__ __forceinline__ bool wall_of(const CavDev &cv, int i, int j, int k, int &wi, int &wj) {
  const int si = i == 1 ? 0 : (i == cv.nx - 2 ? cv.nx - 1 : -1);
  const int sj = j == 1 ? 0 : (j == cv.ny - 2 ? cv.ny - 1 : -1);
  wi = k == 1 ? i : si;
  wj = k == 0 ? j : sj;
  return (k == 1 || si >= 0) && (k == 0 || sj >= 0);
}

// What a gather at node (i, j) takes besides the planes. xi: the nodes x = i + o,
// o = -2..2, that the transposed stencils of row j reach: which are interior
// (none if j is a wall row) and which are next to a wall; eta: the same for
// the rows j + o of column i. Bit o + 2.
struct Gather64 {
  const double *G;        // plane 0 at the node
  int64_t plane;
  int pitch, ix;          // ix: index of the node in the column tables
  unsigned xin, xlo, xhi, ein, elo, ehi;
  double A;               // scale c xi_x / (2 dxi) of the row
};
__device__ __forceinline__ unsigned bits5(int at, int lo, int hi) {
  // bit o + 2 for lo <= at + o <= hi
  unsigned b = 0;
#pragma unroll
  for (int o = -2; o <= 2; ++o) b |= (at + o >= lo && at + o <= hi) ? 1u << (o + 2) : 0u;
  return b;
}
__device__ __forceinline__ Gather64 gather_at(const CavDev &cv, const Geo &geo, int stage, int i,
                                              int j) {
  Gather64 g;
  g.plane = cv.plane;
  g.pitch = cv.pitch;
  g.ix = cv.goff + i;
  const bool row = j >= 1 && j <= cv.ny - 2, col = i >= 1 && i <= cv.nx - 2;
  g.xin = row ? bits5(i, 1, cv.nx - 2) : 0u;
  g.xlo = bits5(i, 1, 1);
  g.xhi = bits5(i, cv.nx - 2, cv.nx - 2);
  g.ein = col ? bits5(j, 1, cv.ny - 2) : 0u;
  g.elo = bits5(j, 1, 1);
  g.ehi = bits5(j, cv.ny - 2, cv.ny - 2);
  g.A = geo.ax[stage][cv.goff + j];
  g.G = nullptr;
  return g;
}

// Sum over the nodes x = y + o d of one line through y of G(x) m(x) times the
// coefficient of F(y) in the mixed difference at x, added to acc: x = y is the
// centre, x one node upwind of y takes y as its downwind neighbour (ka), one
// node downwind as its upwind one (kb), two downwind as the far one (kf).
// `pos`: bit o + 2, the side of x; `in`, `lo`, `hi` as in Gather64. UNIT: m = 1.
// Where the side changes between y - 2 (from above) and y + 2 (from below)
// both far terms are there; elsewhere there is one at most.
template <bool UNIT>
__device__ __forceinline__ double line_T(const double *G, int d, unsigned pos, unsigned in,
                                         unsigned lo, unsigned hi, const double m[5],
                                         const Mix64 &c, double acc) {
  const unsigned edge = (pos & lo) | (~pos & hi);
  auto side = [&](unsigned b, unsigned bit) { return (b & bit) != 0; };
  auto put = [&](int o, double k) {
    const bool on = side(in, 1u << (o + 2));
    const double w = on ? (UNIT ? k : k * m[o + 2]) : 0.0;
    acc = fma(w, G[on ? o * d : 0], acc);
  };
  const double km = side(edge, 2u) ? c.wb : c.kb, kp = side(edge, 8u) ? c.wb : c.kb;
  put(0, side(edge, 4u) ? c.w0 : c.k0);
  put(-1, side(pos, 2u) ? c.ka : km);
  put(1, side(pos, 8u) ? kp : c.ka);
  const bool up = side(pos & in, 16u), down = side(~pos & in, 1u);
  const double mf = UNIT ? 1.0 : (up ? m[4] : m[0]);
  acc = fma((up || down) ? (UNIT ? c.kf : c.kf * mf) : 0.0, G[up ? 2 * d : (down ? -2 * d : 0)], acc);
  if (up && down) acc = fma(UNIT ? c.kf : c.kf * m[0], G[-2 * d], acc);
  return acc;
}

// out[q] += -scale (A^T G)_q at the gather's node, all moving populations.
__device__ __forceinline__ void advect_T(const Gather64 &g, const Geo &geo, const Mix64 &mix,
                                         const Mix64 &mixe, double out[9]) {
  auto pair = [&](auto pc) {
    constexpr int p = decltype(pc)::value;
    constexpr int q0 = p == 0 ? 1 : (p == 1 ? 2 : (p == 2 ? 5 : 6)), q1 = p < 2 ? q0 + 2 : q0 + 2;
    // side and magnitude of c_xi / (c xi_x) at the five nodes, for q0
    double m[5] = {1.0, 1.0, 1.0, 1.0, 1.0};
    unsigned pos = 31u;
    if constexpr (p > 0) {
      const double *tab = p == 1 ? geo.xeH : (p == 2 ? geo.xm : geo.xp);
      pos = 0u;
#pragma unroll
      for (int o = -2; o <= 2; ++o) {
        const double v = tab[g.ix + ((g.xin >> (o + 2)) & 1u ? o : 0)];
        const bool neg = negative(v);
        pos |= (p == 2 ? !neg : neg) ? 1u << (o + 2) : 0u;
        m[o + 2] = fabs(v);
      }
    }
    auto one = [&](auto qc, unsigned side) {
      constexpr int q = decltype(qc)::value;
      const double *G = g.G + q * g.plane;
      double r = out[q];
      if constexpr (p > 0) {
        constexpr bool epos = q == 2 || q == 5 || q == 6;
        r = line_T<true>(G, g.pitch, epos ? 31u : 0u, g.ein, g.elo, g.ehi, m, mixe, r);
      }
      out[q] = fma(-g.A, line_T<p == 0>(G, 1, side, g.xin, g.xlo, g.xhi, m, mix, 0.0), r);
    };
    one(Const<q0>(), pos);
    one(Const<q1>(), ~pos);
  };
  pair(Const<0>()), pair(Const<1>()), pair(Const<2>()), pair(Const<3>());
}

// Theta partial of an interior node: sum_q Gb_q dc_{q xi}/dtheta D_xi F_q times
// dt / (2 dxi). With A = c xi_x and x_xi = L + 2 H cot eta, x_eta = H cot (2 xi - 1),
// dc_{q xi}/dtheta = e_y t1 - e_x t2, t2 = A 2 H eta xi_x dcot, t1 = t2 x_eta/H -
// A (2 xi - 1) dcot.
__device__ __forceinline__ double theta_partial(const CavDev &cv, const Geo &geo, const Mix64 &mix,
                                                int i, int j, const double *Gb, const double *F) {
  const double xe = geo.xeH[cv.goff + i];
  const double t2 = geo.ath2[cv.goff + j];
  const double t1 = fma(t2, xe, -geo.ath1[cv.goff + j] * geo.z[cv.goff + i]);
  const int64_t plane = cv.plane;
  const bool clo = i == 1, chi = i == cv.nx - 2;
  // k: dc/dtheta of the pair's first member; pos0, pos1: c >= 0 of either (both at c = 0)
  auto term = [&](int q0, bool pos0, bool pos1, double k, double r) {
    const double *F0 = F + q0 * plane, *F1 = F0 + 2 * plane;
    const double a = mix64(F0, pos0 ? 1 : -1, pos0 ? clo : chi, mix, F0[0]);
    const double b = mix64(F1, pos1 ? 1 : -1, pos1 ? clo : chi, mix, F1[0]);
    const double g0 = Gb[q0 * plane], g1 = Gb[(q0 + 2) * plane];
    return fma(fma(pos0 ? g0 : -g0, a, (pos1 ? -g1 : g1) * b), k, r);
  };
  const double xm = geo.xm[cv.goff + i], xp = geo.xp[cv.goff + i];
  double r = term(1, true, false, -t2, 0.0);
  r = term(2, nonpositive(xe), nonnegative(xe), t1, r);
  r = term(5, nonnegative(xm), nonpositive(xm), t1 - t2, r);
  return term(6, nonpositive(xp), nonnegative(xp), t1 + t2, r);
}

}  // namespace

// Seed of the kinetic-energy objective (Eq. 5.1) at state g: adjoint of g,
// zero adjoint of lambda, and the direct theta partial (slot 3).
__global__ void k_adj_seed_energy(AdjArgs a) {
  const Ref r = tile_ref(a.tile_cav, a.cav);
  const CavDev &cv = a.cav[r.cav];
  double dth = 0.0;
  if (r.valid) {
    const int64_t node = int64_t(r.j) * cv.pitch + r.i;
    const double *g = a.g + 9 * cv.off;
    double gg[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) gg[q] = g[q * cv.plane + node];
    double ux, uy, P;
    moments(gg, cv.c, cv.cs2, ux, uy, P);
    const double wx = ((r.i == 0 || r.i == cv.nx - 1) ? 0.5 : 1.0) * cv.dxi;
    const double wy = ((r.j == 0 || r.j == cv.ny - 1) ? 0.5 : 1.0) * cv.deta;
    const double J = a.geo.xxi[cv.goff + r.j] * cv.H;
    double *ag = a.adj_g + 9 * cv.off;
#pragma unroll
    for (int q = 0; q < 9; ++q)
      ag[q * cv.plane + node] = wx * wy * J * cv.c * (ex(q) * ux + ey(q) * uy);
    a.adj_lam[cv.off + node] = 0.0;
    const double dJ = 2.0 * cv.H * cv.H * (r.j * cv.deta) * cv.dcot;
    dth = 0.5 * wx * wy * dJ * (ux * ux + uy * uy);
  }
  double v[3] = {0.0, 0.0, dth};
  block_sum<3, TILE_X * TILE_Y / 32>(v, a.ppart, blockIdx.x);
}

// Seed of J = sum over cavities of psi(i*, j*), the stream function at one
// node per cavity (the primary eddy's node for J = psi_min). psi(i, j) =
// sum_{m <= j} w_m deta (u H - v x_eta(xi_i)) with trapezoid weights w_m
// (1/2 at m = 0 and m = j), so dJ/dg_q = w_m deta c (H e_qx - x_eta e_qy) on
// column i*, rows m <= j*, and zero elsewhere; theta enters directly through
// x_eta = H cot(theta) (2 xi - 1).
__global__ void k_adj_seed_psi(AdjArgs a) {
  const Ref r = tile_ref(a.tile_cav, a.cav);
  const CavDev &cv = a.cav[r.cav];
  double dth = 0.0;
  if (r.valid) {
    const int64_t node = int64_t(r.j) * cv.pitch + r.i;
    const int is = a.psi_nodes[2 * r.cav], js = a.psi_nodes[2 * r.cav + 1];
    double *ag = a.adj_g + 9 * cv.off;
    double w = 0.0;
    if (r.i == is && r.j <= js && js > 0) w = ((r.j == 0 || r.j == js) ? 0.5 : 1.0) * cv.deta;
    const double xe = a.geo.xeta[cv.goff + r.i];
#pragma unroll
    for (int q = 0; q < 9; ++q) ag[q * cv.plane + node] = w * cv.c * (cv.H * ex(q) - xe * ey(q));
    a.adj_lam[cv.off + node] = 0.0;
    if (w != 0.0) {
      const double *g = a.g + 9 * cv.off;
      double gg[9];
#pragma unroll
      for (int q = 0; q < 9; ++q) gg[q] = g[q * cv.plane + node];
      double ux, uy, P;
      moments(gg, cv.c, cv.cs2, ux, uy, P);
      dth = -w * uy * cv.H * (2.0 * r.i * cv.dxi - 1.0) * cv.dcot;
    }
  }
  double v[3] = {0.0, 0.0, dth};
  block_sum<3, TILE_X * TILE_Y / 32>(v, a.ppart, blockIdx.x);
}

// Column and row tables of the gathers and of the theta partial (Geo), and the
// cavity of every block of the step's kernels; one block per cavity.
__global__ void __launch_bounds__(256) k_adj_setup(const CavDev *cavs, Geo geo, int *adj_cav,
                                                   int *ring_cav) {
  const CavDev &cv = cavs[blockIdx.x];
  for (int i = threadIdx.x; i < cv.nx; i += 256) {
    const double xe = geo.xeH[cv.goff + i];
    const_cast<double *>(geo.xm)[cv.goff + i] = 1.0 - xe;
    const_cast<double *>(geo.xp)[cv.goff + i] = 1.0 + xe;
    const_cast<double *>(geo.z)[cv.goff + i] = 2.0 * (double(i) / (cv.nx - 1)) - 1.0;
  }
  for (int j = threadIdx.x; j < cv.ny; j += 256) {
    const double r = geo.ax[1][cv.goff + j] * cv.dcot;
    const_cast<double *>(geo.ath1)[cv.goff + j] = r;
    const_cast<double *>(geo.ath2)[cv.goff + j] =
        r * (2.0 * cv.H * (double(j) / (cv.ny - 1)) * geo.xix[cv.goff + j]);
  }
  for (int b = threadIdx.x; b < cv.nblk_adj; b += 256) adj_cav[cv.adj0 + b] = blockIdx.x;
  for (int b = threadIdx.x; b < cv.nblk_adj - cv.nblk_core; b += 256)
    ring_cav[cv.ring0 + b] = blockIdx.x;
}

// Threads per block NT and registers as in staged64.cu: up to 255 registers on
// small batches (8 blocks of a warp on an SM; 10, 12 and 14 blocks with fewer
// registers ran at 0.96-1.04 of its speed), 168 with 128 threads.
template <int NT>
constexpr int ADJ_BLOCKS = NT == 32 ? 8 : 3;

// Ring nodes: Gbar += X^T(sum of the wall nodes' adjoints), at g_{n+1}.
template <int NT>
__global__ void __launch_bounds__(NT, ADJ_BLOCKS<NT>) k_adj_ring(AdjArgs a) {
  const Node64 r = interior_node<NT>(a.ring_cav, a.cav, true);
  const CavDev &cv = a.cav[r.cav];
  const int64_t plane = cv.plane, b9 = 9 * cv.off, node = int64_t(r.j) * cv.pitch + r.i;
  previous_done();
  dependents_may_start();
  if (!r.valid) return;
  double *ag = a.adj_g + b9;
  const double *gn = a.gn + b9 + node;
  double w[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0}, h[9], F[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    F[q] = gn[q * plane];
    h[q] = ag[q * plane + node];
  }
  for (int k = 0; k < 3; ++k) {
    int wi, wj;
    if (!wall_of(cv, r.i, r.j, k, wi, wj)) continue;
    const double *wn = ag + int64_t(wj) * cv.pitch + wi;
#pragma unroll
    for (int q = 0; q < 9; ++q) w[q] += wn[q * plane];
  }
  const Mom64 m = moments64(F);
  wall_T(h, w, m.x, m.y);
#pragma unroll
  for (int q = 0; q < 9; ++q) ag[q * plane + node] = h[q];
}

// The full step's stencil and the half step's collision (interior nodes; the
// walls' FBARbar is zero and is not written).
template <int NT>
__global__ void __launch_bounds__(NT, ADJ_BLOCKS<NT>) k_adj_full(AdjArgs a) {
  const Node64 r = interior_node<NT>(a.adj_cav, a.cav, false);
  const CavDev &cv = a.cav[r.cav];
  const int64_t plane = cv.plane, off = cv.off, b9 = 9 * off;
  const int i = min(r.i, cv.nx - 2), j = min(r.j, cv.ny - 2);
  const int64_t node = int64_t(j) * cv.pitch + i;
  const Mix64 mix = cv.mix, mixe = cv.mixe[1];
  const double dt = cv.dt;
  previous_done();
  dependents_may_start();
  double dth[1] = {0.0};
  if (r.valid) {
    const double *ag = a.adj_g + b9, *fh = a.fh + b9 + node;
    double f[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) f[q] = fh[q * plane];
    const Mom64 m = moments64(f);                  // those of f-bar too (Eq. 2.17)
    // FHbar of the node (the rest plane is not advected); for a ring node then the
    // sum of its wall nodes' and their transposed wall rule
    double h[9], w[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 1
    for (int k = -1; k < (r.wall ? 3 : 0); ++k) {
      int gi = i, gj = j;
      if (k >= 0 && !wall_of(cv, i, j, k, gi, gj)) continue;
      Gather64 g = gather_at(cv, a.geo, 1, gi, gj);
      g.G = ag + int64_t(gj) * cv.pitch + gi;
      advect_T(g, a.geo, mix, mixe, w);
      if (k < 0)
#pragma unroll
        for (int q = 0; q < 9; ++q) {
          h[q] = w[q];
          w[q] = 0.0;
        }
    }
    if (r.wall) wall_T(h, w, m.x, m.y);
    // Eq. (2.17): f = ah f-bar + bh f^eq keeps u and P, so f^eq is that of f and
    // f-bar - f^eq = (f - f^eq) / ah; d ah / d lam = -d bh / d lam = 4 dt / (4 lam + dt)^2
    double geq[9], out[9];
    equilibrium64(m, geq);
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) s = fma(h[q], f[q] - geq[q], s);
    const double lam = a.lam[off + node];
    const double bh = dt * recip(fma(4.0, lam, dt));
    a.lamb2[off + node] = bh * recip(lam) * s;
    Adj64 b = equilibrium_T(h, m.x, m.y);
    b.x *= bh;
    b.y *= bh;
    b.p *= bh;
    moments_T(b, m.x, m.y, 1.0 - bh, h, out);
    double *fbarb = a.fbarb + b9 + node;
#pragma unroll
    for (int q = 0; q < 9; ++q) fbarb[q * plane] = out[q];
    dth[0] = -theta_partial(cv, a.geo, mix, i, j, ag + node, fh);
  }
  block_sum<1, NT / 32>(dth, a.pfull, blockIdx.x);
}

// The half step's stencil and the collision: the adjoint of (g_n, lambda_n).
template <int NT>
__global__ void __launch_bounds__(NT, ADJ_BLOCKS<NT>) k_adj_half(AdjArgs a) {
  const Node64 r = node_of<NT>(a.blk_cav, a.cav);
  const CavDev &cv = a.cav[r.cav];
  const int64_t plane = cv.plane, off = cv.off, b9 = 9 * off;
  const int i = min(r.i, cv.nx - 1), j = min(r.j, cv.ny - 1);
  const int64_t node = int64_t(j) * cv.pitch + i;
  const Mix64 mix = cv.mix, mixe = cv.mixe[0];
  Gather64 gt = gather_at(cv, a.geo, 0, i, j);
  const double dt = cv.dt;
  previous_done();
  dependents_may_start();
  double v[3] = {0.0, 0.0, 0.0};  // n, Re, theta
  if (r.valid) {
    const double *fbarb = a.fbarb + b9 + node;
    double *ag = a.adj_g + b9 + node;
    gt.G = fbarb;
    double B[9], P[9], d[9];      // FBbar, FPbar (f-hat^+ is read at interior nodes only)
#pragma unroll
    for (int q = 0; q < 9; ++q) B[q] = r.wall ? 0.0 : fbarb[q * plane];
    advect_T(gt, a.geo, mix, mixe, B);
    const double *gp = a.g + b9 + node;
    double g[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      P[q] = r.wall ? 0.0 : ag[q * plane];
      g[q] = gp[q * plane];
    }
    const Mom64 m = moments64(g);
    equilibrium64(m, d);
#pragma unroll
    for (int q = 0; q < 9; ++q) d[q] = g[q] - d[q];
    const double diag = (d[5] + d[6]) + (d[7] + d[8]);
    const double pxx = (d[1] + d[3]) + diag, pyy = (d[2] + d[4]) + diag;
    const double pxy = (d[5] - d[6]) + (d[7] - d[8]);
    const double pp = fma(pxx, pxx, fma(pyy, pyy, (pxy + pxy) * pxy));
    const double rD = recip(fma(2.0, a.lam_p[off + node], dt));
    const double q = cv.strain2 * pp * (rD * rD);       // |gamma-dot|^2 (k_collide64)
    const bool free = __double_as_longlong(q) > __double_as_longlong(cv.gmin2);
    const double lam = a.lam[off + node];
    const double i2 = recip(fma(2.0, lam, dt));
    const double bp = 2.0 * dt * i2, bb = 0.75 * bp;    // Eqs. (2.15)-(2.16)
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) s = fma(fma(4.0, P[k], 3.0 * B[k]), d[k], s);
    const double lb = a.adj_lam[off + node] + (r.wall ? 0.0 : a.lamb2[off + node]) +
                      dt * (i2 * i2) * s;
    // lam = K/c_s^2 max(q, gmin2)^m, m = (n-1)/2, K = U^(2-n) H^n / Re
    const double ll = lb * lam;
    v[0] = ll * fma(0.34657359027997265471, log2_fast(free ? q : cv.gmin2, a.powtab), cv.lnHU);
    v[1] = -ll * cv.inv_Re;
    // d lam / d q = m lam / q, q = strain2 pp / (2 lam_p + dt)^2
    const double lm = free ? ll * cv.half_nm1 : 0.0;
    const double e = free ? 2.0 * lm * recip(pp) : 0.0;
    const double xx = e * pxx, yy = e * pyy, xy = 2.0 * e * pxy, t = xx + yy;
    const double db[9] = {0.0, xx, yy, xx, yy, t + xy, t - xy, t + xy, t - xy};
    double gb[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double eb = fma(bp, P[k], bb * B[k]) - db[k];   // f^eq's adjoint
      gb[k] = (P[k] + B[k]) - eb;
      d[k] = eb;
    }
    const Adj64 b = equilibrium_T(d, m.x, m.y);
    double out[9];
    moments_T(b, m.x, m.y, 1.0, gb, out);
#pragma unroll
    for (int k = 0; k < 9; ++k) ag[k * plane] = out[k];
    a.adj_lam[off + node] = -4.0 * lm * rD;
    if (!r.wall) v[2] = -0.5 * theta_partial(cv, a.geo, mix, i, j, fbarb, a.fb + b9 + node);
  }
  block_sum<3, NT / 32>(v, a.phalf, blockIdx.x);
}

// Per cavity, by a cluster of CS blocks (k_residual_reduce): dparams[cav][0..2]
// += the sums of n3 triples of p3 and, for theta, of n1 values of p1, in a
// fixed order. The kernel has called cluster_arrive().
template <int CS>
__device__ __forceinline__ void reduce_params(const double *p3, int n3, const double *p1, int n1,
                                              double *dparams) {
  __shared__ double all[CS][3];
  const int r = blockIdx.x % CS;
  auto from = [&](int n, int b) { return int(int64_t(n) * b / CS); };
  double v[8] = {};
#pragma unroll 2
  for (int t = from(n3, r) + threadIdx.x; t < from(n3, r + 1); t += 256)
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] += p3[3 * int64_t(t) + k];
#pragma unroll 2
  for (int t = from(n1, r) + threadIdx.x; t < from(n1, r + 1); t += 256) v[2] += p1[t];
  __shared__ double sh[8][3];
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  const double s = warp_sums8(v);
  if ((l & 3) == 0 && l < 12) sh[w][l >> 2] = s;
  cluster_running<CS>();
  __syncthreads();
  if (threadIdx.x < 3) {
    double acc = 0.0;
    for (int k = 0; k < 8; ++k) acc += sh[k][threadIdx.x];
    cluster_at<CS>(&all[r][0])[threadIdx.x] = acc;
  }
  cluster_done<CS>();
  if (r == 0 && threadIdx.x < 3) {
    double acc = 0.0;
    for (int b = 0; b < CS; ++b) acc += all[b][threadIdx.x];
    dparams[threadIdx.x] += acc;
  }
}
__global__ void __launch_bounds__(256) k_adj_reduce_seed(AdjArgs a) {
  const CavDev &cv = a.cav[blockIdx.x];
  reduce_params<1>(a.ppart + 3 * int64_t(cv.tile0), cv.tiles_x * cv.tiles_y, nullptr, 0,
                   a.dparams + 3 * blockIdx.x);
}
template <int CS>
__global__ void __launch_bounds__(256) k_adj_reduce(AdjArgs a) {
  const CavDev &cv = a.cav[blockIdx.x / CS];
  cluster_arrive<CS>();
  previous_done();
  dependents_may_start();
  reduce_params<CS>(a.phalf + 3 * int64_t(cv.blk0), cv.nblk, a.pfull + cv.adj0, cv.nblk_adj,
                    a.dparams + 3 * (blockIdx.x / CS));
}

static const dim3 kT(TILE_X, TILE_Y);

void launch_adjoint_setup(const CavDev *cav, const Geo &geo, int *adj_cav, int *ring_cav, int ncav,
                          cudaStream_t s) {
  k_adj_setup<<<ncav, 256, 0, s>>>(cav, geo, adj_cav, ring_cav);
}

void launch_adjoint_seed(const AdjArgs &a, cudaStream_t s) {
  k_adj_seed_energy<<<a.ntiles, kT, 0, s>>>(a);
  k_adj_reduce_seed<<<a.ncav, 256, 0, s>>>(a);
}

void launch_adjoint_seed_psi(const AdjArgs &a, cudaStream_t s) {
  k_adj_seed_psi<<<a.ntiles, kT, 0, s>>>(a);
  k_adj_reduce_seed<<<a.ncav, 256, 0, s>>>(a);
}

void launch_adjoint_step(const AdjArgs &a, cudaStream_t s) {
  if (a.nt == 32) {
    launch_after(k_adj_ring<32>, a.nblk_ring, 32, 0, s, a);
    launch_after(k_adj_full<32>, a.nblk_adj, 32, 0, s, a);
    launch_after(k_adj_half<32>, a.nblk, 32, 0, s, a);
  } else {
    launch_after(k_adj_ring<128>, a.nblk_ring, 128, 0, s, a);
    launch_after(k_adj_full<128>, a.nblk_adj, 128, 0, s, a);
    launch_after(k_adj_half<128>, a.nblk, 128, 0, s, a);
  }
  if (a.most > REDUCE_ONE)
    launch_after(k_adj_reduce<REDUCE_CS>, a.ncav * REDUCE_CS, 256, 0, s, a, REDUCE_CS);
  else
    launch_after(k_adj_reduce<1>, a.ncav, 256, 0, s, a);
}

}  // namespace ifd
