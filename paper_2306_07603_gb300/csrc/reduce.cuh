// Fixed-order block reductions of the residual partials of Eq. (2.19) and
// Eq. (5.1), shared by the step kernels and the stateless residual.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "internal.h"

namespace ifd {

struct Partial {
  double du2, u2, dP2, P2, ek, du2max, u2max;
};

// Sums of eight values over a warp, value k in lane 4 k: at each of the first
// three exchanges a lane hands over half of the values it still carries, so
// that it takes 9 FP64 additions (eight separate shuffle sums take 40; FP64
// instructions are what a reduction costs on GB300).
__device__ __forceinline__ double warp_sums8(const double v[8]) {
  const int lane = threadIdx.x + threadIdx.y * blockDim.x;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  double a[4], c[2];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    a[k] = (b4 ? v[k + 4] : v[k]) + __shfl_xor_sync(0xffffffffu, b4 ? v[k] : v[k + 4], 16);
#pragma unroll
  for (int k = 0; k < 2; ++k)
    c[k] = (b3 ? a[k + 2] : a[k]) + __shfl_xor_sync(0xffffffffu, b3 ? a[k] : a[k + 2], 8);
  double s = (b2 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, b2 ? c[0] : c[1], 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// fmax of values that are >= 0 or NaN, on the bits: those of a double >= 0 order
// as integers, and a NaN (ignored unless every value is one) counts as -1, the
// bits of a NaN.
__device__ __forceinline__ long long max_key(double v) {
  const long long b = __double_as_longlong(v);
  return (b & 0x7FFFFFFFFFFFFFFFll) > 0x7FF0000000000000ll ? -1ll : b;
}
__device__ __forceinline__ long long warp_max_key(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Reduction of the residual partials over a block of NWARPS warps (fixed
// order), into out[0..6] by its first 7 threads; every thread calls it.
template <int NWARPS>
__device__ __forceinline__ void block_reduce(const Partial &p, double *out) {
  __shared__ double sh[NWARPS][7];
  const int lane = threadIdx.x + threadIdx.y * blockDim.x;
  const int w = lane >> 5, l = lane & 31;
  const double v[8] = {p.du2, p.u2, p.dP2, p.P2, p.ek, 0.0, 0.0, 0.0};
  const double s = warp_sums8(v);
  const long long m0 = warp_max_key(max_key(p.du2max)), m1 = warp_max_key(max_key(p.u2max));
  if ((l & 3) == 0 && l < 20) sh[w][l >> 2] = s;
  if (l == 20) sh[w][5] = __longlong_as_double(m0);
  if (l == 24) sh[w][6] = __longlong_as_double(m1);
  __syncthreads();
  if (lane < 7) {
    double acc = sh[0][lane];
    for (int k = 1; k < NWARPS; ++k) acc = lane < 5 ? acc + sh[k][lane] : fmax(acc, sh[k][lane]);
    out[lane] = acc;
  }
}

// ... into slot `slot` of the partials.
template <int NWARPS>
__device__ __forceinline__ void block_partial(const Partial &p, double *part, int slot) {
  block_reduce<NWARPS>(p, part + int64_t(slot) * NPART);
}

// The partials of slots t, t + step, ... < nslots of one thread.
__device__ __forceinline__ Partial sum_slots(const double *part, int t, int step, int nslots) {
  Partial p = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 2
  for (int s = t; s < nslots; s += step) {
    const double *pp = part + int64_t(s) * NPART;
    p.du2 += pp[0];
    p.u2 += pp[1];
    p.dP2 += pp[2];
    p.P2 += pp[3];
    p.ek += pp[4];
    p.du2max = __longlong_as_double(max(max_key(p.du2max), max_key(pp[5])));
    p.u2max = __longlong_as_double(max(max_key(p.u2max), max_key(pp[6])));
  }
  return p;
}

// out[0] = E(u), out[1] = E(P) (Eq. 2.19), out[2] = the max-norm velocity
// residual, out[3] = the kinetic energy (Eq. 5.1) from the reduced partials r.
__device__ __forceinline__ void residual_of(const double *r, double *out) {
  out[0] = sqrt(r[0]) / sqrt(r[1]);
  out[1] = sqrt(r[2]) / sqrt(r[3]);
  out[2] = sqrt(r[5]) / sqrt(r[6]);
  out[3] = r[4];
}

// One block of NWARPS warps: reduces slots [0, nslots) of `part` in an order
// that depends only on nslots and the block size, and writes the residuals.
template <int NWARPS>
__device__ __forceinline__ void reduce_partials_block(const double *part, int nslots, double *out) {
  __shared__ double r[7];
  block_reduce<NWARPS>(sum_slots(part, threadIdx.x, NWARPS * 32, nslots), r);
  __syncthreads();
  if (threadIdx.x == 0) residual_of(r, out);
}

}  // namespace ifd
