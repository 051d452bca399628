// What the column passes share: the op's scalars in the working precision, 1 / |k|^2, and the reductions of the
// dynamic closures.
//
// On this GPU an FP64 instruction holds its quarter of an SM for 64 cycles at best (half a lane a cycle, 1.26 TFLOP/s;
// chains of independent FMAs reach 1.06, one instruction in 76), a conversion to or from FP64 included, so the FP32
// passes take their scalars ready converted, read 1 / |k|^2 of the smallest wavenumbers (inverted in FP64) from a table,
// and keep the FP64 sums short: the two Germano sums share every instruction (one per half warp), and all warps of a
// CTA add up the partial sums where one warp did.
#pragma once

#include <cmath>

#include "qg_kernels.h"

namespace qg {

constexpr int kIk2Small = 16;  // FP32: 1 / |k|^2 up to this |m|^2 is inverted in FP64 before rounding
template <typename T> struct ColScalars {
  T ks, ks2, dt, a, b, beta, U, coeff, rpow, inv_eta, nu, mu, visc_mu, scale;
  T scale_lo;  // FP64: 1 / N^2 less its rounding (the same sign in every step), 0 for N = 2^a
  T ik2s[kIk2Small + 1];
};
template <typename T> ColScalars<T> col_scalars(const Geom& g, const ColDesc& d) {
  ColScalars<T> s;
  const double ks2 = g.kscale * g.kscale;
  s.ks = T(g.kscale);
  s.ks2 = T(ks2);
  s.dt = T(d.dt);
  s.a = T(d.a);
  s.b = T(d.b);
  s.beta = T(d.beta);
  s.U = T(d.U);
  s.coeff = T(d.coeff);
  s.rpow = T(d.rpow);
  s.inv_eta = T(d.inv_eta);
  s.nu = T(d.nu);
  s.mu = T(d.mu);
  s.visc_mu = T(d.visc_mu);
  const double n2 = double(g.n) * double(g.n), inv = 1.0 / n2;
  s.scale = T(inv);
  s.scale_lo = sizeof(T) == 8 ? T(-std::fma(inv, n2, -1.0) * inv) : T(0);
  s.ik2s[0] = T(0);
  for (int m = 1; m <= kIk2Small; ++m) s.ik2s[m] = T(1.0 / (ks2 * double(m)));
  return s;
}
// 1 / |k|^2 of the integer |m|^2, 0 for the mean mode
template <typename T> __device__ __forceinline__ T inv_k2(const ColScalars<T>& s, int m2) {
  return m2 <= kIk2Small ? s.ik2s[m2] : T(1) / (s.ks2 * T(m2));
}

// Sums of hm and mm over the CTA (nw <= 32 warps), in a fixed order: red[0][0] and red[1][0] after the call's last
// barrier.  Every thread of the CTA calls it.
__device__ __forceinline__ void pair_sum(double hm, double mm, double (*red)[32], int nw) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool up = lane >= 16;
  // the lower half warp goes on with hm, the upper one with mm
  double v = (up ? mm : hm) + __shfl_xor_sync(0xffffffffu, up ? hm : mm, 16);
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((lane & 15) == 0) red[up][wid] = v;
  __syncthreads();
  if (wid == 0) {
    v = 0.0;
    for (int i = lane & 15; i < nw; i += 16) v += red[up][i];
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncwarp();
    if ((lane & 15) == 0) red[up][0] = v;
    __syncwarp();
  }
}

// C = max(0, <HM> / <MM>) (0 if <MM> = 0) from the column CTAs' partial sums, the same value in every CTA; all nt
// threads call it.  stop: leave instead (a uniform decision on any thread's flag); the loads overlap its load.
__device__ __forceinline__ bool germano_coefficient(const double* partials, int n, double (*red)[32], int nt, int stop,
                                                    double* out, int* st) {
  double hm = 0.0, mm = 0.0;
  for (int i = threadIdx.x; i < n; i += nt) {
    hm += QG_LD(partials, 2 * i, 2 * n, st);
    mm += QG_LD(partials, 2 * i + 1, 2 * n, st);
  }
  if (__syncthreads_or(stop)) return false;
  pair_sum(hm, mm, red, (nt + 31) >> 5);
  if (threadIdx.x == 0) {
    const double a = red[0][0], b = red[1][0];
    const double c = b > 0.0 ? fmax(0.0, a / b) : 0.0;
    red[0][0] = c;
    if (blockIdx.x == 0 && out) *out = c;
  }
  __syncthreads();
  return true;
}

}  // namespace qg
