// Per-marker pieces of the IB transfers shared by the step's kernels and the
// stand-alone point operators: the stencil of Eq. 14 along one axis and the
// moments (Eq. 11) of one node's post-streaming populations.
#pragma once

#include "df.cuh"
#include "lbm_gather.cuh"
#include "stencil_fixed.cuh"

namespace ibl {

// Eq. 14 at the four nodes around a point at s past its floor node.
__device__ __forceinline__ void cosine_weights(double s, double w[4]) {
  double sn, cs;
  sincospi(0.5 * s, &sn, &cs);
  w[0] = 0.25 * (1.0 - sn);
  w[1] = 0.25 * (1.0 + cs);
  w[2] = 0.25 * (1.0 + sn);
  w[3] = 0.25 * (1.0 - cs);
}

// Eq. 14 at the four nodes base..base+3 of one axis for a point at x.  With
// s = x - floor(x) the nodes sit at |r| = 1+s, s, 1-s, 2-s, whose
// cos(pi |r| / 2) are -sin, cos, sin, -cos of (pi s / 2).  A periodic axis
// reduces the base into [0, n) so that node offsets wrap once at most.  On a
// bounded axis a stencil that leaves [0, n), or a non-finite x, returns false
// and the base is clamped into [0, n - 4], so that no later access leaves the
// arrays (n >= 8 on every axis that carries points).
__device__ __forceinline__ bool stencil_axis(double x, int n, bool per, int& base, double w[4]) {
  const bool finite = isfinite(x);
  const double xx = finite ? x : 0.0;
  const double fl = floor(xx);
  cosine_weights(xx - fl, w);
  if (per) {
    double r = fmod(fl - 1.0, (double)n);
    if (r < 0.0) r += (double)n;
    base = (int)r;
    return finite;
  }
  base = (int)fmin(fmax(fl - 1.0, 0.0), (double)(n - 4));
  return finite && fl - 1.0 >= 0.0 && fl + 2.0 < (double)n;
}

// Floor and position between nodes of x (split_bits); false for |x| >= 2^31 and
// non-finite x, which take the FP64 route (stencil_axis).
__device__ __forceinline__ bool split_coordinate(double x, long long& fl, long long& t) {
  return split_bits((unsigned long long)__double_as_longlong(x), fl, t);
}

// A weight in units of 2^-60 (at most 1/2) as a double-float: pieces of 24, 24
// and 12 bits, the low part rounded once.
__device__ __forceinline__ df df_from_fixed(long long w) {
  const float h = __fmul_rn((float)(int)(w >> 36), 0x1p-24f);
  const float m = __fmul_rn((float)(int)((w >> 12) & 0xffffff), 0x1p-48f);
  const float l = __fmul_rn((float)(int)(w & 0xfff), 0x1p-60f);
  const df s = fast_two_sum(h, m);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, l));
}

// The four weights as double-floats (fixed_weights).  Against 64-bit-mantissa
// arithmetic at 2e4 positions they err by at most 4.4e-16 (root mean square
// 1.43e-16), the FP64 formula rounded to double-float by 5.1e-16 (1.46e-16), and
// a polynomial in double-float by 2.3e-15 (4e-16).
__device__ __forceinline__ void weights_df(long long t, df w[4]) {
  long long f[4];
  fixed_weights(t, f);
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = df_from_fixed(f[k]);
}

// First stencil node of one axis, wrapped into [0, n) on a periodic axis;
// false if the stencil leaves a bounded axis or x is not finite (the base is
// then clamped as stencil_axis does).
__device__ __forceinline__ bool first_node(double x, int n, bool per, int& base, long long& t) {
  long long fl;
  if (!split_coordinate(x, fl, t)) {
    double w[4];
    t = 0;
    return stencil_axis(x, n, per, base, w);
  }
  long long b = fl - 1;
  if (per) {
    if (b < 0 || b >= n) {
      b %= n;
      if (b < 0) b += n;
    }
    base = (int)b;
    return true;
  }
  base = (int)(b < 0 ? 0 : (b > n - 4 ? n - 4 : b));
  return b >= 0 && fl + 2 < n;
}

// Eq. 14's stencil of a point at x on one axis: first node (as stencil_axis)
// and double-float weights; EXACT64: the weights by the FP64 formula.
template <bool EXACT64>
__device__ __forceinline__ bool axis_stencil(double x, int n, bool per, int& base, df w[4]) {
  long long fl, t;
  if (!split_coordinate(x, fl, t)) {
    double wd[4];
    const bool ok = stencil_axis(x, n, per, base, wd);
    for (int k = 0; k < 4; ++k) w[k] = df_from_double(wd[k]);
    return ok;
  }
  if (EXACT64) {
    double wd[4];
    // fl, not floor(x): for x in (-2^-64, 0) the split rounds to node 0, where
    // x - floor(x) rounds to 1, a node further on
    cosine_weights(x - (double)fl, wd);
    for (int k = 0; k < 4; ++k) w[k] = df_from_double(wd[k]);
  } else {
    weights_df(t, w);
  }
  return first_node(x, n, per, base, t);
}

// Fused multiply-add rounded once, with no room for the compiler to round
// differently in different kernels (the point operators compute a node's
// moments either inside the interpolation or once per cell beforehand, and
// both must give the same bits).
__device__ __forceinline__ float rn_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rn_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// drho and u* of one node from its post-streaming deviations, in the
// storage's compute precision (Eq. 11 with the uniform body force G:
// u* = (m + G/2) / rho, formed as m - m drho / rho).
template <int Q, class R>
__device__ __forceinline__ void moments_of(const R gg[Q], const FluidParams<R>& p, R& drho_out, R u[3]) {
  R drho = gg[0], m0 = R(0), m1 = R(0), m2 = R(0);
#pragma unroll
  for (int e = 1; e < Q; e += 2) {
    drho += gg[e] + gg[e + 1];
    const R d = gg[e] - gg[e + 1];
    if (Lat<Q>::cx(e)) m0 += R(Lat<Q>::cx(e)) * d;
    if (Lat<Q>::cy(e)) m1 += R(Lat<Q>::cy(e)) * d;
    if (Lat<Q>::cz(e)) m2 += R(Lat<Q>::cz(e)) * d;
  }
  const R qd = drho / (R(1) + drho);
  R u0 = rn_fma(R(0.5), p.G[0], m0), u1 = rn_fma(R(0.5), p.G[1], m1), u2 = rn_fma(R(0.5), p.G[2], m2);
  u0 = rn_fma(-u0, qd, u0);
  u1 = rn_fma(-u1, qd, u1);
  u2 = rn_fma(-u2, qd, u2);
  drho_out = drho;
  u[0] = u0;
  u[1] = u1;
  u[2] = u2;
}

template <int Q, class T, bool PULL>
__device__ __forceinline__ void node_moments(const T* __restrict__ src, int x, int y, int z,
                                             const FluidParams<typename Store<T>::R>& p,
                                             typename Store<T>::R& drho_out, typename Store<T>::R u[3]) {
  typename Store<T>::R gg[Q];
  pull_cell<Q, T, PULL>(src, x, y, z, p, gg);
  moments_of<Q, typename Store<T>::R>(gg, p, drho_out, u);
}

// A storage-precision value as a double-float (exact).
__device__ __forceinline__ df to_df(float v) { return df_from_float(v); }
__device__ __forceinline__ df to_df(double v) { return df_from_double(v); }

}  // namespace ibl
