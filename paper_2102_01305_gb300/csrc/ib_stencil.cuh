// Per-marker pieces of the IB transfers shared by the step's kernels and the
// stand-alone point operators: the stencil of Eq. 14 along one axis and the
// moments (Eq. 11) of one node's post-streaming populations.
#pragma once

#include "df.cuh"
#include "lbm_gather.cuh"

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

// First stencil node of a point at x on one axis and the position between
// nodes, x - floor(x) - 1/2, as a 64-bit signed fraction (units of 2^-64), in
// integer arithmetic on the bits of x: FP64 instructions issue at about 1/64
// of the FP32 rate here.  False for |x| >= 2^31 and non-finite x, which take
// the FP64 route (stencil_axis).
__device__ __forceinline__ bool split_coordinate(double x, long long& fl, long long& t) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((bits >> 52) & 0x7ff) - 1023;
  if (e >= 31) return false;
  const unsigned long long mant = (bits & 0xfffffffffffffull) | (e > -1023 ? 0x10000000000000ull : 0ull);
  long long ip = e >= 0 ? (long long)(mant >> (52 - e)) : 0;
  const int sh = e + 12;
  // fraction in units of 2^-64 (the integer bits leave the word)
  unsigned long long f = sh >= 0 ? mant << sh : (sh > -64 ? mant >> -sh : 0ull);
  if (bits >> 63) {
    ip = -ip - (f != 0 ? 1 : 0);
    f = 0ull - f;
  }
  fl = ip;
  t = (long long)(f ^ 0x8000000000000000ull);
  return true;
}

// The four weights of Eq. 14 from t = s - 1/2 (s = x - floor(x)) in
// double-float arithmetic.  The nodes sit at |r| = 1+s, s, 1-s, 2-s, and with
// p = pi t / 2 (|p| <= pi/4) the weights are 1/4 -/+ k (cos p + sin p) and
// 1/4 +/- k (cos p - sin p), k = sqrt(2)/8.  k cos p and k sin p are the Taylor
// polynomials in t^2 through p^16 and p^15 (remainder below 1e-17), the terms
// below 1e-8 summed in FP32, the others in double-float.  Against 80-bit
// arithmetic on 4e5 positions the weights are within 2.3e-15 (root mean square 4e-16; the
// FP64 formula rounded to double-float: 4.9e-16 and 2e-16): under the products'
// own rounding, and far under the spreading's resolution (1.4e-14) and FP32
// storage.  FP64 storage keeps the FP64 formula for its interpolation.
__device__ __forceinline__ df horner_step(df y, df p, df c) {
  // c + y p with |y p| <= 0.32 |c|
  const float q = __fmul_rn(y.hi, p.hi);
  float e = fmaf(y.hi, p.hi, -q);
  e = fmaf(y.hi, p.lo, e);
  e = fmaf(y.lo, p.hi, e);
  const float s = __fadd_rn(c.hi, q);
  const float r = __fsub_rn(q, __fsub_rn(s, c.hi));
  return fast_two_sum(s, __fadd_rn(r, __fadd_rn(e, c.lo)));
}

__device__ __forceinline__ df quarter_plus(df a) {
  // 1/4 + a with |a| <= 1/4
  const float s = __fadd_rn(0.25f, a.hi);
  const float e = __fsub_rn(a.hi, __fsub_rn(s, 0.25f));
  return fast_two_sum(s, __fadd_rn(e, a.lo));
}

__device__ __forceinline__ void weights_df(long long t64, df w[4]) {
  const float h = (float)(int)(t64 >> 40), l = (float)(int)((t64 >> 16) & 0xffffff), r = (float)(int)(t64 & 0xffff);
  const df t = fast_two_sum(__fmul_rn(h, 0x1p-24f), fmaf(r, 0x1p-64f, __fmul_rn(l, 0x1p-48f)));
  const df y = df_mul(t, t);
  // k sin(pi t / 2) = t P(y)
  float u = fmaf(-0x1.03fcf0p-33f, y.hi, 0x1.59be1ep-27f);
  u = fmaf(u, y.hi, -0x1.558d82p-21f);
  df p = horner_step(y, df_make(u, 0.f), df_make(0x1.dbd6fep-16f, -0x1.52a032p-41f));
  p = horner_step(y, p, df_make(-0x1.b1e9f4p-11f, 0x1.66adc2p-36f));
  p = horner_step(y, p, df_make(0x1.cda106p-7f, 0x1.c1070cp-34f));
  p = horner_step(y, p, df_make(-0x1.d3ba5cp-4f, -0x1.c5f47ep-32f));
  p = horner_step(y, p, df_make(0x1.1c5832p-2f, -0x1.48a746p-28f));
  const df s = df_mul(t, p);
  // k cos(pi t / 2) = Q(y)
  u = fmaf(0x1.986366p-37f, y.hi, -0x1.36567ep-30f);
  u = fmaf(u, y.hi, 0x1.65ac58p-24f);
  u = fmaf(u, y.hi, -0x1.2afa9ep-18f);
  df c = horner_step(y, df_make(u, 0.f), df_make(0x1.54cb90p-13f, -0x1.5f0bbap-38f));
  c = horner_step(y, c, df_make(-0x1.e36ab0p-9f, -0x1.827174p-34f));
  c = horner_step(y, c, df_make(0x1.6f5a4ap-5f, -0x1.35a078p-31f));
  c = horner_step(y, c, df_make(-0x1.bea5b6p-3f, -0x1.cac988p-33f));
  c = horner_step(y, c, df_make(0x1.6a09e6p-3f, 0x1.9fcef4p-29f));
  const df a = df_add(c, s), b = df_sub(c, s);   // k (cos + sin), k (cos - sin)
  w[0] = quarter_plus(df_neg(a));
  w[1] = quarter_plus(b);
  w[2] = quarter_plus(a);
  w[3] = quarter_plus(df_neg(b));
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
__device__ __forceinline__ void node_moments(const T* __restrict__ src, int x, int y, int z, long long cell,
                                             const FluidParams<typename Store<T>::R>& p,
                                             typename Store<T>::R& drho_out, typename Store<T>::R u[3]) {
  using R = typename Store<T>::R;
  R gg[Q];
  gather_q<Q, T, PULL, R>(src, x, y, z, cell, p, gg);
  moments_of<Q, R>(gg, p, drho_out, u);
}

// node_moments with the short pull (the same populations, and so the same bits).
template <int Q, class T, bool PULL>
__device__ __forceinline__ void node_moments_fast(const T* __restrict__ src, int x, int y, int z,
                                                  const FluidParams<typename Store<T>::R>& p,
                                                  typename Store<T>::R& drho_out, typename Store<T>::R u[3]) {
  typename Store<T>::R gg[Q];
  pull_cell<Q, T, PULL>(src, x, y, z, p, gg);
  moments_of<Q, typename Store<T>::R>(gg, p, drho_out, u);
}

// The same moments as FP64 rho and u*.
template <int Q, class T, bool PULL>
__device__ __forceinline__ void node_rho_u(const T* __restrict__ src, int x, int y, int z, long long cell,
                                           const FluidParams<typename Store<T>::R>& p, double& rho,
                                           double u[3]) {
  typename Store<T>::R drho, uu[3];
  node_moments<Q, T, PULL>(src, x, y, z, cell, p, drho, uu);
  rho = 1.0 + (double)drho;
  u[0] = (double)uu[0];
  u[1] = (double)uu[1];
  u[2] = (double)uu[2];
}

// A storage-precision value as a double-float (exact).
__device__ __forceinline__ df to_df(float v) { return df_from_float(v); }
__device__ __forceinline__ df to_df(double v) { return df_from_double(v); }

}  // namespace ibl
