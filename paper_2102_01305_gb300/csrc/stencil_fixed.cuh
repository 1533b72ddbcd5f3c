// Stencil position and delta weights (Eq. 14) of a coordinate in 64-bit integer
// arithmetic: FP64 instructions issue at about 1/64 of the FP32 rate on this
// GPU, and 64 bits hold more than FP64 does.  Plain integer code, which a host
// compiler takes too.
#pragma once

#ifdef __CUDACC__
#define IBL_HD __host__ __device__ __forceinline__
#else
#define IBL_HD inline
#endif

namespace ibl {

// First node's floor and the position between nodes, x - floor(x) - 1/2, as a
// 64-bit signed fraction (units of 2^-64), from the bits of x.  False for
// |x| >= 2^31 and non-finite x.  For x in (-2^-64, 0), whose fraction has no
// bits left in the word, the floor is 0.
IBL_HD bool split_bits(unsigned long long bits, long long& fl, long long& t) {
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

IBL_HD unsigned long long mulhi64(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (unsigned long long)((unsigned __int128)a * b >> 64);
#endif
}
IBL_HD unsigned mulhi32(unsigned a, unsigned b) { return (unsigned)((unsigned long long)a * b >> 32); }

// The four weights in units of 2^-60 from t = s - 1/2, s = x - floor(x).  The
// nodes sit at |r| = 1+s, s, 1-s, 2-s, and with p = pi t / 2 (|p| <= pi/4) the
// weights are 1/4 -/+ k (cos p + sin p) and 1/4 +/- k (cos p - sin p), k =
// sqrt(2)/8.  k cos p and k sin p are the Taylor polynomials in (2t)^2 through
// p^18 and p^17 (remainder under two units of 2^-66), coefficients k (pi/4)^n /
// n! in units of 2^-66; the terms from p^11 on fit 32 bits.  Every step drops
// less than one unit, so a weight is within 2^-60 of the exact one (the FP64
// formula: 2^-54), the weights of a point on a node are exactly 1/4, 1/2, 1/4
// and 0, and each pair of opposite weights sums to 1/2.
IBL_HD void fixed_weights(long long t, long long w[4]) {
  const unsigned long long m = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;   // |2t|, 2^-63
  const unsigned long long mh = mulhi64(m, m), ml = m * m;
  const unsigned long long y = mh >> 62 ? ~0ull : mh << 2 | ml >> 62;                          // (2t)^2, 2^-64
  const unsigned yh = (unsigned)(y >> 32);
  unsigned r = 0x40ff4u - mulhi32(0x25cu, yh);
  r = 0x566f877u - mulhi32(r, yh);
  unsigned long long q = 0x5563609deull - mulhi32(r, yh);
  q = 0x3b7adfaad60ull - mulhi64(q, y);
  q = 0x1b1e9f34ca91full - mulhi64(q, y);
  q = 0x7368418e083860ull - mulhi64(q, y);
  q = 0xe9dd2e0e2fa3eefull - mulhi64(q, y);
  q = 0x8e2c18d6eb17214full - mulhi64(q, y);
  const long long sn = (long long)(mulhi64(q, m) >> 1);   // k |sin p|, 2^-64
  r = 0x330cu - mulhi32(0x1au, yh);
  r = 0x4d95a0u - mulhi32(r, yh);
  r = 0x596b1624u - mulhi32(r, yh);
  q = 0x4abea760deull - mulhi32(r, yh);
  q = 0x2a9971ea0f44ull - mulhi64(q, y);
  q = 0xf1b558609c5cfull - mulhi64(q, y);
  q = 0x2deb493652fc3c4ull - mulhi64(q, y);
  q = 0x37d4b6c0e564c456ull - mulhi64(q, y);
  q = 0xb504f333f9de6484ull - mulhi64(q, y);
  const long long cs = (long long)(q >> 2);               // k cos p, 2^-64
  const long long si = t < 0 ? -sn : sn;
  const long long a = (cs + si + 8) >> 4, b = (cs - si + 8) >> 4, quarter = 1ll << 58;
  w[0] = quarter - a;
  w[1] = quarter + b;
  w[2] = quarter + a;
  w[3] = quarter - b;
}

}  // namespace ibl
