// Fixed-point evaluation of the moments of the expansion over wavenumbers (expand64.cu, near.cu).
#pragma once

#include <math.h>

#include "expand64.h"

namespace bem {

constexpr int kAngles = 1024;
constexpr long long kOne = 1ll << 62;

struct Split {   // x = h 2^32 + l, both signed
  int h, l;
};
__device__ __forceinline__ Split split(long long x) {
  return Split{(int)((x + 0x80000000ll) >> 32), (int)x};
}
// a b 2^-64 to about a unit, plus add; |a|, |b| <= 2^62
__device__ __forceinline__ long long mulh(Split a, Split b, long long add = 0) {
  const long long m = (long long)a.h * b.l + ((long long)a.l * b.h + 0x80000000ll);
  return (long long)a.h * b.h + add + (m >> 32);
}
// round(v 2^(62 - e)), 0 <= v < 2^e (or = 2^e)
__device__ __forceinline__ long long fixed62(double v, int e) {
  const unsigned long long bits = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
  const int be = (int)(bits >> 52);
  const long long m = (long long)((bits & 0xFFFFFFFFFFFFFull) | (be ? 0x10000000000000ull : 0ull));
  const int sh = max(be, 1) - 1013 - e;
  if (sh >= 0) return m << min(sh, 10);
  return sh > -63 ? (m + (1ll << (-sh - 1))) >> -sh : 0;
}
// a 2^(e - 60), rounded to FP64
__device__ __forceinline__ double from_fixed60(long long a, int e) {
  if (a == 0) return 0.0;
  const unsigned long long u = (unsigned long long)llabs(a);
  const int lz = __clzll((long long)u);
  const int be = 1023 + 3 - lz + e;
  if (be < 1 || be > 2045) return ldexp((double)a, e - 60);
  // 53 bits at the top, rounded half up; a carry runs into the exponent
  const unsigned long long m = ((u << lz) >> 10) + 1;
  return __longlong_as_double((long long)((((unsigned long long)(be - 1) << 52) + (m >> 1)) |
                                          ((unsigned long long)a & 0x8000000000000000ull)));
}

// cos and sin (62 fractional bits) of the angle phi 2^-64 turns.
__device__ __forceinline__ void fixed_sincos(unsigned long long phi, const int4* table, long long& co,
                                             long long& si) {
  const unsigned q = (unsigned)((phi + (1ull << 53)) >> 54);   // (mod kAngles below)
  const long long d = (long long)(phi - ((unsigned long long)q << 54));   // |d| <= 2^53
  constexpr long long kTwoPi = 0x3243F6A8885A308Dll;    // 2 pi 2^59
  constexpr long long kTwoThirds = 0x2AAAAAAAAAAAAAABll;   // 2 / 3 2^62
  const long long th = mulh(split(d << 9), split(kTwoPi)) << 2;   // t 2^70
  const Split t = split(th);
  const long long u = mulh(t, t);                        // t^2 2^76
  const int u47 = (int)(u >> 29);                        // t^2 2^47
  const int f62 = (int)(((long long)u47 * u47) >> 32);   // t^4 2^62
  // t^2 / 6 - t^4 / 120 in 2^-81
  const long long v = (mulh(split(u), split(kTwoThirds)) - (((long long)f62 * 572662306) >> 22)) << 5;
  const Split sn = split(th - (mulh(t, split(v)) >> 17));                       // sin t 2^70
  const Split cm = split((u << 1) - (((long long)f62 * 357913941) >> 17));      // (1 - cos t) 2^78
  const int4 e = table[q % kAngles];
  const Split C{e.x, e.y}, S{e.z, e.w};
  co = (((long long)e.x << 32) + e.y) - (((mulh(C, cm) >> 8) + mulh(S, sn)) >> 6);
  si = (((long long)e.z << 32) + e.w) - (((mulh(S, cm) >> 8) - mulh(C, sn)) >> 6);
}

// 1 / sqrt(r2) and sqrt(r2) from the FP32 root y by one step of Householder's third-order iteration,
// (1 - e)^(-1/2) = 1 + e / 2 + 3 e^2 / 8 + .. with e = 1 - r2 y^2 below 2^-20.8; both to 1.6 units of
// 2^-53.
__device__ __forceinline__ void root_and_inverse(double r2, double& r, double& ri) {
  const float rf = (float)r2;
  if (rf < 1e-30f && r2 == 0.0) {   // coinciding points: k-derivatives have a value there
    r = 0.0;
    ri = INFINITY;
    return;
  }
  const double y = rf > 1e-30f && rf < 1e30f ? (double)rsqrtf(rf) : rsqrt(r2);
  const double t = r2 * y, er = fma(-t, y, 1.0), pe = fma(0.375, er, 0.5);
  r = fma(t * er, pe, t);
  ri = fma(y * er, pe, y);
}

template <int kKind>
constexpr int kFamilies = kKind == kDouble ? 2 : 1;

// The families' weights at a point of weight wq, distance r (ri = 1 / r) and dn = (y - x).n, with the
// factor e^{-ci r} of a complex centre.
template <int kKind>
__device__ __forceinline__ void moment_weights(double (&w)[kFamilies<kKind>], double wq, double r, double ri,
                                               double dn, double ci) {
  double g = kKind == kSingleDeriv ? wq : wq * ri;
  if (ci != 0.0) g *= exp(-ci * r);
  if (kKind == kDouble) {
    w[0] = g * ri * ri * dn;
    w[kFamilies<kKind> - 1] = g * ri * dn;
  } else {
    w[0] = kKind == kDoubleDeriv ? g * dn : g;
  }
}

// acc[f][m] += b_f e^{i phase} T_m(2 rho - 1) in units of 2^-60 of b's scale; b_f and rho as
// 62-bit fractions.
template <int MT, int F>
__device__ __forceinline__ void add_moments(long long (&ar)[F][MT], long long (&ai)[F][MT],
                                            const long long (&b)[F], long long rho, Split K, int kb,
                                            const int4* table) {
  long long co, si;
  fixed_sincos((unsigned long long)mulh(split(rho), K) << (4 + kb), table, co, si);
  const Split sc = split(co), ss = split(si);
  Split br[F], bi[F];
#pragma unroll
  for (int f = 0; f < F; ++f) {
    const Split sb = split(b[f]);
    const long long r0 = mulh(sb, sc), i0 = mulh(sb, ss);   // T_0's terms
    ar[f][0] += r0;
    ai[f][0] += i0;
    br[f] = split(r0 << 2);
    bi[f] = split(i0 << 2);
  }
  const long long x = 2 * rho - kOne;
  const Split sx = split(x);
  long long t0 = kOne, t1 = x;
#pragma unroll
  for (int m = 1; m < MT; ++m) {
    const Split t = split(t1);
#pragma unroll
    for (int f = 0; f < F; ++f) {
      ar[f][m] = mulh(br[f], t, ar[f][m]);
      ai[f][m] = mulh(bi[f], t, ai[f][m]);
    }
    const long long t2 = (mulh(sx, t) << 3) - t0;
    t0 = t1;
    t1 = t2;
  }
}

}  // namespace bem
