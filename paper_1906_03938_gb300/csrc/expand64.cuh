// Moments of one source point in the expansion over wavenumbers (expand64.cu, near.cu).
#pragma once

#include <math.h>

namespace bem {

// acc[f][m] += base_f T_m(x), x = two_over_R r - 1, at y - x = (dx, dy, dz) with weight w
// (1 / 4 pi included): base = w e^{i c r} / r for the single layer's family and, for the double
// layer's, that times s = (y - x).n / r^2.
template <int MT, bool kG, bool kH>
__device__ __forceinline__ void expand_point(double (&ar)[(kG ? 1 : 0) + (kH ? 1 : 0)][MT],
                                             double (&ai)[(kG ? 1 : 0) + (kH ? 1 : 0)][MT],
                                             double w, double dx, double dy, double dz,
                                             const double* nrm, double2 c, double two_over_R) {
  constexpr int F = (kG ? 1 : 0) + (kH ? 1 : 0);
  const double r2 = dx * dx + dy * dy + dz * dz;
  const double ri = rsqrt(r2);
  double r = r2 * ri;
  r = fma(0.5 * ri, fma(-r, r, r2), r);   // sqrt(r2) to its last bit or so
  double s, co;
  sincos(c.x * r, &s, &co);
  w *= ri;
  if (c.y != 0.0) w *= exp(-c.y * r);
  const double x = fma(r, two_over_R, -1.0), x2 = 2.0 * x;
  double br[F], bi[F];
  if (kG) {
    br[0] = w * co;
    bi[0] = w * s;
  }
  if (kH) {
    const double h = w * ri * ri * (dx * nrm[0] + dy * nrm[1] + dz * nrm[2]);
    br[F - 1] = h * co;
    bi[F - 1] = h * s;
  }
  double t0 = 1.0, t1 = x;
#pragma unroll
  for (int m = 0; m < MT; ++m) {
#pragma unroll
    for (int f = 0; f < F; ++f) {
      ar[f][m] = fma(br[f], t0, ar[f][m]);
      ai[f][m] = fma(bi[f], t0, ai[f][m]);
    }
    const double t2 = fma(x2, t1, -t0);
    t0 = t1;
    t1 = t2;
  }
}

}  // namespace bem
