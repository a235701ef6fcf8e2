// FP64 device helpers shared by the kernels that evaluate the singular self term
// A_ll(k) = integral over triangle l of exp(i k r) / (4 pi r) about its centroid.
//
// Polar coordinates about the centroid x in the plane of the triangle: the radial
// integral is R h(i k R) with h(w) = (e^w - 1) / w; along each edge (d the distance from
// x to the edge's line, s the position along the edge from the foot of the perpendicular)
// the angle is traded for u = asinh(s / d), so R = d cosh(u), d(phi) = du / cosh(u) and
// the integrand d h(i k d cosh u) is entire in u; 16-point Gauss-Legendre on each side of
// u = 0.
#pragma once

#include <math.h>

namespace bem {

constexpr double kPiD = 3.141592653589793238462643383279502884;

struct GL16 {
  double x[16];
  double w[16];
};

// Gauss-Legendre nodes as the roots of P_16 by Newton's method (three-term recurrence).
inline GL16 make_gl16() {
  GL16 g;
  const int n = 16;
  for (int i = 0; i < n; ++i) {
    double x = cos(kPiD * (4.0 * i + 3.0) / (4.0 * n + 2.0));
    double dp = 1.0;
    for (int it = 0; it < 60; ++it) {
      double pm = 1.0, p = x;
      for (int k = 1; k < n; ++k) {
        const double pn = ((2 * k + 1) * x * p - k * pm) / (k + 1);
        pm = p;
        p = pn;
      }
      dp = n * (pm - x * p) / (1.0 - x * x);
      const double step = p / dp;
      x -= step;
      if (fabs(step) <= 4e-17) break;
    }
    double pm = 1.0, p = x;
    for (int k = 1; k < n; ++k) {
      const double pn = ((2 * k + 1) * x * p - k * pm) / (k + 1);
      pm = p;
      p = pn;
    }
    dp = n * (pm - x * p) / (1.0 - x * x);
    g.x[i] = x;
    g.w[i] = 2.0 / ((1.0 - x * x) * dp * dp);
  }
  return g;
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// h(w) = (e^w - 1) / w; Taylor series sum_m w^m / (m + 1)! for |w| < 1/2.
__device__ inline double2 h_fun(double2 w) {
  if (w.x * w.x + w.y * w.y < 0.25) {
    double2 s = make_double2(0.0, 0.0), t = make_double2(1.0, 0.0);
    for (int m = 0; m < 24; ++m) {
      s.x += t.x;
      s.y += t.y;
      t = zmul(t, w);
      t.x /= (m + 2.0);
      t.y /= (m + 2.0);
    }
    return s;
  }
  double sn, cs;
  sincos(w.y, &sn, &cs);
  const double e = exp(w.x);
  const double2 num = make_double2(e * cs - 1.0, e * sn);
  const double d = w.x * w.x + w.y * w.y;
  return make_double2((num.x * w.x + num.y * w.y) / d, (num.y * w.x - num.x * w.y) / d);
}

// h'(w) = (w e^w - e^w + 1) / w^2; Taylor series sum_{m>=1} m w^{m-1} / (m + 1)! near 0.
__device__ inline double2 hprime_fun(double2 w) {
  if (w.x * w.x + w.y * w.y < 0.25) {
    double2 s = make_double2(0.0, 0.0), p = make_double2(1.0, 0.0);   // p = w^{m-1}
    double fact = 2.0;                                                // (m + 1)!
    for (int m = 1; m < 26; ++m) {
      s.x += m * p.x / fact;
      s.y += m * p.y / fact;
      p = zmul(p, w);
      fact *= (m + 2.0);
    }
    return s;
  }
  double sn, cs;
  sincos(w.y, &sn, &cs);
  const double e = exp(w.x);
  const double2 ew = make_double2(e * cs, e * sn);
  const double2 num = make_double2(zmul(w, ew).x - ew.x + 1.0, zmul(w, ew).y - ew.y);
  const double2 w2 = zmul(w, w);
  const double d = w2.x * w2.x + w2.y * w2.y;
  return make_double2((num.x * w2.x + num.y * w2.y) / d, (num.y * w2.x - num.x * w2.y) / d);
}

// Edge data of the self term, FP64: for edge e = (v[e], v[e+1]) about the point x, the
// distance d from x to the edge's line and the u = asinh(s / d) range of the edge.
__device__ inline void self_edge(const double v[3][3], const double x[3], int e, double& d,
                                 double& up, double& uq) {
  const double* p = v[e];
  const double* q = v[(e + 1) % 3];
  double tx = q[0] - p[0], ty = q[1] - p[1], tz = q[2] - p[2];
  const double len = sqrt(tx * tx + ty * ty + tz * tz);
  tx /= len;
  ty /= len;
  tz /= len;
  const double px = p[0] - x[0], py = p[1] - x[1], pz = p[2] - x[2];
  const double qx = q[0] - x[0], qy = q[1] - x[1], qz = q[2] - x[2];
  const double sp = px * tx + py * ty + pz * tz;
  const double sq = qx * tx + qy * ty + qz * tz;
  const double ox = px - sp * tx, oy = py - sp * ty, oz = pz - sp * tz;
  d = sqrt(ox * ox + oy * oy + oz * oz);
  up = asinh(sp / d);
  uq = asinh(sq / d);
}

// Self entries c_G A_ll(k) + c_H / 2 of panel l at nk wavenumbers (deriv: c_G A'_ll(k)), by one
// warp: out[j n + l].
// A_ll(k) = (1 / 4 pi) sum_g f_g h(i k R_g) over the 96 angular nodes, f_g their weights, R_g <= rho
// their radii; three nodes a lane. With h(w) = sum_p w^p / (p + 1)! it is sum_p (i k rho)^p c_p,
// c_p = (1 / 4 pi) sum_g f_g (R_g / rho)^p / (p + 1)!, and the moments c_p serve every wavenumber: 24
// terms are exact to 1e-18 for |k| rho <= 2, and a wavenumber costs 24 complex multiply-adds where
// the sum over the angular nodes costs 96 sines, exponentials and complex divisions. Larger |k| rho (a
// panel of a third of a wavelength) take that sum, the warp's lanes together for a wavenumber at a
// time (by the one lane of a wavenumber, and after the moments, 96 nodes took 400 us where one thread
// a panel had taken 200: residuals of one vector on 12 panels at k = 5). FP64-bound; 768 panels, 32
// wavenumbers: 2.94 -> 0.055 ms.
constexpr int kSelfTerms64 = 24;

__device__ inline void self_entries_warp(const double v[3][3], const double x[3], int64_t l,
                                         int64_t n, int nk, const double2* __restrict__ k,
                                         const GL16& gl, bool deriv, double cgr, double cgi,
                                         double chr, double chi, int lane,
                                         double2* __restrict__ out) {
  // edge data by lanes 0..2, then to all
  double d_, up_, uq_;
  self_edge(v, x, lane % 3, d_, up_, uq_);
  double rho2 = 0.0;
  for (int e = 0; e < 3; ++e) {
    double r2 = 0.0;
    for (int c = 0; c < 3; ++c) r2 += (v[e][c] - x[c]) * (v[e][c] - x[c]);
    rho2 = fmax(rho2, r2);
  }
  const double rho = sqrt(rho2), inv = 1.0 / rho;
  double f[3], R[3];   // weights and radii of this lane's nodes, one of every edge
#pragma unroll
  for (int e = 0; e < 3; ++e) {   // side lane / 16, node lane % 16
    const double d = __shfl_sync(0xffffffffu, d_, e), up = __shfl_sync(0xffffffffu, up_, e),
                 uq = __shfl_sync(0xffffffffu, uq_, e);
    const bool split = up < 0.0 && uq > 0.0;
    const int side = lane / 16, gi = lane % 16;
    const double lo = split && side ? 0.0 : up, hi = split && !side ? 0.0 : uq;
    const double half = 0.5 * (hi - lo), mid = 0.5 * (hi + lo);
    f[e] = (split || side == 0) ? half * gl.w[gi] * d : 0.0;
    R[e] = d * cosh(mid + half * gl.x[gi]);
  }
  auto series = [&](double2 kj) { return (kj.x * kj.x + kj.y * kj.y) * rho2 <= 4.0; };
  auto put = [&](int j, double2 a) {
    out[(int64_t)j * n + l] = make_double2(cgr * a.x - cgi * a.y + (deriv ? 0.0 : 0.5 * chr),
                                           cgr * a.y + cgi * a.x + (deriv ? 0.0 : 0.5 * chi));
  };
  bool near = false, far = false;
  for (int j = lane; j < nk; j += 32) (series(k[j]) ? near : far) = true;
  near = __any_sync(0xffffffffu, near);
  far = __any_sync(0xffffffffu, far);
  if (near) {
    double mom[kSelfTerms64];
#pragma unroll
    for (int p = 0; p < kSelfTerms64; ++p) mom[p] = 0.0;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      const double t = R[e] * inv;
      double g = f[e];
#pragma unroll
      for (int p = 0; p < kSelfTerms64; ++p) {
        mom[p] += g;
        g *= t;
      }
    }
    double fact = 1.0;
#pragma unroll
    for (int p = 0; p < kSelfTerms64; ++p) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) mom[p] += __shfl_xor_sync(0xffffffffu, mom[p], off);
      fact *= 1.0 / (p + 1);
      mom[p] *= fact * (1.0 / (4.0 * kPiD));
    }
    for (int j = lane; j < nk; j += 32) {
      const double2 kj = k[j];
      if (!series(kj)) continue;
      const double2 w = make_double2(-kj.y * rho, kj.x * rho);   // i k rho
      double2 a = make_double2(0.0, 0.0);
      if (deriv) {   // i rho sum_p p c_p w^{p-1}
#pragma unroll
        for (int p = kSelfTerms64 - 1; p >= 1; --p)
          a = make_double2(fma(a.x, w.x, fma(-a.y, w.y, p * mom[p])), fma(a.x, w.y, a.y * w.x));
        a = make_double2(-rho * a.y, rho * a.x);
      } else {
#pragma unroll
        for (int p = kSelfTerms64 - 1; p >= 0; --p)
          a = make_double2(fma(a.x, w.x, fma(-a.y, w.y, mom[p])), fma(a.x, w.y, a.y * w.x));
      }
      put(j, a);
    }
  }
  if (!far) return;
  for (int j = 0; j < nk; ++j) {
    const double2 kj = k[j];
    if (series(kj)) continue;
    double2 a = make_double2(0.0, 0.0);
#pragma unroll 1
    for (int e = 0; e < 3; ++e) {
      const double fe = e == 0 ? f[0] : e == 1 ? f[1] : f[2];
      const double Re = e == 0 ? R[0] : e == 1 ? R[1] : R[2];
      const double2 w = make_double2(-kj.y * Re, kj.x * Re);   // i k R
      if (deriv) {   // the integral of i R^2 h'(i k R): f_g holds one R
        const double2 hp = hprime_fun(w);
        a.x -= fe * Re * hp.y;
        a.y += fe * Re * hp.x;
      } else {
        const double2 h = h_fun(w);
        a.x += fe * h.x;
        a.y += fe * h.y;
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      a.x += __shfl_xor_sync(0xffffffffu, a.x, off);
      a.y += __shfl_xor_sync(0xffffffffu, a.y, off);
    }
    if (lane == 0) put(j, make_double2(a.x / (4.0 * kPiD), a.y / (4.0 * kPiD)));
  }
}

// FP32 version for the mixed path: given the edge data (d, u range per edge, computed in
// FP64), the angular quadrature and h(i k R) in FP32 (relative accuracy ~1e-6, the level
// of the mixed path). Returns the part of the sum over the angular nodes t = part,
// part + nparts, ... of the 96 = 3 edges x 2 sides x 16 nodes.
__device__ inline float2 self_term32_part(const float d3[3], const float up3[3],
                                          const float uq3[3], float kr, float ki,
                                          const GL16& gl, int part, int nparts) {
  float tr = 0.f, ti = 0.f;
  for (int t = part; t < 96; t += nparts) {
    const int e = t / 32, side = (t / 16) % 2, gi = t % 16;
    const float d = d3[e], up = up3[e], uq = uq3[e];
    // the two sides of u = 0 when the foot lies inside the edge, else the whole range once
    const bool split = up < 0.f && uq > 0.f;
    float lo, hi;
    if (split) {
      lo = side == 0 ? up : 0.f;
      hi = side == 0 ? 0.f : uq;
    } else {
      if (side == 1) continue;
      lo = up;
      hi = uq;
    }
    const float half = 0.5f * (hi - lo), mid = 0.5f * (hi + lo);
    const float R = d * coshf(mid + half * (float)gl.x[gi]);
    const float wr = -ki * R, wi = kr * R;   // w = i k R
    float hr, hi2;
    if (wr * wr + wi * wi < 0.25f) {
      // sum_m w^m / (m + 1)!, 10 terms
      float sr = 0.f, si = 0.f, cr = 1.f, ci = 0.f;
      for (int m = 0; m < 10; ++m) {
        sr += cr;
        si += ci;
        const float nr = (cr * wr - ci * wi) / (m + 2.0f);
        const float ni = (cr * wi + ci * wr) / (m + 2.0f);
        cr = nr;
        ci = ni;
      }
      hr = sr;
      hi2 = si;
    } else {
      float sn, cs;
      sincosf(wi, &sn, &cs);
      const float ex = expf(wr);
      const float nr = ex * cs - 1.f, ni = ex * sn;
      const float dd = wr * wr + wi * wi;
      hr = (nr * wr + ni * wi) / dd;
      hi2 = (ni * wr - nr * wi) / dd;
    }
    const float f = half * (float)gl.w[gi] * d;
    tr += f * hr;
    ti += f * hi2;
  }
  const float inv4pi = (float)(1.0 / (4.0 * kPiD));
  return make_float2(tr * inv4pi, ti * inv4pi);
}

}  // namespace bem
