// FP64 products with A(k) at many wavenumbers from one evaluation of the operator.
//
// Every entry is A_il(k) = sum_q w_q e^{i k r_q} / r_q with r in [0, R]. About a centre c,
// e^{i k r} = e^{i c r} e^{i (k - c) r}, and on [0, R] the second factor is a Chebyshev series
// in x = 2 r / R - 1 whose terms fall like (|k - c| R / 4)^m / m!: M = 12 .. 20 terms give
// FP64 rounding for a contour of radius ~1 about a body of diameter ~2, whatever the number
// of wavenumbers. So
//     A(k_j) = sum_m a_m(k_j) G_m,   G_m,il = sum_q w_q e^{i c r_q} / r_q T_m(x_q),
// and A(k_j) X = sum_m a_m(k_j) (G_m X): one evaluation (a sine, cosine and root per point)
// and M matrix products in the place of N of each. All families of moments take this one series;
// powers of r go into their weights. The general operator c_G G + c_H (1/2 I + K), whose second kernel
// is (i k r - 1) e^{ikr} s / r, s = (y - x).n / r^2, adds H_m of weight w s / r with the factor -c_H and
// J_m of weight w s with i k c_H; the k-derivative has G_m of weight w with i c_G and J_m of weight
// w s r with -k c_H. (A series of (i k r - 1) e^{i (k - c) r} has coefficients of ~k R / 2 beside a
// value of 1 at r = 0, and with them the rounding of near entries: residuals of the Robin operator at
// k R = 14 were off by 7.3e-16 against 128-bit sums, the direct form by 3.0e-16, now by 2.6e-16.)
//
// Bound by arithmetic: 7 points of 15 FP64 operations and ~(110 + 26 M) integer ones per entry
// (below), and M nu products, in FP64 (1/64 of the FP32 rate on this part) or, the larger ones,
// on the tensor core (split64.cu), against N (7 x 77 + 4 nu) FP64 operations of the direct form;
// the moments' round trip through memory (32 bytes a moment, three times that with the digits) is
// ~20 %. Measured: the products of the 768-panel cube (N = 32, nu = 64) 28.1 -> 0.95 ms, of the
// residuals of 8 vectors on 5120 panels 258 -> 19 ms, with the same or a smaller error against
// 64-bit references.
#include <math.h>

#include <algorithm>

#include "expand64.cuh"
#include "expand64.h"

namespace bem {
namespace {

constexpr int kCoefPoints = 64;    // Chebyshev points of the coefficients' quadrature (> kMaxTerms)
constexpr int kRowsE = 128;        // rows per block of the evaluation (a thread each)
constexpr int kColsE = 8;          // columns per block of the evaluation
constexpr size_t kMomentBytes = (size_t)1 << 30;   // moments held at a time
// n^2 S (padded columns - 4) from which the split products pay (split64.cu; conversions of 20 ps a
// moment and three more launches against 5.6 ps a moment and column). Split against FP64, in us:
// 192 panels, 4 columns 354 / 335, 300 panels, 8 residuals 380 / 350 below it; projections of 192
// panels, 16 columns 362 / 450 (2^23.9), 300 x 10 401 / 615, 588 x 60 765 / 2785, residuals of 588
// panels, 8 vectors 580 / 601, 3072 panels, 2 vectors 5853 / 8346 above.
constexpr double kSplitWork = 0x1.cp23;
constexpr size_t kMaxWork = (size_t)24 << 30;      // workspace beyond which the direct form runs
// Panels below which the direct form runs: its threads pass over the columns one after the other (7 us
// a column in a projection, 16 in a residual), the expansion's launches take the same time for any few
// panels. Expanded against direct, in us: projections at 16 nodes 250 / 125 (12 panels), 282 / 233 (24),
// 280 / 266 (32), 288 / 355 (48), with both operators 372 / 140, 425 / 283, 420 / 334, 424 / 456;
// residuals 170 / 158 (2), 183 / 195 (4), 217 / 321 (12).
constexpr int64_t kMinNodes = 40, kMinColumns = 4;
// |Re c| R beyond which the direct form runs. The fixed-point phase of every pair is off by up to
// 2^-59 |Re c| R radians, whatever their distance, the direct form's by 2^-53 k r: for bodies far
// apart (R of 1e4, 1e6 bodies' sizes at k = 10: 5e-14, 8e-12 in their own entries) that is the
// larger error. Up to here it is at most 2^-52, an ulp.
constexpr double kMaxPhase = 128.0;
// max |Im (k - c)| R beyond which the direct form runs. The series of e^{i (k - c) r} has coefficients
// of up to e^{|Im (k - c)| R} whatever r, so the rounding of moments and slot products enters near
// entries that much larger. Against 128-bit products, expanded / direct, error of ||A X|| (300 panels,
// single layer, Neumann, Robin):
//   projections at the lowest nodes: 4.6e-16 / 8.3e-16, 2.6e-16 / 6.1e-16, 2.8e-16 / 8.8e-16 at 1.2,
//     1.3e-15 / 1.4e-15, 6.6e-16 / 8.8e-16, 1.2e-15 / 1.4e-15 at 3.2 (a contour of radius 1.6); the
//     other nodes and V^H A V a third of the direct form's. Vectors of four panels lose more, by
//     component of (|A| |x|)_i 4.0e-15 / 8e-16 at 4.0 (80 panels) and 1.7e-14 at 5.6.
//   residuals, whose direct form sums more exactly: 4.7e-16 / 5.5e-16, 2.9e-16 / 3.0e-16,
//     2.9e-16 / 3.1e-16 near the axis, 5.4e-16 / 5.5e-16, 3.1e-16 / 3.2e-16, 3.1e-16 / 3.2e-16 at 0.6,
//     but 7.3e-16 / 5.7e-16, 3.7e-16 / 3.5e-16 at 1.4.
constexpr double kMaxGrowthNodes = 4.0, kMaxGrowthColumns = 0.6;

// a[f][j][m], f the family: Chebyshev coefficients on [0, R] of e^{i (k_j - c) r}, times the family's
// factor. One block per (j, f): a thread
// per Chebyshev point for the function, a thread per angle for the cosines cos(pi t / 128) that
// the sums take, then a warp per coefficient. (A thread per coefficient with the cosines of all
// its points took 196 us, the points shared 56 us at 32 wavenumbers; now 8 us.)
constexpr int kCoefThreads = 256;

__global__ void __launch_bounds__(kCoefThreads)
expand_coef_kernel(const double2* __restrict__ k, int nk, double2 c, double R, int M, bool hasG,
                   bool deriv, OpCoef op, double2* __restrict__ a) {
  static_assert(kCoefThreads == 4 * kCoefPoints, "an angle a thread");
  __shared__ double2 fv[kCoefPoints];
  __shared__ double cosine[kCoefThreads];
  const int j = blockIdx.x, q = threadIdx.x;
  const double2 kj = k[j];
  cosine[q] = cospi(q / (2.0 * kCoefPoints));
  __syncthreads();
  if (q < kCoefPoints) {
    const double r = 0.5 * R * (cosine[2 * q + 1] + 1.0);
    const double dr = kj.x - c.x, di = kj.y - c.y;
    double sn, cs;
    sincos(dr * r, &sn, &cs);
    const double e = exp(-di * r);
    fv[q] = make_double2(e * cs, e * sn);
  }
  __syncthreads();
  // the family's factor
  double2 fac;
  if (hasG && blockIdx.y == 0) {
    fac = deriv ? make_double2(-op.cgi, op.cgr) : make_double2(op.cgr, op.cgi);
  } else {
    const double2 kc = make_double2(kj.x * op.chr - kj.y * op.chi, kj.x * op.chi + kj.y * op.chr);   // k c_H
    if (deriv) fac = make_double2(-kc.x, -kc.y);
    else if (blockIdx.y == (hasG ? 1 : 0)) fac = make_double2(-op.chr, -op.chi);
    else fac = make_double2(-kc.y, kc.x);
  }
  const int lane = q % 32;
  for (int m = q / 32; m < M; m += kCoefThreads / 32) {
    double2 s = make_double2(0.0, 0.0);
#pragma unroll
    for (int p = lane; p < kCoefPoints; p += 32) {
      const double w = cosine[m * (2 * p + 1) % kCoefThreads];   // period 2 pi: kCoefThreads angles
      s.x = fma(w, fv[p].x, s.x);
      s.y = fma(w, fv[p].y, s.y);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
    }
    const double sc = (m == 0 ? 1.0 : 2.0) / kCoefPoints;
    if (lane == 0)
      a[((int64_t)blockIdx.y * nk + j) * M + m] =
          make_double2(sc * (s.x * fac.x - s.y * fac.y), sc * (s.x * fac.y + s.y * fac.x));
  }
}

// ---- the moments ----
//
// In FP64 a point took ~98 operations on a pipe of 2 a clock and SM: distance, root, sine and
// cosine, and 3 a term for the Chebyshev polynomials and the sums; 34 ms for 5120 panels and 14
// terms. Only the distance and its root need a floating exponent. With r <= R and |T_m| <= 1
// the rest is fixed-point arithmetic of 62 fractional bits, on the integer pipe: a product is
// three 32 x 32 -> 64 multiply-adds, rounded to 2^-60 of its operands' bounds, finer than FP64's
// 2^-53. So a point takes 15 FP64 operations and ~(110 + 26 M) integer instructions beside them.
//   rho = r / R -> x = 2 rho - 1; the phase c r in turns, K rho mod 1, exact to 2^-60 max(1, K);
//   its sine and cosine from a table of 1024 angles and a Taylor series of the rest (|t| <=
//   pi / 1024: t - t^3 / 6 + t^5 / 120 and 1 - t^2 / 2 + t^4 / 24, the next terms below 2^-59);
//   the seven weights w / r scaled together so that their sum fills 62 bits.
// Measured: 5120 panels, 14 terms 34.3 -> 11.0 ms; 768 panels, 17 terms 730 -> 319 us; the residuals
// and products keep their error against 64-bit references (7.6e-16, 9.5e-16).
// cos and sin of 2 pi q / kAngles as 62-bit fractions, split: (cos h, cos l, sin h, sin l).
__global__ void expand_angles_kernel(int4* __restrict__ table) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= kAngles) return;
  double sn, cs;
  sincospi(2.0 * q / kAngles, &sn, &cs);
  const Split c = split(llrint(ldexp(cs, 62))), s = split(llrint(ldexp(sn, 62)));
  table[q] = make_int4(c.h, c.l, s.h, s.l);
}

// Moments of the columns [l0, l0 + kc): G[f M + m][l - l0][i] (i fastest). One thread per row;
// the block's columns' geometry is staged in shared memory and read by broadcast. The
// diagonal is zero (the self terms are added in closed form).
template <int MT, int kKind>
__global__ void __launch_bounds__(kRowsE)
expand_moments_kernel(Geometry g, double2 c, FixedPhase fp, int M, int64_t l0, int kc,
                      const int4* __restrict__ angles, double2* __restrict__ G) {
  constexpr int F = kFamilies<kKind>;
  __shared__ int4 table[kAngles];
  __shared__ double sq[kColsE][7][4];
  __shared__ double sn3[kColsE][3];
  __shared__ long long srho[7][kRowsE];
  __shared__ double sbase[7][F][kRowsE];   // the weights, then the same as fixed-point numbers
  const int64_t n = g.n;
  const int tid = threadIdx.x;
  const int64_t i = (int64_t)blockIdx.x * kRowsE + tid;
  const int c0 = blockIdx.y * kColsE;
  const int nc = min(kColsE, kc - c0);
  for (int t = tid; t < kAngles; t += kRowsE) table[t] = angles[t];
  for (int t = tid; t < nc * 7; t += kRowsE) {
    const int cc = t / 7, q = t % 7;
    const int64_t l = l0 + c0 + cc;
    sq[cc][q][0] = g.qp[q * n + l];
    sq[cc][q][1] = g.qp[(7 + q) * n + l];
    sq[cc][q][2] = g.qp[(14 + q) * n + l];
    sq[cc][q][3] = g.qw[q * n + l];
  }
  if (kKind >= kDouble)
    for (int t = tid; t < nc * 3; t += kRowsE) sn3[t / 3][t % 3] = g.nrm[(t % 3) * n + l0 + c0 + t / 3];
  __syncthreads();
  if (i >= n) return;
  const double xi = g.cx[i], yi = g.cx[n + i], zi = g.cx[2 * n + i];
  const Split K = split(fp.K);
  for (int cc = 0; cc < nc; ++cc) {
    long long ar[F][MT], ai[F][MT];
#pragma unroll
    for (int f = 0; f < F; ++f)
#pragma unroll
      for (int m = 0; m < MT; ++m) ar[f][m] = ai[f][m] = 0;
    int e[F];                    // exponents of the families' scales
    bool finite = true;
#pragma unroll
    for (int f = 0; f < F; ++f) e[f] = 0;
    if (l0 + c0 + cc != i) {
      // distances and weights
      int top[F];
#pragma unroll
      for (int f = 0; f < F; ++f) top[f] = 0;
#pragma unroll 1
      for (int q = 0; q < 7; ++q) {
        const double dx = sq[cc][q][0] - xi, dy = sq[cc][q][1] - yi, dz = sq[cc][q][2] - zi;
        const double r2 = dx * dx + dy * dy + dz * dz;
        double r, ri;
        root_and_inverse(r2, r, ri);
        srho[q][tid] = fixed62(r * fp.inv_R, 0);
        const double dn = kKind >= kDouble ? dx * sn3[cc][0] + dy * sn3[cc][1] + dz * sn3[cc][2] : 0.0;
        double w[F];
        moment_weights<kKind>(w, sq[cc][q][3], r, ri, dn, c.y);
#pragma unroll
        for (int f = 0; f < F; ++f) sbase[q][f][tid] = w[f];
#pragma unroll
        for (int f = 0; f < F; ++f)
          top[f] = max(top[f], __double2hiint(sbase[q][f][tid]) & 0x7FFFFFFF);
      }
      // the weights as 62-bit fractions of a scale just above the sum of their magnitudes
#pragma unroll
      for (int f = 0; f < F; ++f) {
        finite = finite && top[f] < 0x7FF00000;
        e[f] = (top[f] >> 20) - 1022 + 3;
        long long sum = 0;
#pragma unroll 1
        for (int q = 0; q < 7; ++q) {
          const double v = sbase[q][f][tid];
          const long long b = fixed62(v, e[f]);
          sum += b;
          sbase[q][f][tid] = __longlong_as_double(__double2hiint(v) < 0 ? -b : b);
        }
        const int sh = sum ? __clzll(sum) - 2 : 0;
        e[f] -= sh;
#pragma unroll 1
        for (int q = 0; q < 7; ++q)
          sbase[q][f][tid] = __longlong_as_double(__double_as_longlong(sbase[q][f][tid]) << sh);
      }
#pragma unroll 1
      for (int q = 0; q < 7; ++q) {
        long long b[F];
#pragma unroll
        for (int f = 0; f < F; ++f) b[f] = __double_as_longlong(sbase[q][f][tid]);
        add_moments<MT, F>(ar, ai, b, srho[q][tid], K, fp.kb, table);
      }
    }
#pragma unroll
    for (int f = 0; f < F; ++f)
#pragma unroll
      for (int m = 0; m < MT; ++m)
        if (m < M)
          G[((int64_t)(f * M + m) * kc + c0 + cc) * n + i] =
              finite ? make_double2(from_fixed60(ar[f][m], e[f]), from_fixed60(ai[f][m], e[f]))
                     : make_double2(NAN, NAN);
  }
}

constexpr int kTM = 32;    // rows of a product tile
constexpr int kTK = 16;    // columns of the moments staged at a time
constexpr int kThreadsM = 128;

// Yp[split][s] (+)= G_s[:, ks] X[l0 + ks, :] for slot s = blockIdx.z % S and its share ks of
// the kc columns. Three real products per complex term, as the Gram kernel's. FP64-bound: a
// thread's 2 x (TN / 8) outputs take 6 .. 24 FP64 operations per k against 9 .. 18 8-byte
// shared-memory reads at 1/16 of their cost.
template <int TN>
__global__ void __launch_bounds__(kThreadsM)
expand_product_kernel(const double2* __restrict__ G, int64_t n, int kc, int S, int splits,
                      const double2* __restrict__ X, int64_t ldx, int nu, int64_t l0, bool add,
                      double2* __restrict__ Yp) {
  __shared__ double ar[kTK][kTM], ai[kTK][kTM], as[kTK][kTM];
  __shared__ double br[kTK][TN + 1], bi[kTK][TN + 1], bs[kTK][TN + 1];
  constexpr int kCT = TN / 8;   // columns per thread (16 row pairs x 8 column groups)
  const int s = blockIdx.z % S, split = blockIdx.z / S;
  const int64_t i0 = (int64_t)blockIdx.x * kTM;
  const int j0 = blockIdx.y * TN;
  const int kb = (int)((int64_t)kc * split / splits), ke = (int)((int64_t)kc * (split + 1) / splits);
  const int tid = threadIdx.x, tr = tid % 16, tc = tid / 16;
  const double2* Gs = G + (int64_t)s * kc * n;
  double s1[2][kCT], s2[2][kCT], s3[2][kCT];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < kCT; ++b) s1[a][b] = s2[a][b] = s3[a][b] = 0.0;
  for (int k0 = kb; k0 < ke; k0 += kTK) {
    __syncthreads();
    for (int t = tid; t < kTK * kTM; t += kThreadsM) {
      const int r = t % kTM, k = t / kTM;
      const double2 v = (k0 + k < ke && i0 + r < n) ? Gs[(int64_t)(k0 + k) * n + i0 + r]
                                                    : make_double2(0.0, 0.0);
      ar[k][r] = v.x;
      ai[k][r] = v.y;
      as[k][r] = v.x + v.y;
    }
    for (int t = tid; t < kTK * TN; t += kThreadsM) {
      const int k = t % kTK, cl = t / kTK;
      const double2 v = (k0 + k < ke && j0 + cl < nu) ? X[(int64_t)(j0 + cl) * ldx + l0 + k0 + k]
                                                      : make_double2(0.0, 0.0);
      br[k][cl] = v.x;
      bi[k][cl] = v.y;
      bs[k][cl] = v.x + v.y;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTK; ++k) {
      double a1[2], a2[2], a3[2];
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        a1[a] = ar[k][tr + 16 * a];
        a2[a] = ai[k][tr + 16 * a];
        a3[a] = as[k][tr + 16 * a];
      }
#pragma unroll
      for (int b = 0; b < kCT; ++b) {
        const int cl = tc + 8 * b;
        const double b1 = br[k][cl], b2 = bi[k][cl], b3 = bs[k][cl];
#pragma unroll
        for (int a = 0; a < 2; ++a) {
          s1[a][b] = fma(a1[a], b1, s1[a][b]);
          s2[a][b] = fma(a2[a], b2, s2[a][b]);
          s3[a][b] = fma(a3[a], b3, s3[a][b]);
        }
      }
    }
  }
  double2* Ys = Yp + ((int64_t)split * S + s) * n * nu;
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int64_t i = i0 + tr + 16 * a;
    if (i >= n) continue;
#pragma unroll
    for (int b = 0; b < kCT; ++b) {
      const int cl = j0 + tc + 8 * b;
      if (cl >= nu) continue;
      double2 y = make_double2(s1[a][b] - s2[a][b], s3[a][b] - s1[a][b] - s2[a][b]);
      if (add) {
        const double2 o = Ys[(int64_t)cl * n + i];
        y.x += o.x;
        y.y += o.y;
      }
      Ys[(int64_t)cl * n + i] = y;
    }
  }
}

// Yp[0][s] = sum over the splits, in order.
__global__ void expand_sum_kernel(int64_t count, int splits, double2* __restrict__ Yp) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= count) return;
  double2 s = Yp[t];
  for (int q = 1; q < splits; ++q) {
    const double2 v = Yp[(int64_t)q * count + t];
    s.x += v.x;
    s.y += v.y;
  }
  Yp[t] = s;
}

constexpr int kNodesC = 8;   // wavenumbers per thread of the combination

// Y_j = sum_s a_s(k_j) Y_s + self_j V (the self terms of the table, node-major), 8 nodes a thread.
__global__ void __launch_bounds__(128)
expand_nodes_kernel(const double2* __restrict__ Ys, int64_t n, int nu, int M, int fams, int N,
                    const double2* __restrict__ a, const double2* __restrict__ self,
                    const double2* __restrict__ V, int64_t ldv, double2* __restrict__ Y) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n * nu) return;
  const int64_t i = t % n;
  const int cl = (int)(t / n);
  const int j0 = blockIdx.y * kNodesC;
  const double2 v = V[(int64_t)cl * ldv + i];
  double2 acc[kNodesC];   // the slots' sum; the self term, half of the vector for K, last
#pragma unroll
  for (int u = 0; u < kNodesC; ++u) acc[u] = make_double2(0.0, 0.0);
  for (int f = 0; f < fams; ++f)
    for (int m = 0; m < M; ++m) {
      const double2 y = Ys[(int64_t)(f * M + m) * n * nu + t];
#pragma unroll
      for (int u = 0; u < kNodesC; ++u) {
        const double2 w = a[((int64_t)f * N + min(j0 + u, N - 1)) * M + m];
        acc[u].x = fma(w.x, y.x, fma(-w.y, y.y, acc[u].x));
        acc[u].y = fma(w.x, y.y, fma(w.y, y.x, acc[u].y));
      }
    }
#pragma unroll
  for (int u = 0; u < kNodesC; ++u)
    if (j0 + u < N) {
      const double2 d = self[(int64_t)(j0 + u) * n + i];
      Y[(int64_t)(j0 + u) * n * nu + t] = make_double2(acc[u].x + (d.x * v.x - d.y * v.y),
                                                       acc[u].y + (d.x * v.y + d.y * v.x));
    }
}

// R_c = sum_s a_s(k_c) Y_s,c + R_c x_c (R holds the self terms at k_c).
__global__ void expand_columns_kernel(const double2* __restrict__ Ys, int64_t n, int m, int M,
                                      int fams, const double2* __restrict__ a,
                                      const double2* __restrict__ X, int64_t ldx,
                                      double2* __restrict__ R) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n * m) return;
  const int64_t i = t % n;
  const int c = (int)(t / n);
  double2 acc = make_double2(0.0, 0.0);   // the slots' sum; the self term last (expand_nodes_kernel)
  for (int f = 0; f < fams; ++f)
    for (int q = 0; q < M; ++q) {
      const double2 y = Ys[(int64_t)(f * M + q) * n * m + t];
      const double2 w = a[((int64_t)f * m + c) * M + q];
      acc.x = fma(w.x, y.x, fma(-w.y, y.y, acc.x));
      acc.y = fma(w.x, y.y, fma(w.y, y.x, acc.y));
    }
  const double2 x = X[(int64_t)c * ldx + i], d = R[t];
  R[t] = make_double2(acc.x + (d.x * x.x - d.y * x.y), acc.y + (d.x * x.y + d.y * x.x));
}

using MomentKernel = void (*)(Geometry, double2, FixedPhase, int, int64_t, int, const int4*, double2*);

template <int kKind>
MomentKernel moment_kernel(int M) {
  if (M <= 1) return expand_moments_kernel<1, kKind>;
  if (M <= 8) return expand_moments_kernel<8, kKind>;
  if (M <= 10) return expand_moments_kernel<10, kKind>;
  if (M <= 12) return expand_moments_kernel<12, kKind>;
  if (M <= 13) return expand_moments_kernel<13, kKind>;
  if (M <= 14) return expand_moments_kernel<14, kKind>;
  if (M <= 15) return expand_moments_kernel<15, kKind>;
  if (M <= 16) return expand_moments_kernel<16, kKind>;
  if (M <= 17) return expand_moments_kernel<17, kKind>;
  if (M <= 18) return expand_moments_kernel<18, kKind>;
  if (M <= 20) return expand_moments_kernel<20, kKind>;
  if (M <= 24) return expand_moments_kernel<24, kKind>;
  return expand_moments_kernel<kMaxTerms, kKind>;
}

// K = c / (2 pi inv_R) in turns, in two FP64 parts before it is rounded to 62 - kb bits.
FixedPhase fixed_phase(double c, double R) {
  FixedPhase fp;
  fp.inv_R = 1.0 / R;
  const double i2p = 0.15915494309189535, i2p_lo = -9.839338337591243e-18;   // 1 / (2 pi)
  const double rhi = 1.0 / fp.inv_R, rlo = fma(-rhi, fp.inv_R, 1.0) / fp.inv_R;   // 1 / inv_R
  const double a = c * rhi, al = fma(c, rhi, -a) + c * rlo;
  const double k = a * i2p, kl = fma(a, i2p, -k) + (a * i2p_lo + al * i2p);
  fp.kb = 0;
  while (ldexp(1.0, fp.kb) <= fabs(k)) ++fp.kb;
  fp.K = llrint(ldexp(k, 62 - fp.kb)) + llrint(ldexp(kl, 62 - fp.kb));
  return fp;
}

// Largest distance between two points of the panels (vertices that no panel has do not count), from
// above: the smaller of their box's diagonal and twice the largest distance of a vertex from the
// box's centre.
double mesh_reach(bem_ctx* ctx) {
  if (ctx->reach_version == ctx->mesh_version) return ctx->reach;
  double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  const std::vector<double>& p = ctx->h_xyz;
  std::vector<char> used(p.size() / 3, 0);
  for (const int32_t v : ctx->h_tri) used[v] = 1;
  for (size_t v = 0; v < used.size(); ++v)
    if (used[v])
      for (int c = 0; c < 3; ++c) {
        lo[c] = std::min(lo[c], p[3 * v + c]);
        hi[c] = std::max(hi[c], p[3 * v + c]);
      }
  double far2 = 0.0, diag2 = 0.0;
  for (int c = 0; c < 3; ++c) diag2 += (hi[c] - lo[c]) * (hi[c] - lo[c]);
  for (size_t v = 0; v < used.size(); ++v) {
    if (!used[v]) continue;
    double d2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      const double d = p[3 * v + c] - 0.5 * (lo[c] + hi[c]);
      d2 += d * d;
    }
    far2 = std::max(far2, d2);
  }
  ctx->reach = std::min(sqrt(diag2), 2.0 * sqrt(far2)) * (1.0 + 1e-12);
  ctx->reach_version = ctx->mesh_version;
  return ctx->reach;
}

// Terms after which the series of e^{i d r}, |d| <= dmax, on [0, R] is below 2^-56 of the
// function's size (coefficients bounded by 2 (kappa / 2)^m / m!, kappa = dmax R / 2); the
// factors r and r^2 of the other families cost two more.
int series_terms(double dmax, double R) {
  const double h = 0.25 * dmax * R;
  if (!(h < 8.0)) return kMaxTerms + 1;
  double t = 2.0;
  int m = 0;
  while (t > 0x1p-56 && m <= kMaxTerms) {
    ++m;
    t *= h / m;
  }
  return m;   // h = 0: the constant alone
}

}  // namespace

ExpandPlan expand_plan(bem_ctx* ctx, int nk, const double* k, double c_re, double c_im, int ncols,
                       bool nodes, bool deriv, int arith) {
  ExpandPlan p;
  const OpCoef& op = ctx->op;
  const bool hasG = op.cgr != 0.0 || op.cgi != 0.0, hasH = op.chr != 0.0 || op.chi != 0.0;
  const int64_t n = ctx->geo.n;
  if (n < (nodes ? kMinNodes : kMinColumns)) return p;
  p.R = mesh_reach(ctx);
  if (!(p.R > 0.0) || !isfinite(p.R) || !isfinite(1.0 / p.R)) return p;
  double dmax = 0.0, growth = 0.0;
  for (int j = 0; j < nk; ++j) {
    dmax = std::max(dmax, hypot(k[2 * j] - c_re, k[2 * j + 1] - c_im));
    growth = std::max(growth, fabs(k[2 * j + 1] - c_im));
  }
  // (double-FP32 residuals, good to 1e-13, have the projections' bound)
  const double max_growth = nodes || arith == 1 ? kMaxGrowthNodes : kMaxGrowthColumns;
  p.M = series_terms(dmax, p.R);
  // about a real centre no exponential is evaluated: for values near the axis, at most a term more
  if (c_im != 0.0 && series_terms(dmax + fabs(c_im), p.R) <= p.M + 1 &&
      (growth + fabs(c_im)) * p.R <= max_growth) {
    dmax += fabs(c_im);
    growth += fabs(c_im);
    c_im = 0.0;
    p.M = series_terms(dmax, p.R);
  }
  if (!(growth * p.R <= max_growth)) return p;
  p.c = make_double2(c_re, c_im);
  if (!(fabs(c_re) * p.R <= kMaxPhase)) return p;
  p.phase = fixed_phase(c_re, p.R);
  if (p.M < 1 || p.M > kMaxTerms) return p;
  p.hasG = hasG;
  p.nh = hasH ? (deriv ? 1 : 2) : 0;
  p.fams = (hasG ? 1 : 0) + p.nh;
  p.deriv = deriv;
  p.S = p.fams * p.M;
  const int tn = ncols <= 8 ? 8 : 32;
  const double padded = (double)((ncols + tn - 1) / tn * tn);
  p.split = (double)n * (double)n * p.S * (padded - 4.0) >= kSplitWork;
  // Time per entry of the two forms, in FP64 operations (5.3e11 a second); the smaller wins. The
  // evaluation's integer instructions count a 28th, as measured (5120 panels, 14 terms: 222
  // together), the split products 7 a moment and 4 per 32 columns. The direct forms take ~1950 a
  // column for residuals (4800 panels, one vector: 85 ms, expanded 12.4 ms) and 540 + 4 nu a node
  // or more for projections (768 panels, 64 columns: 1000).
  auto evaluation = [&](int fams) {
    return fams == 0 ? 0.0 : 7.0 * (15.0 + (p.c.y != 0.0 ? 22.0 : 0.0) + (110.0 + (12.0 + 14.0 * fams) * p.M) / 28.0);
  };
  p.cost = evaluation(hasG ? 1 : 0) + evaluation(p.nh) + (p.split ? p.S * (7.0 + 4.0 * ((ncols + 31) / 32)) : 3.0 * p.S * padded);
  const double expand = p.cost;
  const double direct = nodes ? nk * (7.0 * 77.0 + 4.0 * ncols) : ncols * 1950.0;
  if (!(expand < direct)) return p;
  // workspace: coefficients, moments of kc columns, slot products (per k split)
  p.kc = (int)std::min<int64_t>(n, std::max<int64_t>(32, (int64_t)(kMomentBytes / ((size_t)p.S * n * 16))));
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  const int64_t tiles = (n + kTM - 1) / kTM * ((ncols + tn - 1) / tn) * p.S;
  if (p.split) {
    p.kc = (int)std::min<int64_t>(n, std::max<int64_t>(64, (int64_t)(kMomentBytes / ((size_t)p.S * n * 16)) / 16 * 16));
    p.batch = split64_batch_plan(n, p.kc, p.S, ncols);
  }
  // enough blocks for eight small blocks on each SM, at least 64 columns each
  p.splits = p.split ? 1 : (int)std::max<int64_t>(1, std::min<int64_t>(8 * (int64_t)std::max(1, sms) / tiles, p.kc / 64));
  auto up = [](size_t b) { return (b + 255) / 256 * 256; };
  p.coef_off = kAngles * sizeof(int4);   // (the angles' table first)
  p.mom_off = p.coef_off + up((size_t)p.S * nk * 16);
  p.y_off = p.mom_off + up((size_t)p.S * p.kc * n * 16);
  p.batch_off = p.y_off + up((size_t)p.splits * p.S * n * ncols * 16);
  p.bytes = p.batch_off + p.batch.bytes;
  p.use = p.bytes <= kMaxWork;
  p.near_off = up(p.bytes);
  if (near_active(ctx)) p.bytes = p.near_off + near_expand_bytes(ctx, p, ncols);
  return p;
}

namespace {

// The slot products Y_s = G_s X into the workspace, near-field corrections included.
bem_status expand_products(bem_ctx* ctx, const ExpandPlan& p, int nk, const double* k_dev,
                     const double* X, int64_t ldx, int ncols, char* work, cudaStream_t s) {
  const int64_t n = ctx->geo.n;
  double2* a = reinterpret_cast<double2*>(work + p.coef_off);
  double2* G = reinterpret_cast<double2*>(work + p.mom_off);
  double2* Yp = reinterpret_cast<double2*>(work + p.y_off);
  expand_coef_kernel<<<dim3((unsigned)nk, (unsigned)p.fams), kCoefThreads, 0, s>>>(
      reinterpret_cast<const double2*>(k_dev), nk, p.c, p.R, p.M, p.hasG, p.deriv, ctx->op, a);
  // the single layer's family and the double layer's by a launch each (the sums of three do not fit
  // the registers)
  const MomentKernel single = p.deriv ? moment_kernel<kSingleDeriv>(p.M) : moment_kernel<kSingle>(p.M);
  const MomentKernel dbl = p.deriv ? moment_kernel<kDoubleDeriv>(p.M) : moment_kernel<kDouble>(p.M);
  int4* angles = reinterpret_cast<int4*>(work);
  expand_angles_kernel<<<kAngles / 128, 128, 0, s>>>(angles);
  const FixedPhase fp = p.phase;
  ctx->launches += 2;
  const double2* Xd = reinterpret_cast<const double2*>(X);
  if (p.split) {
    const bem_status st = split64_batch_scales(ctx, p.batch, work + p.batch_off, Xd, ldx, s);
    if (st != BEM_OK) return st;
  }
  for (int64_t l0 = 0; l0 < n; l0 += p.kc) {
    const int kc = (int)std::min<int64_t>(p.kc, n - l0);
    const dim3 ge((unsigned)((n + kRowsE - 1) / kRowsE), (unsigned)((kc + kColsE - 1) / kColsE));
    if (p.hasG) single<<<ge, kRowsE, 0, s>>>(ctx->geo, p.c, fp, p.M, l0, kc, angles, G);
    if (p.nh > 0)
      dbl<<<ge, kRowsE, 0, s>>>(ctx->geo, p.c, fp, p.M, l0, kc, angles, G + (p.hasG ? (int64_t)p.M * kc * n : 0));
    ctx->launches += (p.hasG ? 1 : 0) + (p.nh > 0 ? 1 : 0);
    if (p.split) {
      const bem_status st = split64_batch(ctx, p.batch, work + p.batch_off, G, (int64_t)kc * n, kc,
                                          Xd + l0, ldx, l0 > 0, Yp, s);
      if (st != BEM_OK) return st;
      continue;
    }
    const int tn = ncols <= 8 ? 8 : 32;
    const dim3 gp((unsigned)((n + kTM - 1) / kTM), (unsigned)((ncols + tn - 1) / tn),
                  (unsigned)(p.S * p.splits));
    auto* pk = tn == 8 ? expand_product_kernel<8> : expand_product_kernel<32>;
    pk<<<gp, kThreadsM, 0, s>>>(G, n, kc, p.S, p.splits, Xd, ldx,
                                ncols, l0, l0 > 0, Yp);
    ctx->launches++;
  }
  if (p.splits > 1) {
    const int64_t count = (int64_t)p.S * n * ncols;
    expand_sum_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(count, p.splits, Yp);
    ctx->launches++;
  }
  return near_active(ctx) ? near_expand64(ctx, p, angles, X, ldx, ncols, Yp, work + p.near_off, s)
                          : BEM_OK;
}

}  // namespace

bem_status expand_apply_nodes(bem_ctx* ctx, const ExpandPlan& p, const double* V, int64_t ldv,
                               int nu, double* Y, void* work, cudaStream_t s) {
  char* w = static_cast<char*>(work);
  const int N = ctx->con.N;
  const int64_t n = ctx->geo.n;
  const bem_status st = expand_products(ctx, p, N, ctx->con.z, V, ldv, nu, w, s);
  if (st != BEM_OK) return st;
  const dim3 g((unsigned)((n * nu + 127) / 128), (unsigned)((N + kNodesC - 1) / kNodesC));
  expand_nodes_kernel<<<g, 128, 0, s>>>(reinterpret_cast<const double2*>(w + p.y_off), n, nu, p.M,
                                        p.fams, N, reinterpret_cast<const double2*>(w + p.coef_off),
                                        reinterpret_cast<const double2*>(ctx->con.self),
                                        reinterpret_cast<const double2*>(V), ldv,
                                        reinterpret_cast<double2*>(Y));
  ctx->launches++;
  return cuda_check(ctx, cudaGetLastError(), "expanded products");
}

bem_status expand_apply_columns(bem_ctx* ctx, const ExpandPlan& p, int m, const double* lam_dev,
                                 const double* X, int64_t ldx, double* R, void* work, cudaStream_t s) {
  char* w = static_cast<char*>(work);
  const int64_t n = ctx->geo.n;
  bem_status st = cuda_check(ctx, launch_self_at(ctx, m, lam_dev, R, p.deriv, s), "self terms");
  if (st == BEM_OK) st = expand_products(ctx, p, m, lam_dev, X, ldx, m, w, s);
  if (st != BEM_OK) return st;
  expand_columns_kernel<<<(unsigned)((n * m + 127) / 128), 128, 0, s>>>(
      reinterpret_cast<const double2*>(w + p.y_off), n, m, p.M, p.fams,
      reinterpret_cast<const double2*>(w + p.coef_off), reinterpret_cast<const double2*>(X), ldx,
      reinterpret_cast<double2*>(R));
  ctx->launches++;
  return cuda_check(ctx, cudaGetLastError(), "expanded products");
}

}  // namespace bem
