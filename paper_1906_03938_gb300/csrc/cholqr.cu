// CholeskyQR2 orthonormalisation of the Ritz basis.
//
// The paper orthonormalises the basis U before the Rayleigh-Ritz projection (Section 4,
// Example 1). CholeskyQR2: G = V^H V, G = R^H R (R upper, positive diagonal),
// V <- V R^{-1}, and the same once more, which restores orthogonality to working
// precision for well-conditioned V. All steps are deterministic (fixed-order sums).
// FP64 runs at a small fraction of the FP32 rate on this part, so the FP64 work is kept to
// the Gram matrix and the multiplication by the inverse factor: the first pass factors in
// FP32, and the second pass, whose Gram matrix is then near the identity, obtains its
// inverse factor from a few small products instead of a sequential factorisation.
#include <math.h>

#include <algorithm>

#include "internal.h"
#include "sm100.cuh"
#include "split64.h"

namespace bem {
namespace {

// In-place Cholesky of the Hermitian nu x nu matrix G (column-major, upper triangle used):
// on exit the upper triangle holds R with G = R^H R, the strict lower triangle is zero.
// A pivot below 1e-13 of the largest diagonal entry of G counts as loss of rank. One block;
// G is staged in shared memory when the dynamic allocation holds it (nu <= 64).
// With `deficient` non-null, a collapsed pivot does not fail: its column of R becomes the
// unit vector (the column of V is then replaced by the caller) and deficient[k] = 1.
__global__ void __launch_bounds__(1024) cholesky_kernel(double2* Gg, int nu, int* status,
                                                        int* deficient, const int* gate) {
  if (gate && *gate == 0) return;   // gated pass not needed
  extern __shared__ double2 sG[];
  __shared__ double rkk, dmax;
  const bool staged = nu <= 64;
  double2* G = staged ? sG : Gg;
  const int tid = threadIdx.x;
  if (staged)
    for (int t = tid; t < nu * nu; t += blockDim.x) sG[t] = Gg[t];
  __syncthreads();
  if (tid == 0) {
    dmax = 0.0;
    for (int k = 0; k < nu; ++k) dmax = fmax(dmax, G[(int64_t)k * nu + k].x);
  }
  __syncthreads();
  bool failed = false;
  for (int k = 0; k < nu; ++k) {
    if (tid == 0) {
      const double d = G[(int64_t)k * nu + k].x;
      if (!(d > 1e-13 * dmax) || !isfinite(d)) {
        if (deficient) {
          deficient[k] = 1;
          rkk = -1.0;   // marker: unit column, no trailing update
        } else {
          atomicOr(status, kStatusNotSPD);
          rkk = 0.0;
        }
      } else {
        if (deficient) deficient[k] = 0;
        rkk = sqrt(d);
      }
      G[(int64_t)k * nu + k] = make_double2(rkk < 0.0 ? 1.0 : rkk, 0.0);
    }
    __syncthreads();
    if (rkk == 0.0) {
      failed = true;
      break;
    }
    if (rkk < 0.0) {
      for (int jj = k + 1 + tid; jj < nu; jj += blockDim.x)
        G[(int64_t)jj * nu + k] = make_double2(0.0, 0.0);
      __syncthreads();
      continue;
    }
    for (int jj = k + 1 + tid; jj < nu; jj += blockDim.x) {
      double2 g = G[(int64_t)jj * nu + k];
      G[(int64_t)jj * nu + k] = make_double2(g.x / rkk, g.y / rkk);
    }
    __syncthreads();
    // trailing update of the upper triangle: G_ij -= conj(R_ki) R_kj, k < i <= j
    const int m = nu - k - 1;
    const int64_t total = (int64_t)m * m;
    for (int64_t t = tid; t < total; t += blockDim.x) {
      const int i = k + 1 + (int)(t % m);
      const int jj = k + 1 + (int)(t / m);
      if (i > jj) continue;
      const double2 a = G[(int64_t)i * nu + k];
      const double2 b = G[(int64_t)jj * nu + k];
      double2 g = G[(int64_t)jj * nu + i];
      g.x -= a.x * b.x + a.y * b.y;
      g.y -= a.x * b.y - a.y * b.x;
      G[(int64_t)jj * nu + i] = g;
    }
    __syncthreads();
  }
  for (int64_t t = tid; t < (int64_t)nu * nu; t += blockDim.x) {
    const int i = (int)(t % nu), jj = (int)(t / nu);
    const double2 v = (i > jj) ? make_double2(0.0, 0.0) : G[t];
    Gg[t] = failed ? make_double2(NAN, NAN) : v;
  }
}

// Columns flagged deficient get fresh pseudo-random entries (SplitMix64 of seed, index).
__global__ void refresh_columns_kernel(double2* V, int64_t ldv, int64_t n, int nu,
                                       const int* deficient, uint64_t seed) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n * nu) return;
  const int c = (int)(t / n);
  if (!deficient[c]) return;
  const int64_t r = t % n;
  uint64_t a = seed + (2 * (uint64_t)t + 1) * 0x9E3779B97F4A7C15ull;
  uint64_t b = seed + (2 * (uint64_t)t + 2) * 0x9E3779B97F4A7C15ull;
  a = (a ^ (a >> 30)) * 0xBF58476D1CE4E5B9ull; a = (a ^ (a >> 27)) * 0x94D049BB133111EBull; a ^= a >> 31;
  b = (b ^ (b >> 30)) * 0xBF58476D1CE4E5B9ull; b = (b ^ (b >> 27)) * 0x94D049BB133111EBull; b ^= b >> 31;
  V[(int64_t)c * ldv + r] = make_double2((double)(a >> 11) * 0x1.0p-52 - 1.0,
                                         (double)(b >> 11) * 0x1.0p-52 - 1.0);
}

constexpr int kGT = 32;   // Gram output tile
constexpr int kGR = 16;   // rows of V staged at a time by the FP64 Gram kernel

// Tile pair (ta, tb), ta <= tb, of the idx-th upper tile: tb = 0, 1, ..., ta = 0..tb.
__device__ __forceinline__ void upper_tile(int idx, int& ta, int& tb) {
  int b = 0;
  while ((b + 1) * (b + 2) / 2 <= idx) ++b;
  tb = b;
  ta = idx - b * (b + 1) / 2;
}

// Partial Gram matrices, FP64: block (tile, r) sums conj(V[i][a]) V[i][b] over its row
// range for the upper tiles only (the Gram matrix is Hermitian; every consumer reads the
// upper triangle). Three real products per complex term: with x = V[i][a], y = V[i][b],
// conj(x) y = (S1 + S2) + i (S3 - S1 + S2), S1 = x.re y.re, S2 = x.im y.im,
// S3 = (x.re - x.im)(y.re + y.im); the sums of the parts are formed once per staged element.
__global__ void __launch_bounds__(256)
gram_partial_kernel(const double2* __restrict__ V, int64_t ldv, int64_t n, int nu,
                    int64_t rows_per_part, double2* __restrict__ part, const int* gate) {
  if (gate && *gate == 0) return;
  __shared__ double xr[kGR][kGT + 1], xi[kGR][kGT + 1], xd[kGR][kGT + 1];
  __shared__ double yr[kGR][kGT + 1], yi[kGR][kGT + 1], ys[kGR][kGT + 1];
  int ta, tb;
  upper_tile(blockIdx.x, ta, tb);
  const int64_t r_begin = (int64_t)blockIdx.y * rows_per_part;
  const int64_t r_end = min(n, r_begin + rows_per_part);
  const int tid = threadIdx.x;
  const int oa = tid % kGT, ob0 = tid / kGT;
  double s1[4], s2[4], s3[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) s1[m] = s2[m] = s3[m] = 0.0;
  for (int64_t r0 = r_begin; r0 < r_end; r0 += kGR) {
    __syncthreads();
    for (int x = tid; x < kGR * kGT; x += 256) {
      const int rr = x % kGR, cc = x / kGR;
      const int64_t r = r0 + rr;
      const int a = ta * kGT + cc, b = tb * kGT + cc;
      const double2 va = (r < r_end && a < nu) ? V[(int64_t)a * ldv + r] : make_double2(0.0, 0.0);
      const double2 vb = (r < r_end && b < nu) ? V[(int64_t)b * ldv + r] : make_double2(0.0, 0.0);
      xr[rr][cc] = va.x;
      xi[rr][cc] = va.y;
      xd[rr][cc] = va.x - va.y;
      yr[rr][cc] = vb.x;
      yi[rr][cc] = vb.y;
      ys[rr][cc] = vb.x + vb.y;
    }
    __syncthreads();
    const int rows = (int)(r_end - r0 < kGR ? r_end - r0 : kGR);
    for (int rr = 0; rr < rows; ++rr) {
      const double ar = xr[rr][oa], ai = xi[rr][oa], ad = xd[rr][oa];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int cb = ob0 + 8 * m;
        s1[m] = fma(ar, yr[rr][cb], s1[m]);
        s2[m] = fma(ai, yi[rr][cb], s2[m]);
        s3[m] = fma(ad, ys[rr][cb], s3[m]);
      }
    }
  }
  const int a = ta * kGT + oa;
  if (a < nu) {
    double2* P = part + (int64_t)blockIdx.y * nu * nu;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int b = tb * kGT + ob0 + 8 * m;
      if (b < nu) P[(int64_t)b * nu + a] = make_double2(s1[m] + s2[m], s3[m] - s1[m] + s2[m]);
    }
  }
}

// Partial Gram matrices in FP32 (first pass), upper tiles; partial sums stored as double2.
__global__ void __launch_bounds__(256)
gram_partial32_kernel(const double2* __restrict__ V, int64_t ldv, int64_t n, int nu,
                      int64_t rows_per_part, double2* __restrict__ part) {
  __shared__ float2 sX[kGT][kGT + 1];
  __shared__ float2 sY[kGT][kGT + 1];
  int ta, tb;
  upper_tile(blockIdx.x, ta, tb);
  const int64_t r_begin = (int64_t)blockIdx.y * rows_per_part;
  const int64_t r_end = min(n, r_begin + rows_per_part);
  const int tid = threadIdx.x;
  const int oa = tid % kGT, ob0 = tid / kGT;
  float2 acc[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) acc[m] = make_float2(0.f, 0.f);
  for (int64_t r0 = r_begin; r0 < r_end; r0 += kGT) {
    __syncthreads();
    for (int x = tid; x < kGT * kGT; x += 256) {
      const int rr = x % kGT, cc = x / kGT;
      const int64_t r = r0 + rr;
      const int a = ta * kGT + cc, b = tb * kGT + cc;
      double2 va = make_double2(0.0, 0.0), vb = va;
      if (r < r_end && a < nu) va = V[(int64_t)a * ldv + r];
      if (r < r_end && b < nu) vb = V[(int64_t)b * ldv + r];
      sX[rr][cc] = make_float2((float)va.x, (float)va.y);
      sY[rr][cc] = make_float2((float)vb.x, (float)vb.y);
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < kGT; ++rr) {
      const float2 x = sX[rr][oa];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float2 y = sY[rr][ob0 + 8 * m];
        acc[m].x = fmaf(x.x, y.x, fmaf(x.y, y.y, acc[m].x));
        acc[m].y = fmaf(x.x, y.y, fmaf(-x.y, y.x, acc[m].y));
      }
    }
  }
  const int a = ta * kGT + oa;
  if (a < nu) {
    double2* P = part + (int64_t)blockIdx.y * nu * nu;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int b = tb * kGT + ob0 + 8 * m;
      if (b < nu) P[(int64_t)b * nu + a] = make_double2(acc[m].x, acc[m].y);
    }
  }
}

// G = sum of the partials (deterministic): eight threads per element, thread q adding the
// parts q, q + 8, ... in order, then a fixed shuffle tree. Elements of lower tiles are not
// formed. epsp, if given: the block's sum of |G - I|^2 (off-diagonal entries twice).
__global__ void __launch_bounds__(256)
sum_parts_kernel(const double2* __restrict__ part, int parts, int nu, double2* __restrict__ G,
                 float* __restrict__ epsp, const int* gate) {
  if (gate && *gate == 0) return;
  __shared__ float red[32];
  const int64_t count = (int64_t)nu * nu;
  const int64_t gt = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t t = gt / 8;
  const int q = (int)(gt % 8);
  double2 sum = make_double2(0.0, 0.0);
  bool live = t < count;
  if (live) {
    const int a = (int)(t % nu), b = (int)(t / nu);
    live = a / kGT <= b / kGT;
  }
  if (live)
    for (int r = q; r < parts; r += 8) {
      const double2 v = part[(int64_t)r * count + t];
      sum.x += v.x;
      sum.y += v.y;
    }
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) {
    sum.x += __shfl_xor_sync(0xffffffffu, sum.x, off);
    sum.y += __shfl_xor_sync(0xffffffffu, sum.y, off);
  }
  if (live && q == 0) G[t] = sum;
  if (!epsp) return;
  if (q == 0) {
    const int a = (int)(t % nu), b = (int)(t / nu);
    const float er = (float)(sum.x - (a == b ? 1.0 : 0.0)), ei = a == b ? 0.f : (float)sum.y;
    red[threadIdx.x / 8] = live && a <= b ? (er * er + ei * ei) * (a == b ? 1.f : 2.f) : 0.f;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    float e2 = red[threadIdx.x];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, off);
    if (threadIdx.x == 0) epsp[blockIdx.x] = e2;
  }
}

// FP32 first-pass factor: Z = R^{-1} for G = R^H R (nu <= 128; wider ones in two diagonal
// blocks, chol_block32_kernel), one block, by Gaussian elimination of [G | I] without pivoting:
// the left part becomes D L^H and the right part L^{-1} (G = L D L^H, L unit lower), so
// Z = L^{-H} D^{-1/2}. Element (r, c) of the working matrix is the trailing G[r][c] for r >= c
// and W[c][r], W = L^{-1}, for r < c; step k changes only columns c > k and reads column k. A
// pivot below 1e-6 of the largest diagonal entry (of Gd, nd columns) sets *fallback (V too
// ill-conditioned for an FP32 pass) and Z is not written.
//
// nu dependent steps of little work each: kGrid x kGrid threads keep kT x kT elements each in
// registers (rows and columns kGrid apart, so that the shrinking part stays spread over all
// warps), and only the next column goes through shared memory, in two buffers with one barrier a
// step. With the whole matrix in shared memory its bandwidth set the time: 41 us at nu = 64,
// 237 us at 128; now 29 us and 107 us. Run by the first kGrid^2 threads of a block.
template <int kGrid, int kT>   // nu <= kGrid kT
__device__ void chol_inv32_block(const double2* Gg, int ldg, int nu, const double2* Gd, int nd,
                                 double2* __restrict__ Z, int ldz, int* fallback) {
  __shared__ float2 col[2][kGrid * kT];
  __shared__ float diag[kGrid * kT];
  __shared__ float dmax_s;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int tr = lane % 8 + 8 * (w % (kGrid / 8)), tc = lane / 8 + 4 * (w / (kGrid / 8));
  auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(kGrid * kGrid) : "memory"); };
  float2 g[kT][kT];   // [row slot][column slot]
#pragma unroll
  for (int i = 0; i < kT; ++i)
#pragma unroll
    for (int j = 0; j < kT; ++j) {
      const int r = tr + kGrid * i, c = tc + kGrid * j;
      g[i][j] = make_float2(0.f, 0.f);
      if (r >= c && r < nu) {
        const double2 v = __ldcg(Gg + (int64_t)r * ldg + c);   // G[r][c] = conj(G[c][r])
        g[i][j] = make_float2((float)v.x, -(float)v.y);
      }
    }
  if (tid < 32) {
    float m = 0.f;
    for (int k = tid; k < nd; k += 32) m = fmaxf(m, (float)__ldcg(Gd + (int64_t)k * nd + k).x);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if (tid == 0) dmax_s = m;
  }
  if (tc == 0)
#pragma unroll
    for (int i = 0; i < kT; ++i) col[0][tr + kGrid * i] = g[i][0];
  sync();
  const float dmax = dmax_s;
  for (int k = 0; k < nu; ++k) {
    const float2* s = col[k & 1];
    const float d = s[k].x;
    if (!(d > 1e-6f * dmax) || !isfinite(d)) {
      if (tid == 0) *fallback = 1;
      return;   // d is the same for every thread: the whole block leaves
    }
    if (tid == 0) diag[k] = d;
    const float rd = 1.f / d;
    float2 a[kT];   // column k at this thread's rows: G[r][k], 1 at r = k, W[k][r] above
#pragma unroll
    for (int i = 0; i < kT; ++i) a[i] = tr + kGrid * i == k ? make_float2(1.f, 0.f) : s[tr + kGrid * i];
#pragma unroll
    for (int j = 0; j < kT; ++j) {
      if (kGrid * j + kGrid - 1 <= k) continue;
      const int c = tc + kGrid * j;
      float2 l = s[c];
      l = c > k ? make_float2(l.x * rd, l.y * rd) : make_float2(0.f, 0.f);   // L[c][k]
#pragma unroll
      for (int i = 0; i < kT; ++i) {
        if (i < j && kGrid * i > k) continue;
        const int r = tr + kGrid * i;
        // r >= c: G[r][c] -= G[r][k] conj(L[c][k]); r <= k: W[c][r] -= L[c][k] W[k][r]
        const float ly = r >= c ? -l.y : l.y;
        if (r >= c || r <= k) {
          g[i][j].x -= a[i].x * l.x - a[i].y * ly;
          g[i][j].y -= a[i].x * ly + a[i].y * l.x;
        }
      }
      if (c == k + 1)
#pragma unroll
        for (int i = 0; i < kT; ++i) col[(k + 1) & 1][tr + kGrid * i] = g[i][j];
    }
    sync();
  }
  // Z[c][k] = conj(W[k][c]) / sqrt(d_k) for c <= k, zero below the diagonal
#pragma unroll
  for (int j = 0; j < kT; ++j) {
    const int c = tc + kGrid * j;
    if (c >= nu) continue;
    const float inv = 1.f / sqrtf(diag[c]);
#pragma unroll
    for (int i = 0; i < kT; ++i) {
      const int r = tr + kGrid * i;
      if (r >= nu) continue;
      Z[(int64_t)c * ldz + r] = r > c ? make_double2(0.0, 0.0)
                                : r == c ? make_double2(inv, 0.0)
                                         : make_double2(g[i][j].x * inv, -g[i][j].y * inv);
    }
  }
}

template <int kT>
__global__ void __launch_bounds__(1024)
chol_inv32_kernel(const double2* __restrict__ Gg, int ldg, int nu, const double2* __restrict__ Gd,
                  int nd, double2* __restrict__ Z, int ldz, int* fallback, const int* gate) {
  if ((gate && *gate == 0) || *fallback != 0) return;
  __syncthreads();   // (read by every thread before one may set it)
  chol_inv32_block<32, kT>(Gg, ldg, nu, Gd, nd, Z, ldz, fallback);
}

// Inverse factor of a wider Gram matrix from two diagonal blocks, G = [G11 G12; . G22] at
// kChol32 columns: Z11 = chol_inv32(G11), W = Z11^H G12 (= R12), S = G22 - W^H W,
// Z22 = chol_inv32(S), T = W Z22, Z12 = -Z11 T. FP32 products (the first pass only has to make V
// well conditioned); one thread per entry, 16 x 16 a block.
//  kMode 0: W (h x r), 1: S (upper, r x r), 2: T (h x r), 3: Z12, with h = kChol32, r = nu - h.
constexpr int kChol32 = 128;

template <int kMode>
__global__ void __launch_bounds__(256)
chol_block32_kernel(const double2* __restrict__ G, double2* __restrict__ Z, int nu,
                    double2* __restrict__ W, double2* __restrict__ S, double2* __restrict__ T,
                    const int* fallback, const int* gate) {
  if ((gate && *gate == 0) || *fallback != 0) return;
  constexpr int h = kChol32;
  const int r = nu - h;
  const int i = blockIdx.x * 16 + threadIdx.x % 16, j = blockIdx.y * 16 + threadIdx.x / 16;
  if (j >= r || i >= (kMode == 1 ? r : h)) return;
  float2 acc = make_float2(0.f, 0.f);
  auto f2of = [](double2 v) { return make_float2((float)v.x, (float)v.y); };
  auto mac = [&](float2 a, float2 b) {   // a b
    acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
    acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
  };
  auto cj = [](float2 a) { return make_float2(a.x, -a.y); };
  if (kMode == 0) {
    for (int k = 0; k <= i; ++k)
      mac(cj(f2of(Z[(int64_t)i * nu + k])), f2of(G[(int64_t)(h + j) * nu + k]));
    W[(int64_t)j * h + i] = make_double2(acc.x, acc.y);
  } else if (kMode == 1) {
    if (i > j) return;
    for (int k = 0; k < h; ++k)
      mac(cj(f2of(W[(int64_t)i * h + k])), f2of(W[(int64_t)j * h + k]));
    const double2 g = G[(int64_t)(h + j) * nu + h + i];
    S[(int64_t)j * r + i] = make_double2(g.x - acc.x, i == j ? 0.0 : g.y - acc.y);
  } else if (kMode == 2) {
    for (int k = 0; k <= j; ++k)
      mac(f2of(W[(int64_t)k * h + i]), f2of(Z[(int64_t)(h + j) * nu + h + k]));
    T[(int64_t)j * h + i] = make_double2(acc.x, acc.y);
  } else {
    for (int k = i; k < h; ++k)
      mac(f2of(Z[(int64_t)k * nu + i]), f2of(T[(int64_t)j * h + k]));
    Z[(int64_t)(h + j) * nu + i] = make_double2(-acc.x, -acc.y);
  }
}

// ||G - I||_F up to which the near-identity factor is used; its error is O(||G - I||^4)
// (at 8e-4 it still matches the Cholesky factor to rounding)
constexpr float kNearEps = 5e-4f;
// ||G - I||_F up to which the first step alone is exact to rounding
constexpr float kNearEpsSmall = 1e-5f;

// ---- second pass near the identity ----
//
// After a first pass G = V^H V = I + E with ||E|| small. The inverse factor Z = R^{-1} is
// I + Y with Y upper triangular with a real diagonal, and Z^H G Z = I reads
// Y + Y^H = -H(Y), H(Y) = E + Y^H E + E Y + Y^H Y + Y^H E Y. The fixed point
// Y <- -U(H(Y)) (U keeps the strict upper triangle and half the diagonal) gains one order
// of ||E|| per step: Y0 = -U(E) is exact to O(||E||^2), Y1 (without the cubic term) to
// O(||E||^3) and Y2 to O(||E||^4). Only small products are needed, spread over many
// blocks, instead of a sequential Cholesky factorisation and triangular inverse.

// E entry (m, j) from the upper triangle of G.
__device__ __forceinline__ double2 e_entry(const double2* G, int nu, int m, int j) {
  if (m <= j) {
    const double2 g = G[(int64_t)j * nu + m];
    return make_double2(g.x - (m == j ? 1.0 : 0.0), m == j ? 0.0 : g.y);
  }
  const double2 g = G[(int64_t)m * nu + j];
  return make_double2(g.x, -g.y);
}

// Y0 = -U(E) entry (m, i), m <= i.
__device__ __forceinline__ double2 y_entry(const double2* G, int nu, int m, int i) {
  const double2 g = G[(int64_t)i * nu + m];
  return m < i ? make_double2(-g.x, -g.y) : make_double2(-0.5 * (g.x - 1.0), 0.0);
}

constexpr int kNT = 8;     // output tile of the near-identity products (kNT x kNT per block)
constexpr int kNM = 16;    // inner-dimension chunk staged in shared memory

// Tiled small products of the near-identity factor's second step; one 8 x 8 output tile per
// block of 64 threads, the inner dimension staged 16 at a time in shared memory.
//  kMode 1: P = Y^H E, Q = Y^H Y for the explicit Y;
//  kMode 2: Z = I + Y2, Y2 = -U(E + P + P^H + Q + P Y) (P, Q, Y of mode 1).
template <int kMode>
__global__ void __launch_bounds__(64)
near_tile_kernel(const double2* __restrict__ G, const double2* __restrict__ Y,
                 const double2* __restrict__ Pin, const double2* __restrict__ Qin, int nu,
                 double2* __restrict__ P, double2* __restrict__ Q, double2* __restrict__ Z,
                 const int* gate, const int* skip_if) {
  if ((gate && *gate == 0) || (skip_if && *skip_if != 0)) return;
  __shared__ double2 sA[kNM][kNT], sB[kNM][kNT], sC[kNM][kNT];
  const int tid = threadIdx.x;
  const int ti = tid % kNT, tj = tid / kNT;
  const int i0 = blockIdx.x * kNT, j0 = blockIdx.y * kNT;
  const int i = i0 + ti, j = j0 + tj;
  double2 p = make_double2(0.0, 0.0), q = p;
  // inner index m runs to the last row where the upper-triangular factor is non-zero
  const int mend = min(nu, (kMode == 2 ? j0 : i0) + kNT);
  for (int m0 = 0; m0 < mend; m0 += kNM) {
    __syncthreads();
    for (int x = tid; x < kNM * kNT; x += 64) {
      const int mm = x / kNT, cc = x % kNT;
      const int m = m0 + mm;
      const int ic = i0 + cc, jc = j0 + cc;
      const bool mv = m < nu;
      if (kMode == 2) {
        sA[mm][cc] = (mv && ic < nu) ? Pin[(int64_t)m * nu + ic] : make_double2(0.0, 0.0);   // P(i, m)
        sB[mm][cc] = (mv && jc < nu && m <= jc) ? Y[(int64_t)jc * nu + m] : make_double2(0.0, 0.0);
      } else {
        sA[mm][cc] = (mv && ic < nu && m <= ic) ? Y[(int64_t)ic * nu + m]
                                                : make_double2(0.0, 0.0);
        sB[mm][cc] = (mv && jc < nu) ? e_entry(G, nu, m, jc) : make_double2(0.0, 0.0);
        sC[mm][cc] = (mv && jc < nu && m <= jc) ? Y[(int64_t)jc * nu + m]
                                                : make_double2(0.0, 0.0);
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int mm = 0; mm < kNM; ++mm) {
      const double2 a = sA[mm][ti], b = sB[mm][tj];
      if (kMode == 2) {   // P(i, m) Y(m, j)
        p.x += a.x * b.x - a.y * b.y;
        p.y += a.x * b.y + a.y * b.x;
      } else {            // conj(Y(m, i)) E(m, j), conj(Y(m, i)) Y(m, j)
        const double2 c = sC[mm][tj];
        p.x += a.x * b.x + a.y * b.y;
        p.y += a.x * b.y - a.y * b.x;
        q.x += a.x * c.x + a.y * c.y;
        q.y += a.x * c.y - a.y * c.x;
      }
    }
  }
  const bool in = i < nu && j < nu;
  const int64_t t = (int64_t)j * nu + i;
  if (kMode == 2) {
    if (in) {
      if (i > j) {
        Z[t] = make_double2(0.0, 0.0);
      } else {
        double2 h = e_entry(G, nu, i, j);
        const double2 pp = Pin[t], pt = Pin[(int64_t)i * nu + j], qq = Qin[t];
        h.x += pp.x + pt.x + qq.x + p.x;
        h.y += pp.y - pt.y + qq.y + p.y;
        Z[t] = i < j ? make_double2(-h.x, -h.y) : make_double2(1.0 - 0.5 * h.x, 0.0);
      }
    }
    return;
  }
  if (in) {
    P[t] = p;
    if (i <= j) Q[t] = q;
  }
}

// The first step, Y1 = -U(E + Y0^H E + E Y0 + Y0^H Y0), Y0 = -U(E). E = -(Y0 + Y0^H), so the
// second-order terms are -(Y0^H Y0 + Y0^2 + (Y0^2)^H), triangular products with a third of the
// terms. Every block first sums the block sums of |E|^2 in order:
//  ||E||_F > eps_max: the near-identity route is abandoned (*classic = 1) and a Cholesky
//    factorisation runs instead, in FP64 (classic[1] = 1) unless refused is given and *refused == 0
//    (see near_pass);
//  ||E||_F <= eps_small: Y1 is exact to rounding (its error is O(||E||^3)), Z = I + Y1 is
//    written here and the second step is skipped (*done = 1). The second-order terms are then
//    below 1e-10 and their rounding in FP32 (6e-18) far below Z's own in FP64, so they are
//    formed on the FP32 pipe (at nu = 256 42 us; all terms in FP64 took 298 + 20 us).
// One 8 x 8 output tile per block of 64 threads, upper tiles only.
template <typename T, typename T2>
__device__ __forceinline__ T2 near_second_order(const double2* __restrict__ G, int nu, int i0, int j0) {
  __shared__ T2 sA[kNM][kNT], sB[kNM][kNT], sC[kNM][kNT];   // Y0(m, i), Y0(m, j), Y0(i, m)
  const int tid = threadIdx.x, ti = tid % kNT, tj = tid / kNT;
  T2 h;
  h.x = h.y = 0;
  T tdiag = 0;   // Re of Y0^2 on the diagonal once more: its conjugate
  const int mend = min(nu, j0 + kNT);
  for (int m0 = 0; m0 < mend; m0 += kNM) {
    __syncthreads();
    for (int x = tid; x < kNM * kNT; x += 64) {
      const int mm = x / kNT, cc = x % kNT, m = m0 + mm;
      auto y0 = [&](int r, int c) {
        const double2 v = r <= c && c < nu ? y_entry(G, nu, r, c) : make_double2(0.0, 0.0);
        T2 o;
        o.x = (T)v.x;
        o.y = (T)v.y;
        return o;
      };
      sA[mm][cc] = y0(m, i0 + cc);
      sB[mm][cc] = y0(m, j0 + cc);
      sC[mm][cc] = y0(i0 + cc, m);
    }
    __syncthreads();
#pragma unroll 4
    for (int mm = 0; mm < kNM; ++mm) {
      const T2 a = sA[mm][ti], b = sB[mm][tj], c = sC[mm][ti];
      h.x += a.x * b.x + a.y * b.y + (c.x * b.x - c.y * b.y);
      h.y += a.x * b.y - a.y * b.x + (c.x * b.y + c.y * b.x);
      tdiag += c.x * b.x - c.y * b.y;
    }
  }
  if (i0 + ti == j0 + tj) h.x += tdiag;
  return h;
}

__global__ void __launch_bounds__(64)
near_y1_kernel(const double2* __restrict__ G, const float* __restrict__ epsp, int nparts, int nu,
               float eps_max, float eps_small, double2* __restrict__ Y, double2* __restrict__ Z,
               int* classic, int* done, const int* refused, const int* gate) {
  if (gate && *gate == 0) return;
  __shared__ float red[64];
  const int tid = threadIdx.x;
  float s = 0.f;
  for (int b = tid; b < nparts; b += 64) s += epsp[b];
  red[tid] = s;
  __syncthreads();
  for (int k = 32; k > 0; k >>= 1) {
    if (tid < k) red[tid] += red[tid + k];
    __syncthreads();
  }
  const float e2s = red[0];
  const bool first = blockIdx.x == 0 && blockIdx.y == 0 && tid == 0;
  if (!(e2s <= eps_max * eps_max)) {
    if (first) {
      *classic = 1;
      *done = 1;
      if (!refused || *refused != 0) classic[1] = 1;
    }
    return;
  }
  const bool small = e2s <= eps_small * eps_small;
  if (small && first) *done = 1;
  const int i0 = blockIdx.x * kNT, j0 = blockIdx.y * kNT;
  const int i = i0 + tid % kNT, j = j0 + tid / kNT;
  double2 y = make_double2(0.0, 0.0);
  if (i0 <= j0) {
    double2 h;
    if (small) {
      const float2 f = near_second_order<float, float2>(G, nu, i0, j0);
      h = make_double2(f.x, f.y);
    } else {
      h = near_second_order<double, double2>(G, nu, i0, j0);
    }
    if (i <= j && j < nu) {
      const double2 e = e_entry(G, nu, i, j);
      y = i < j ? make_double2(h.x - e.x, h.y - e.y) : make_double2(-0.5 * (e.x - h.x), 0.0);
    }
  }
  if (i >= nu || j >= nu) return;
  const int64_t t = (int64_t)j * nu + i;
  if (small)
    Z[t] = i == j ? make_double2(1.0 + y.x, 0.0) : y;
  else
    Y[t] = y;
}

// Rinv = R^{-1} for upper-triangular R: one block per column j, back substitution
// x_i = (delta_ij - sum_{m=i+1..j} R_im x_m) / R_ii for i = j..0, each sum split over the
// block's threads and combined in a fixed order (deterministic). The column lives in
// shared memory; R is read through the cache.
__global__ void __launch_bounds__(128)
triangular_inverse_kernel(const double2* __restrict__ R, int nu, double2* __restrict__ Rinv,
                          const int* gate) {
  if (gate && *gate == 0) return;
  __shared__ double2 x[kMaxNu];
  __shared__ double2 red[4];
  const int j = blockIdx.x;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  for (int i = tid; i < nu; i += blockDim.x) x[i] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int i = j; i >= 0; --i) {
    double2 acc = make_double2(0.0, 0.0);
    for (int m = i + 1 + tid; m <= j; m += blockDim.x) {
      const double2 r = R[(int64_t)m * nu + i];
      const double2 xm = x[m];
      acc.x += r.x * xm.x - r.y * xm.y;
      acc.y += r.x * xm.y + r.y * xm.x;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
      acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
    }
    if (lane == 0) red[w] = acc;
    __syncthreads();
    if (tid == 0) {
      double2 s = make_double2(i == j ? 1.0 : 0.0, 0.0);
      for (int k = 0; k < 4; ++k) {
        s.x -= red[k].x;
        s.y -= red[k].y;
      }
      const double d = R[(int64_t)i * nu + i].x;   // real positive
      x[i] = make_double2(s.x / d, s.y / d);
    }
    __syncthreads();
  }
  for (int i = tid; i < nu; i += blockDim.x) Rinv[(int64_t)j * nu + i] = x[i];
}

constexpr int kRMRows = 8;    // rows of V per block
constexpr int kRMK = 16;      // k chunk of M staged at a time

size_t right_multiply_smem(int nu) {
  return (size_t)(3 * nu * kRMRows + 3 * kRMK * (nu + 1)) * sizeof(double);
}

// V <- V M in place, M nu x nu upper triangular (column-major, zero below the diagonal);
// each block owns kRMRows complete rows of V, staged in shared memory before any is
// overwritten. Three real products per complex term: a b = (S1 - S2) + i (S3 - S1 - S2),
// S1 = a.re b.re, S2 = a.im b.im, S3 = (a.re + a.im)(b.re + b.im). kOut: outputs a thread.
template <int kOut>
__device__ __forceinline__ void multiply64_rows(double* rm_smem, double2* V, int64_t ldv, int64_t n,
                                                int nu, const double2* __restrict__ M) {
  double* vr = rm_smem;                  // [nu][kRMRows]
  double* vi = vr + nu * kRMRows;
  double* vs = vi + nu * kRMRows;
  double* mr = vs + nu * kRMRows;        // [kRMK][nu + 1]
  double* mi = mr + kRMK * (nu + 1);
  double* ms = mi + kRMK * (nu + 1);
  const int tid = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.x * kRMRows;
  for (int t = tid; t < kRMRows * nu; t += blockDim.x) {
    const int rr = t % kRMRows, c = t / kRMRows;
    const int64_t r = r0 + rr;
    const double2 v = (r < n) ? V[(int64_t)c * ldv + r] : make_double2(0.0, 0.0);
    vr[c * kRMRows + rr] = v.x;
    vi[c * kRMRows + rr] = v.y;
    vs[c * kRMRows + rr] = v.x + v.y;
  }
  const int outs = kRMRows * nu;
  double s1[kOut], s2[kOut], s3[kOut];
#pragma unroll
  for (int m = 0; m < kOut; ++m) s1[m] = s2[m] = s3[m] = 0.0;
  for (int k0 = 0; k0 < nu; k0 += kRMK) {
    const int kn = min(kRMK, nu - k0);
    __syncthreads();
    for (int t = tid; t < kRMK * nu; t += blockDim.x) {
      const int kk = t % kRMK, c = t / kRMK;
      const double2 b = kk < kn ? M[(int64_t)c * nu + k0 + kk] : make_double2(0.0, 0.0);
      mr[kk * (nu + 1) + c] = b.x;
      mi[kk * (nu + 1) + c] = b.y;
      ms[kk * (nu + 1) + c] = b.x + b.y;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kOut; ++m) {
      const int o = tid + 256 * m;
      if (o >= outs) break;
      const int c = o % nu, rr = o / nu;
      if (c < k0) continue;   // M[k][c] = 0 for k > c
      for (int kk = 0; kk < kn; ++kk) {
        const int k = k0 + kk;
        s1[m] = fma(vr[k * kRMRows + rr], mr[kk * (nu + 1) + c], s1[m]);
        s2[m] = fma(vi[k * kRMRows + rr], mi[kk * (nu + 1) + c], s2[m]);
        s3[m] = fma(vs[k * kRMRows + rr], ms[kk * (nu + 1) + c], s3[m]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < kOut; ++m) {
    const int o = tid + 256 * m;
    if (o >= outs) break;
    const int c = o % nu, rr = o / nu;
    const int64_t r = r0 + rr;
    if (r < n) V[(int64_t)c * ldv + r] = make_double2(s1[m] - s2[m], s3[m] - s1[m] - s2[m]);
  }
}

// gate, need: skip unless *gate != 0 and *need != 0; skip_if: skip when *skip_if != 0.
__global__ void __launch_bounds__(256)
right_multiply_kernel(double2* V, int64_t ldv, int64_t n, int nu, const double2* __restrict__ M,
                      const int* gate, const int* skip_if, const int* need) {
  if ((gate && *gate == 0) || (need && *need == 0) || (skip_if && *skip_if != 0)) return;
  extern __shared__ double rm_smem[];
  multiply64_rows<kMaxNu * kRMRows / 256>(rm_smem, V, ldv, n, nu, M);
}

// V <- V + V (M - I) for the near-identity factor M = I + Y (upper triangular), with the
// small product V Y in double-FP32 arithmetic on the FP32 pipe (this GPU's FP64 pipe runs at
// ~1/65 of its rate). Each FP64 value x is carried as hi + lo, hi = fl32(x),
// lo = fl32(x - hi); the product hi_v hi_y is formed exactly (its rounding error recovered by
// an FMA) and added to the running sum by an error-free two-sum; the error terms and the
// hi x lo cross products gather in an FP32 companion, whose own rounding leaves a relative
// error of ~1e-13 of the sum of the terms' magnitudes. Since ||Y|| <= ~||G - I|| (at most
// 5e-4 on this route, ~1e-6 after an FP32 first pass), that is ~1e-17 of |V| or less: below
// V's own FP64 rounding, which the final FP64 addition V + V Y then sets.
// Same blocking as right_multiply_kernel: kRMRows complete rows per block, staged first.
// gate: skip unless *gate != 0; skip_if: skip when *skip_if != 0.
constexpr int kDFK = 8;   // k chunk of M staged at a time
size_t right_multiply_df_smem(int nu) {
  return (size_t)(nu * kRMRows + kDFK * nu) * sizeof(float4);
}

// Error-free transformations, written with the _rn intrinsics so that the compiler neither
// contracts a product into a following addition nor reorders the sums.
__device__ __forceinline__ void two_sum(float& s, float b, float& err) {
  const float t = __fadd_rn(s, b);
  const float bb = __fsub_rn(t, s);
  err = __fadd_rn(err, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(b, bb)));
  s = t;
}
// s + lo += x y with the product's rounding error recovered exactly
__device__ __forceinline__ void df_mac(float& s, float& lo, float x, float y) {
  const float p = __fmul_rn(x, y);
  lo = __fadd_rn(lo, __fmaf_rn(x, y, -p));
  two_sum(s, p, lo);
}

// Y = M - I split once into FP32 (re hi, im hi, re lo, im lo) for every block of the
// multiply (the conversions run on the FP64 pipe).
__global__ void split_near_factor_kernel(const double2* __restrict__ M, int nu,
                                         float4* __restrict__ Ms, const int* gate,
                                         const int* skip_if) {
  if ((gate && *gate == 0) || (skip_if && *skip_if != 0)) return;
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nu * nu) return;
  double2 b = M[t];
  if (t % nu == t / nu) b.x -= 1.0;   // exact: the diagonal is near 1
  const float br = (float)b.x, bi = (float)b.y;
  Ms[t] = make_float4(br, bi, (float)(b.x - br), (float)(b.y - bi));
}

template <int kOut>
__device__ __forceinline__ void multiply_df_rows(float4* df_smem, double2* V, int64_t ldv, int64_t n,
                                                 int nu, const float4* __restrict__ Ms) {
  float4* sV = df_smem;                 // [nu][kRMRows]: (re hi, im hi, re lo, im lo)
  float4* sM = sV + nu * kRMRows;       // [kDFK][nu]
  const int tid = threadIdx.x;
  const int64_t r0 = (int64_t)blockIdx.x * kRMRows;
  for (int t = tid; t < kRMRows * nu; t += blockDim.x) {
    const int rr = t % kRMRows, c = t / kRMRows;
    const int64_t r = r0 + rr;
    const double2 v = (r < n) ? V[(int64_t)c * ldv + r] : make_double2(0.0, 0.0);
    const float hr = (float)v.x, hi = (float)v.y;
    sV[c * kRMRows + rr] = make_float4(hr, hi, (float)(v.x - hr), (float)(v.y - hi));
  }
  const int outs = kRMRows * nu;
  float sr[kOut], srl[kOut], si[kOut], sil[kOut];
#pragma unroll
  for (int m = 0; m < kOut; ++m) sr[m] = srl[m] = si[m] = sil[m] = 0.f;
  for (int k0 = 0; k0 < nu; k0 += kDFK) {
    const int kn = min(kDFK, nu - k0);
    __syncthreads();
    for (int t = tid; t < kDFK * nu; t += blockDim.x) {
      const int kk = t / nu, c = t % nu;
      sM[kk * nu + c] = kk < kn ? Ms[(int64_t)c * nu + k0 + kk] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kOut; ++m) {
      const int o = tid + 256 * m;
      if (o >= outs) break;
      const int c = o % nu, rr = o / nu;
      const int kend = min(kn, c - k0 + 1);   // M[k][c] = 0 for k > c
      for (int kk = 0; kk < kend; ++kk) {
        const float4 a = sV[(k0 + kk) * kRMRows + rr];
        const float4 b = sM[kk * nu + c];
        // real part: a.re b.re - a.im b.im, then the hi x lo cross terms
        df_mac(sr[m], srl[m], a.x, b.x);
        df_mac(sr[m], srl[m], -a.y, b.y);
        srl[m] = __fmaf_rn(a.x, b.z, srl[m]);
        srl[m] = __fmaf_rn(a.z, b.x, srl[m]);
        srl[m] = __fmaf_rn(-a.y, b.w, srl[m]);
        srl[m] = __fmaf_rn(-a.w, b.y, srl[m]);
        // imaginary part: a.re b.im + a.im b.re
        df_mac(si[m], sil[m], a.x, b.y);
        df_mac(si[m], sil[m], a.y, b.x);
        sil[m] = __fmaf_rn(a.x, b.w, sil[m]);
        sil[m] = __fmaf_rn(a.z, b.y, sil[m]);
        sil[m] = __fmaf_rn(a.y, b.z, sil[m]);
        sil[m] = __fmaf_rn(a.w, b.x, sil[m]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < kOut; ++m) {
    const int o = tid + 256 * m;
    if (o >= outs) break;
    const int c = o % nu, rr = o / nu;
    const int64_t r = r0 + rr;
    if (r >= n) continue;
    // V + V Y: the block's own rows, still unchanged in global memory
    const double2 v = V[(int64_t)c * ldv + r];
    V[(int64_t)c * ldv + r] = make_double2(v.x + ((double)sr[m] + (double)srl[m]),
                                           v.y + ((double)si[m] + (double)sil[m]));
  }
}

__global__ void __launch_bounds__(256)
right_multiply_near_df_kernel(double2* V, int64_t ldv, int64_t n, int nu,
                              const float4* __restrict__ Ms, const int* gate, const int* skip_if) {
  if ((gate && *gate == 0) || (skip_if && *skip_if != 0)) return;
  extern __shared__ float4 df_smem[];
  multiply_df_rows<kMaxNu * kRMRows / 256>(df_smem, V, ldv, n, nu, Ms);
}

// ---- nu <= kSmallNu: one launch a factor ----
//
// The steps between a Gram matrix and its multiplication are short and dependent; as kernels of
// their own (sum, products, norm, Cholesky, inverse, second step, split) each costs a launch,
// most of them only to find that it is not needed: ~25 launches of 2-4 us against 10 us of work
// at 320 x 16. Here one cluster of eight blocks does them all, with cluster barriers between
// the steps that exchange data (through global memory; a block reads what others wrote with
// ld.cg) and plain branches where the flags were. A CholeskyQR2 takes 9 launches instead of 36:
// 150 -> 62 us at 320 x 16,
// 170 -> 94 us at 1452 x 30.
constexpr int kSmallNu = 64;
constexpr int kFactorBlocks = 8, kFactorThreads = 1024;
enum { kFactor32 = 0, kFactorNear = 1, kFactorClassic = 2 };

struct FactorArgs {
  const double2* part;   // partial Gram matrices
  int parts, nu;
  double2 *G, *Y, *Z;
  float4* Ms;            // Z - I split for the double-FP32 multiply
  int* flag;             // kFactor32: 1 = too ill-conditioned for FP32; kFactorNear: 1 = near route
  int* status;
  int* deficient;        // kFactorClassic: see cholesky_kernel
  const int* gate;
};

size_t factor_smem(int mode, int nu) {
  return mode == kFactorNear ? (size_t)(2 * nu * (nu + 1) + kFactorBlocks * (nu + 1)) * sizeof(double2) : 0;
}

// Z = R^{-1} of G = R^H R in FP64 by the elimination of chol_inv32_kernel, with the pivot rule
// of cholesky_kernel. entry(r, c): G(r, c), r <= c. Whole block; false on a failed pivot.
template <int kT, typename Entry>
__device__ bool eliminate64(const Entry& entry, int nu, double2* __restrict__ Z, int* deficient) {
  __shared__ double2 col[2][32 * kT], scaled[32 * kT];
  __shared__ double diag[32 * kT];
  __shared__ long long bound;
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32;
  const int tr = lane % 8 + 8 * (w % 4), tc = lane / 8 + 4 * (w / 4);
  double2 g[kT][kT];
#pragma unroll
  for (int i = 0; i < kT; ++i)
#pragma unroll
    for (int j = 0; j < kT; ++j) {
      const int r = tr + 32 * i, c = tc + 32 * j;
      g[i][j] = make_double2(0.0, 0.0);
      if (r >= c && r < nu) {
        const double2 v = entry(c, r);
        g[i][j] = make_double2(v.x, -v.y);
        if (r == c) diag[r] = v.x;
      }
    }
  if (tc == 0)
#pragma unroll
    for (int i = 0; i < kT; ++i) col[0][tr + 32 * i] = g[i][0];
  __syncthreads();
  // the pivots' bound, compared as integers (positive numbers order alike): operations of every
  // thread on the FP64 pipe are what this loop cannot afford
  if (tid < 32) {
    double dmax = 0.0;
    for (int k = tid; k < nu; k += 32) dmax = fmax(dmax, diag[k]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) dmax = fmax(dmax, __shfl_xor_sync(0xffffffffu, dmax, off));
    if (tid == 0) bound = __double_as_longlong(1e-13 * dmax);
  }
  __syncthreads();
  bool ok = true;
  for (int k = 0; k < nu; ++k) {
    const double2* s = col[k & 1];
    double d = s[k].x;
    const bool bad = __double_as_longlong(d) <= bound || (__double2hiint(d) >> 20) == 2047;
    if (bad && !deficient) {
      ok = false;
      break;
    }
    if (tid == 0 && deficient) deficient[k] = bad ? 1 : 0;
    if (bad) d = 1.0;   // unit pivot, no update
    if (tid == 0) diag[k] = d;
    // column k over the pivot, by as many threads as it has entries (by every thread the division
    // alone kept the pipe busy for 5000 clocks)
    if (tid < 32 * kT) {
      const double rd = 1.0 / d;
      const double2 l = s[tid];
      scaled[tid] = tid > k && !bad ? make_double2(l.x * rd, l.y * rd) : make_double2(0.0, 0.0);
    }
    __syncthreads();
    double2 a[kT];
#pragma unroll
    for (int i = 0; i < kT; ++i) a[i] = tr + 32 * i == k ? make_double2(1.0, 0.0) : s[tr + 32 * i];
#pragma unroll
    for (int j = 0; j < kT; ++j) {
      if (32 * j + 31 <= k) continue;
      const int c = tc + 32 * j;
      const double2 l = scaled[c];
#pragma unroll
      for (int i = 0; i < kT; ++i) {
        if (i < j && 32 * i > k) continue;
        const int r = tr + 32 * i;
        const double ly = r >= c ? -l.y : l.y;
        if (c > k && !bad && (r >= c || r <= k)) {
          g[i][j].x -= a[i].x * l.x - a[i].y * ly;
          g[i][j].y -= a[i].x * ly + a[i].y * l.x;
        }
      }
      if (c == k + 1)
#pragma unroll
        for (int i = 0; i < kT; ++i) col[(k + 1) & 1][tr + 32 * i] = g[i][j];
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < kT; ++j) {
    const int c = tc + 32 * j;
    if (c >= nu) continue;
    const double inv = ok ? 1.0 / sqrt(diag[c]) : NAN;
#pragma unroll
    for (int i = 0; i < kT; ++i) {
      const int r = tr + 32 * i;
      if (r >= nu) continue;
      Z[(int64_t)c * nu + r] = r > c ? make_double2(0.0, 0.0)
                               : r == c ? make_double2(inv, 0.0)
                                        : make_double2(g[i][j].x * inv, -g[i][j].y * inv);
    }
  }
  return ok;
}

// Second-order terms Y0^H Y0 + Y0^2 (+ its conjugate on the diagonal) at (i, j), i <= j.
template <typename T2, typename Y0>
__device__ __forceinline__ T2 second_order_at(const Y0& y0, int i, int j) {
  T2 h;
  h.x = h.y = 0;
  for (int m = 0; m <= i; ++m) {
    const T2 a = y0(m, i), b = y0(m, j);
    h.x += a.x * b.x + a.y * b.y;
    h.y += a.x * b.y - a.y * b.x;
  }
  for (int m = i; m <= j; ++m) {
    const T2 a = y0(i, m), b = y0(m, j);
    h.x += a.x * b.x - a.y * b.y;
    h.y += a.x * b.y + a.y * b.x;
    if (i == j) h.x += a.x * b.x - a.y * b.y;
  }
  return h;
}

template <int kMode, int kT>
__global__ void __cluster_dims__(kFactorBlocks, 1, 1) __launch_bounds__(kFactorThreads)
cq_factor_kernel(FactorArgs p) {
  if (p.gate && *p.gate == 0) return;
  extern __shared__ double2 factor_mem[];
  __shared__ double2 red[32][32];
  __shared__ float redf[32];
  const int tid = threadIdx.x, lane = tid % 32, w = tid / 32, nu = p.nu;
  const int rank = (int)sm100::cluster_ctarank();
  // G = sum of the partials: a warp adds every eighth part of 32 elements
  for (int t0 = rank * 128; t0 < nu * nu; t0 += kFactorBlocks * 128) {
    const int q = w % 8, t = t0 + (w / 8) * 32 + lane;
    const bool live = t < nu * nu && t % nu / kGT <= t / nu / kGT;
    double2 sum = make_double2(0.0, 0.0);
    if (live)
#pragma unroll 8
      for (int r = q; r < p.parts; r += 8) {
        const double2 v = p.part[(int64_t)r * nu * nu + t];
        sum.x += v.x;
        sum.y += v.y;
      }
    red[w][lane] = sum;
    __syncthreads();
    if (live && q == 0) {
#pragma unroll
      for (int k = 1; k < 8; ++k) {
        sum.x += red[w + k][lane].x;
        sum.y += red[w + k][lane].y;
      }
      p.G[t] = sum;
    }
    __syncthreads();
  }
  sm100::cluster_sync_all();
  if (kMode == kFactor32) {
    if (rank != 0 || tid >= 256) return;
    if (tid == 0) *p.flag = 0;   // (chol_inv32_block: same thread)
    if (nu <= 16)
      chol_inv32_block<16, 1>(p.G, nu, nu, p.G, nu, p.Z, nu, p.flag);
    else
      chol_inv32_block<16, 2 * kT>(p.G, nu, nu, p.G, nu, p.Z, nu, p.flag);
    return;
  }
  if (kMode == kFactorClassic) {
    if (rank == 0) {
      const bool ok = eliminate64<kT>([&](int r, int c) { return __ldcg(p.G + (int64_t)c * nu + r); },
                                      nu, p.Z, p.deficient);
      if (!ok && tid == 0) atomicOr(p.status, kStatusNotSPD);
    }
    return;
  }
  const int ld = nu + 1;   // (odd in 16-byte words: columns over all banks)
  double2* sG = factor_mem;            // [c][r], r <= c
  double2* sY = sG + nu * ld;
  double2* sP = sY + nu * ld;          // this block's columns of E + Y + E Y
  float2* yf = reinterpret_cast<float2*>(sY);
  float e2 = 0.f;
  for (int t = tid; t < nu * nu; t += kFactorThreads) {
    const int r = t % nu, c = t / nu;
    if (r > c) continue;
    const double2 g = __ldcg(p.G + t);
    sG[c * ld + r] = g;
    const float ex = (float)(r == c ? g.x - 1.0 : g.x), ey = r == c ? 0.f : (float)g.y;
    e2 += (ex * ex + ey * ey) * (r == c ? 1.f : 2.f);
    yf[c * ld + r] = r == c ? make_float2(-0.5f * ex, 0.f) : make_float2(-ex, -ey);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, off);
  if (lane == 0) redf[w] = e2;
  __syncthreads();
  e2 = redf[lane];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, off);
  const bool near = e2 <= kNearEps * kNearEps, small = e2 <= kNearEpsSmall * kNearEpsSmall;
  if (rank == 0 && tid == 0) *p.flag = near ? 1 : 0;
  if (!near) {
    if (rank == 0) {
      const bool ok = eliminate64<kT>([&](int r, int c) { return sG[c * ld + r]; }, nu, p.Z, nullptr);
      if (!ok && tid == 0) atomicOr(p.status, kStatusNotSPD);
    }
    return;
  }
  auto finish = [&](int i, int j, double2 y) {   // Z = I + Y at (i, j), and its split
    const int t = j * nu + i;
    const double2 z = i > j ? make_double2(0.0, 0.0) : i == j ? make_double2(1.0 + y.x, 0.0) : y;
    const double br = i == j ? z.x - 1.0 : z.x;
    p.Z[t] = z;
    const float fr = (float)br, fi = (float)z.y;
    p.Ms[t] = make_float4(fr, fi, (float)(br - fr), (float)(z.y - fi));
  };
  auto y1_of = [&](int i, int j, double2 e, double2 h) {
    return i < j ? make_double2(h.x - e.x, h.y - e.y) : make_double2(-0.5 * (e.x - h.x), 0.0);
  };
  if (small) {   // as near_y1_kernel: FP32 second-order terms
    // this thread's output: rows rank, rank + 8, ... of the block, a column each
    const int i = rank + kFactorBlocks * (tid / kSmallNu), j = tid % kSmallNu;
    if (i >= nu || j >= nu) return;
    double2 y = make_double2(0.0, 0.0);
    if (i <= j) {
      const double2 g = sG[j * ld + i];
      const float2 h = second_order_at<float2>([&](int r, int c) { return yf[c * ld + r]; }, i, j);
      y = y1_of(i, j, i == j ? make_double2(g.x - 1.0, 0.0) : g, make_double2(h.x, h.y));
    }
    finish(i, j, y);
    return;
  }
  // Both steps in FP64. The second-order terms of the first are Y0^H Y0 + Y0^2 = -E Y0 in the upper
  // triangle (E = -(Y0 + Y0^H)), and once more y0_ii^2 on the diagonal; the second step is
  // -U(E + W + Y^H (E + Y + W)), W = E Y, of which its upper triangle needs W's alone. So a block
  // takes columns rank, rank + 8, ..., a row a thread, and only Y1 goes round the cluster. FP64-bound:
  // 3.3 nu^3 multiply-adds (P = Y^H E and Q = Y^H Y in full, by rows, took 6.7 and as many operations
  // again to form Y0 and E: 222 us at nu = 64; now 137).
  for (int c = tid; c < nu; c += kFactorThreads) sG[c * ld + c] = make_double2(sG[c * ld + c].x - 1.0, 0.0);
  __syncthreads();   // sG holds E's upper triangle
  const int i = tid % kSmallNu, own = tid / kSmallNu, j = rank + kFactorBlocks * own;
  const bool upper = i <= j && j < nu;
  auto e_at = [&](int r, int c) {
    const double2 g = r > c ? sG[r * ld + c] : sG[c * ld + r];
    return make_double2(g.x, r > c ? -g.y : g.y);
  };
  auto mac = [](double2& s, double2 a, double2 b) {
    s.x += a.x * b.x - a.y * b.y;
    s.y += a.x * b.y + a.y * b.x;
  };
  const double2 eij = upper ? e_at(i, j) : make_double2(0.0, 0.0);
  if (upper) {
    const double2* ej = sG + j * ld;
    double2 h = make_double2(0.0, 0.0);
    for (int m = 0; m < j; ++m) mac(h, e_at(i, m), ej[m]);
    mac(h, eij, make_double2(0.5 * ej[j].x, 0.0));
    if (i == j) h.x += 0.25 * eij.x * eij.x;
    p.Y[j * nu + i] = y1_of(i, j, eij, h);
  }
  sm100::cluster_sync_all();
  for (int t = tid; t < nu * nu; t += kFactorThreads) {
    const int r = t % nu, c = t / nu;
    if (r <= c) sY[c * ld + r] = __ldcg(p.Y + t);
  }
  __syncthreads();
  double2 x = make_double2(0.0, 0.0);
  if (upper) {
    const double2* yj = sY + j * ld;
    for (int m = 0; m <= j; ++m) mac(x, e_at(i, m), yj[m]);
    x.x += eij.x;
    x.y += eij.y;
    sP[own * ld + i] = make_double2(x.x + yj[i].x, x.y + yj[i].y);
  }
  __syncthreads();
  if (i >= nu || j >= nu) return;
  double2 y = make_double2(0.0, 0.0);
  if (upper) {
    const double2 *yi = sY + i * ld, *pj = sP + own * ld;
    for (int m = 0; m <= i; ++m) mac(x, make_double2(yi[m].x, -yi[m].y), pj[m]);
    y = i < j ? make_double2(-x.x, -x.y) : make_double2(-0.5 * x.x, 0.0);
  }
  finish(i, j, y);
}

// V <- V Z for nu <= kSmallNu: the near-identity product where *near says so, else in FP64.
__global__ void __launch_bounds__(256)
multiply_small_kernel(double2* V, int64_t ldv, int64_t n, int nu, const double2* __restrict__ Z,
                      const float4* __restrict__ Ms, const int* gate, const int* skip_if,
                      const int* near) {
  if ((gate && *gate == 0) || (skip_if && *skip_if != 0)) return;
  extern __shared__ double rm_smem[];
  constexpr int kOut = kSmallNu * kRMRows / 256;
  if (near && *near != 0)
    multiply_df_rows<kOut>(reinterpret_cast<float4*>(rm_smem), V, ldv, n, nu, Ms);
  else
    multiply64_rows<kOut>(rm_smem, V, ldv, n, nu, Z);
}

// C = A * B for upper-triangular nu x nu A, B (one block).
__global__ void upper_product_kernel(const double2* A, const double2* B, int nu, double2* C) {
  for (int64_t t = threadIdx.x; t < (int64_t)nu * nu; t += blockDim.x) {
    const int i = (int)(t % nu), jj = (int)(t / nu);
    double2 acc = make_double2(0.0, 0.0);
    for (int k = i; k <= jj; ++k) {
      const double2 a = A[(int64_t)k * nu + i];
      const double2 b = B[(int64_t)jj * nu + k];
      acc.x += a.x * b.x - a.y * b.y;
      acc.y += a.x * b.y + a.y * b.x;
    }
    C[t] = acc;
  }
}

}  // namespace

namespace {

struct CqLayout {
  int tiles_u = 0;           // upper Gram tiles
  int64_t parts = 0, rows_per_part = 0;
  int64_t parts32 = 0, rows32 = 0;   // of the FP32 Gram matrix
  int64_t parts_max = 0;     // with those of the split products
  unsigned sum_blocks = 0;   // blocks of sum_parts_kernel (eight threads per element)
};

CqLayout cq_layout(bem_ctx* ctx, int64_t n, int nu) {
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  CqLayout L;
  const int T = (nu + kGT - 1) / kGT;
  L.tiles_u = T * (T + 1) / 2;
  // no fewer than 4 rows a part: a 32 x 32 tile of a row is 0.8 us of an SM's FP64 pipe, so a short
  // V is spread thin (320 x 16: 27 us at 32 rows a part, 5.6 us at 4); at most one block an SM where
  // a single cluster adds the parts (one block more, 51 parts of 3 tiles, doubles the time of the
  // slowest SM: 3000 x 33 with R 690 us, now 591)
  const int64_t blocks = (nu <= kSmallNu ? 1 : 2) * (int64_t)std::max(1, sms);
  L.parts = nu <= kSmallNu ? blocks / L.tiles_u : (blocks + L.tiles_u - 1) / L.tiles_u;
  // room for the parts of any n: the workspace a call finds does not grow (and move) with n, so that
  // what a captured call holds is there after calls on longer bases
  L.parts_max = std::max<int64_t>(std::max<int64_t>(1, L.parts), split64_parts(ctx, INT64_MAX / 2, nu));
  L.parts = std::max<int64_t>(1, std::min<int64_t>((n + 3) / 4, L.parts));
  L.rows_per_part = (n + L.parts - 1) / L.parts;
  L.parts = (n + L.rows_per_part - 1) / L.rows_per_part;
  L.rows32 = std::max<int64_t>(L.rows_per_part, kGT);
  L.parts32 = (n + L.rows32 - 1) / L.rows32;
  L.sum_blocks = (unsigned)((8 * (int64_t)nu * nu + 255) / 256);
  return L;
}

// Work space: nine nu x nu complex matrices (G, Z, R1, R2, P, Q, Y, P1, Q1), the Gram
// partials, then 256 deficiency flags, 8 pass flags and the |E|^2 block sums.
struct CqWork {
  double2 *G, *Z, *R1, *R2, *P, *Q, *Y, *P1, *Q1, *part;
  int* deficient;
  int* flags;
  float* epsp;
};

CqWork cq_work(void* work, int nu, const CqLayout& L) {
  CqWork w;
  double2* p = reinterpret_cast<double2*>(work);
  const size_t m = (size_t)nu * nu;
  w.G = p; w.Z = p + m; w.R1 = p + 2 * m; w.R2 = p + 3 * m; w.P = p + 4 * m; w.Q = p + 5 * m;
  w.Y = p + 6 * m; w.P1 = p + 7 * m; w.Q1 = p + 8 * m; w.part = p + 9 * m;
  w.deficient = reinterpret_cast<int*>(w.part + (size_t)L.parts_max * m);
  w.flags = w.deficient + 256;
  w.epsp = reinterpret_cast<float*>(w.flags + 8);
  return w;
}

bem_status set_smem(bem_ctx* ctx, const void* fn, size_t bytes) {
  if (bytes <= 48 * 1024) return BEM_OK;
  return cuda_check(ctx, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)bytes),
                    "cholqr attribute");
}

// Partial sums of the FP64 Gram matrix into w.part (their count in parts): on the tensor core
// where the plan says so (split64.cu), else on the FP64 pipe.
bem_status gram_parts64(bem_ctx* ctx, const Split64& sp, const double2* V, int64_t ldv, int64_t n,
                        int nu, const CqLayout& L, const CqWork& w, const int* gate, int& parts,
                        cudaStream_t s) {
  parts = sp.use ? sp.parts : (int)L.parts;
  if (sp.use) return split64_gram(ctx, sp, V, w.part, gate, s);
  gram_partial_kernel<<<dim3((unsigned)L.tiles_u, (unsigned)L.parts), 256, 0, s>>>(
      V, ldv, n, nu, L.rows_per_part, w.part, gate);
  ctx->launches++;
  return BEM_OK;
}

// V <- V Z in FP64 (skipped when gate and *gate == 0, or skip and *skip != 0). same: V is the one
// whose Gram matrix was formed last (the split products then have its scales).
bem_status multiply64(bem_ctx* ctx, const Split64& sp, bool same, double2* V, int64_t ldv,
                      int64_t n, int nu, const double2* Z, const int* gate, const int* skip,
                      cudaStream_t s) {
  if (sp.use) return split64_multiply(ctx, sp, same, V, Z, gate, skip, s);
  const unsigned rb = (unsigned)((n + kRMRows - 1) / kRMRows);
  if (nu <= kSmallNu)
    multiply_small_kernel<<<rb, 256, right_multiply_smem(nu), s>>>(V, ldv, n, nu, Z, nullptr, gate,
                                                                   skip, nullptr);
  else
    right_multiply_kernel<<<rb, 256, right_multiply_smem(nu), s>>>(V, ldv, n, nu, Z, gate, skip, nullptr);
  ctx->launches++;
  return BEM_OK;
}

// The factor of a Gram matrix in w.part for nu <= kSmallNu (cq_factor_kernel).
template <int kMode>
bem_status small_factor(bem_ctx* ctx, const CqWork& w, int parts, int nu, int* flag, int* deficient,
                        const int* gate, cudaStream_t s) {
  const FactorArgs a{w.part, parts, nu, w.G, w.Y, w.Z, reinterpret_cast<float4*>(w.Q1),
                     flag, ctx->d_status, deficient, gate};
  auto* kernel = nu <= 32 ? cq_factor_kernel<kMode, 1> : cq_factor_kernel<kMode, 2>;
  if (factor_smem(kMode, nu) > 0) {   // (beside ~19 KB of its static arrays)
    const bem_status st = cuda_check(
        ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)factor_smem(kMode, nu)),
        "cholqr attribute");
    if (st != BEM_OK) return st;
  }
  kernel<<<kFactorBlocks, kFactorThreads, factor_smem(kMode, nu), s>>>(a);
  ctx->launches++;
  return BEM_OK;
}

// Z = R^{-1} of w.G in FP32 for nu > kSmallNu, in one or two diagonal blocks; *fallback is set
// where a pivot is too small. Skipped when gate is given and *gate == 0, or *fallback != 0 (the
// rest is, once it is set).
void factor32(bem_ctx* ctx, const CqWork& w, int nu, int* fallback, const int* gate, cudaStream_t s) {
  const int h = std::min(nu, kChol32), r = nu - h;   // diagonal blocks
  auto inverse32 = [&](const double2* G, int ldg, int m, double2* Z) {
    auto* kernel = m <= 32 ? chol_inv32_kernel<1> : m <= 64 ? chol_inv32_kernel<2> : chol_inv32_kernel<4>;
    kernel<<<1, 1024, 0, s>>>(G, ldg, m, w.G, nu, Z, nu, fallback, gate);
    ctx->launches++;
  };
  inverse32(w.G, nu, h, w.Z);
  if (r == 0) return;
  const dim3 gh((unsigned)((h + 15) / 16), (unsigned)((r + 15) / 16)), gr(gh.y, gh.y);
  chol_block32_kernel<0><<<gh, 256, 0, s>>>(w.G, w.Z, nu, w.P, w.Q, w.Y, fallback, gate);
  chol_block32_kernel<1><<<gr, 256, 0, s>>>(w.G, w.Z, nu, w.P, w.Q, w.Y, fallback, gate);
  inverse32(w.Q, r, r, w.Z + (size_t)h * nu + h);
  chol_block32_kernel<2><<<gh, 256, 0, s>>>(w.G, w.Z, nu, w.P, w.Q, w.Y, fallback, gate);
  chol_block32_kernel<3><<<gh, 256, 0, s>>>(w.G, w.Z, nu, w.P, w.Q, w.Y, fallback, gate);
  ctx->launches += 4;
}

// One FP64 pass V <- V R^{-1} whose Gram matrix is expected near the identity: the
// near-identity factor, or the classic Cholesky factorisation and triangular inverse when
// ||G - I||_F > kNearEps (flag *classic, set on the device; three ints). Everything is skipped
// unless *gate != 0 (gate null: always runs). refused, if given: where *refused == 0 and another
// near pass follows this one, the factor is an FP32 one again (nu > kSmallNu; FP64 if it fails).
bem_status near_pass(bem_ctx* ctx, double* V_dev, int64_t ldv, int64_t n, int nu,
                     const CqLayout& L, const CqWork& w, const Split64& sp, const int* gate,
                     int* classic, const int* refused, cudaStream_t s) {
  double2* V = reinterpret_cast<double2*>(V_dev);
  const unsigned rb = (unsigned)((n + kRMRows - 1) / kRMRows);
  int parts;
  bem_status st = gram_parts64(ctx, sp, V, ldv, n, nu, L, w, gate, parts, s);
  if (st != BEM_OK) return st;
  float4* Zs = reinterpret_cast<float4*>(w.Q1);   // Z - I split (Q1 is free by then)
  if (nu <= kSmallNu) {
    int* near = classic;
    if ((st = small_factor<kFactorNear>(ctx, w, parts, nu, near, nullptr, gate, s)) != BEM_OK) return st;
    if (sp.use) return split64_multiply(ctx, sp, true, V, w.Z, gate, nullptr, s);
    multiply_small_kernel<<<rb, 256, right_multiply_smem(nu), s>>>(V, ldv, n, nu, w.Z, Zs, gate,
                                                                   nullptr, near);
    ctx->launches++;
    return cuda_check(ctx, cudaGetLastError(), "cholqr kernels");
  }
  int* done = classic + 2;   // classic flag and its "second step not needed" companion
  st = cuda_check(ctx, cudaMemsetAsync(classic, 0, 3 * sizeof(int), s), "cholqr flag");
  if (st != BEM_OK) return st;
  sum_parts_kernel<<<L.sum_blocks, 256, 0, s>>>(w.part, parts, nu, w.G, w.epsp, gate);
  const unsigned nt = (unsigned)((nu + kNT - 1) / kNT);
  const dim3 tgrid(nt, nt);
  near_y1_kernel<<<tgrid, 64, 0, s>>>(w.G, w.epsp, (int)L.sum_blocks, nu, kNearEps, kNearEpsSmall,
                                      w.Y, w.Z, classic, done, refused, gate);
  if (refused) factor32(ctx, w, nu, classic + 1, classic, s);
  cholesky_kernel<<<1, 1024, 0, s>>>(w.G, nu, ctx->d_status, nullptr, classic + 1);
  triangular_inverse_kernel<<<nu, 128, 0, s>>>(w.G, nu, w.Z, classic + 1);
  near_tile_kernel<1><<<tgrid, 64, 0, s>>>(w.G, w.Y, nullptr, nullptr, nu, w.P1, w.Q1, nullptr,
                                           gate, done);
  near_tile_kernel<2><<<tgrid, 64, 0, s>>>(w.G, w.Y, w.P1, w.Q1, nu, nullptr, nullptr, w.Z,
                                           gate, done);
  ctx->launches += 6;
  // V <- V Z: on the tensor core; else the classic inverse in FP64, the near-identity factor as
  // V + V (Z - I)
  if (sp.use) return split64_multiply(ctx, sp, true, V, w.Z, gate, nullptr, s);
  right_multiply_kernel<<<rb, 256, right_multiply_smem(nu), s>>>(V, ldv, n, nu, w.Z, gate,
                                                                 nullptr, classic);
  split_near_factor_kernel<<<(unsigned)((nu * nu + 255) / 256), 256, 0, s>>>(w.Z, nu, Zs, gate,
                                                                            classic);
  right_multiply_near_df_kernel<<<rb, 256, right_multiply_df_smem(nu), s>>>(V, ldv, n, nu, Zs,
                                                                            gate, classic);
  ctx->launches += 3;
  return cuda_check(ctx, cudaGetLastError(), "cholqr kernels");
}

// Classic FP64 pass: Gram, Cholesky (optionally refreshing collapsed columns), inverse,
// V <- V R^{-1}; R kept in R_out if it is given.
bem_status classic_pass(bem_ctx* ctx, double* V_dev, int64_t ldv, int64_t n, int nu,
                        const CqLayout& L, const CqWork& w, const Split64& sp, double2* R_out,
                        uint64_t refresh_seed, cudaStream_t s) {
  double2* V = reinterpret_cast<double2*>(V_dev);
  int parts;
  bem_status st = gram_parts64(ctx, sp, V, ldv, n, nu, L, w, nullptr, parts, s);
  if (st != BEM_OK) return st;
  int* deficient = refresh_seed ? w.deficient : nullptr;
  if (!R_out && nu <= kSmallNu) {
    if ((st = small_factor<kFactorClassic>(ctx, w, parts, nu, nullptr, deficient, nullptr, s)) != BEM_OK)
      return st;
  } else {
    double2* R = R_out ? R_out : w.R1;
    sum_parts_kernel<<<L.sum_blocks, 256, 0, s>>>(w.part, parts, nu, R, nullptr, nullptr);
    const size_t chol_smem = nu <= 64 ? (size_t)nu * nu * sizeof(double2) : 0;
    cholesky_kernel<<<1, 1024, chol_smem, s>>>(R, nu, ctx->d_status, deficient, nullptr);
    triangular_inverse_kernel<<<nu, 128, 0, s>>>(R, nu, w.Z, nullptr);
    ctx->launches += 3;
  }
  if ((st = multiply64(ctx, sp, true, V, ldv, n, nu, w.Z, nullptr, nullptr, s)) != BEM_OK) return st;
  if (refresh_seed) {
    refresh_columns_kernel<<<(unsigned)((n * nu + 255) / 256), 256, 0, s>>>(V, ldv, n, nu,
                                                                           w.deficient,
                                                                           refresh_seed);
    ctx->launches++;
  }
  return cuda_check(ctx, cudaGetLastError(), "cholqr kernels");
}

}  // namespace

size_t cholqr2_work_bytes(bem_ctx* ctx, int64_t n, int nu) {
  const CqLayout L = cq_layout(ctx, n, nu);
  return (9 + (size_t)L.parts_max) * (size_t)nu * nu * sizeof(double2) +
         (256 + 8) * sizeof(int) + (size_t)L.sum_blocks * sizeof(float);
}

// CholeskyQR2 of V (n x nu, ld ldv) with caller-provided work (cholqr2_work_bytes);
// asynchronous; a Gram matrix that is not positive definite is flagged in the context's
// status word.
//
// Without R (and no refresh): the first pass runs in FP32: it only has to make V well
// conditioned. The FP64 second pass then sees G = I + E with small E and uses the
// near-identity factor. If V is too ill-conditioned for FP32 the first pass leaves V alone
// (device flag) and a third pass runs (its kernels return at once otherwise); the second
// pass then falls back to the classic factorisation by itself. With R: two classic passes
// and R = R2 R1.
// nu > kChol32: a basis of condition ~30 .. 1000 passes FP32 but is left too far from orthonormal for
// the near-identity factor. A classic second pass is then neither as orthogonal as two FP64 passes
// (400 x 200, condition 100: 2.9e-15 against 1.1e-15) nor fast; the second pass takes another FP32
// factor instead and the third one finishes. Columns of up to kChol32 keep the classic second pass.
bem_status cholqr2_impl(bem_ctx* ctx, double* V_dev, int64_t n, int64_t ldv, int nu,
                        double* R_dev, void* work, cudaStream_t s, uint64_t refresh_seed) {
  const CqLayout L = cq_layout(ctx, n, nu);
  const CqWork w = cq_work(work, nu, L);
  bem_status st = BEM_OK;
  const size_t chol_smem = nu <= 64 ? (size_t)nu * nu * sizeof(double2) : 0;
  if ((st = set_smem(ctx, (const void*)cholesky_kernel, chol_smem)) != BEM_OK) return st;
  if ((st = set_smem(ctx, (const void*)right_multiply_kernel, right_multiply_smem(nu))) != BEM_OK)
    return st;
  if ((st = set_smem(ctx, (const void*)right_multiply_near_df_kernel,
                     right_multiply_df_smem(nu))) != BEM_OK)
    return st;
  // the split products' planes, given up if they cannot be had: apart from the factors' workspace,
  // whose size does not depend on n
  Split64 sp;
  const size_t split = split64_bytes(ctx, n, nu);
  ExpandUse planes(ctx, s);
  if (split > 0 && planes.get(split)) split64_plan(ctx, ldv, n, nu, planes.work, sp);
  if (R_dev) {
    if ((st = classic_pass(ctx, V_dev, ldv, n, nu, L, w, sp, w.R1, refresh_seed, s)) != BEM_OK) return st;
    if ((st = classic_pass(ctx, V_dev, ldv, n, nu, L, w, sp, w.R2, 0, s)) != BEM_OK) return st;
    upper_product_kernel<<<1, 256, 0, s>>>(w.R2, w.R1, nu, reinterpret_cast<double2*>(R_dev));
    ctx->launches++;
    return cuda_check(ctx, cudaGetLastError(), "cholqr kernels");
  }
  if (refresh_seed != 0) {
    if ((st = classic_pass(ctx, V_dev, ldv, n, nu, L, w, sp, nullptr, refresh_seed, s)) != BEM_OK) return st;
    return near_pass(ctx, V_dev, ldv, n, nu, L, w, sp, nullptr, w.flags + 1, nullptr, s);
  }
  int* fallback = w.flags;
  double2* V = reinterpret_cast<double2*>(V_dev);
  int parts;
  const bool wide = sp.use && nu > kChol32;   // the split Gram matrix, else FP32
  if (wide) {
    if ((st = gram_parts64(ctx, sp, V, ldv, n, nu, L, w, nullptr, parts, s)) != BEM_OK) return st;
  } else {
    parts = (int)L.parts32;
    gram_partial32_kernel<<<dim3((unsigned)L.tiles_u, (unsigned)L.parts32), 256, 0, s>>>(
        V, ldv, n, nu, L.rows32, w.part);
    ctx->launches++;
  }
  if (nu <= kSmallNu) {
    if ((st = small_factor<kFactor32>(ctx, w, parts, nu, fallback, nullptr, nullptr, s)) != BEM_OK) return st;
  } else {
    st = cuda_check(ctx, cudaMemsetAsync(fallback, 0, sizeof(int), s), "cholqr flag");
    if (st != BEM_OK) return st;
    sum_parts_kernel<<<L.sum_blocks, 256, 0, s>>>(w.part, parts, nu, w.G, nullptr, nullptr);
    ctx->launches++;
    factor32(ctx, w, nu, fallback, nullptr, s);
  }
  if ((st = multiply64(ctx, sp, wide, V, ldv, n, nu, w.Z, nullptr, fallback, s)) != BEM_OK) return st;
  if ((st = cuda_check(ctx, cudaGetLastError(), "cholqr kernels")) != BEM_OK) return st;
  const bool again = nu > kChol32;   // the third pass follows every second one that is not near
  st = near_pass(ctx, V_dev, ldv, n, nu, L, w, sp, nullptr, w.flags + 1, again ? fallback : nullptr, s);
  if (st != BEM_OK) return st;
  // the third pass rarely runs: for the smaller bases the form with the fewest launches
  Split64 third = sp;
  if (nu <= kSmallNu && n * (int64_t)nu * nu < ((int64_t)1 << 25)) third.use = false;
  return near_pass(ctx, V_dev, ldv, n, nu, L, w, third, again ? w.flags + 1 : fallback, w.flags + 4, nullptr, s);
}

}  // namespace bem

using namespace bem;

extern "C" bem_status bem_cholqr2(bem_ctx* ctx, double* V_dev, int64_t n, int64_t ldv, int nu,
                                  double* R_dev, void* stream) {
  if (!ctx) return BEM_EINVAL;
  if (!V_dev || n < 1 || nu < 1 || nu > kMaxNu || ldv < n || nu > n)
    return fail(ctx, BEM_EINVAL, "bem_cholqr2: need V, 1 <= nu <= min(n, 256), ldv >= n");
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  bem_status st = ensure_small(ctx, cholqr2_work_bytes(ctx, n, nu));
  if (st != BEM_OK) return st;
  st = cholqr2_impl(ctx, V_dev, n, ldv, nu, R_dev, ctx->d_small, s, 0);
  if (st != BEM_OK) return st;
  if (ctx->async) return cuda_check(ctx, cudaGetLastError(), "bem_cholqr2");
  return take_status(ctx, s, "bem_cholqr2");
}
