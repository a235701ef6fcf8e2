// The eigen-decomposition of small_eig.h by one block (same algorithm, same deflation rule
// and shifts).
//
// Bound by the serial chain of Givens rotations: about 3 m sweeps of up to m rotations, each
// needing the previous one's result in two entries. On one thread every rotation also paid
// for its ~3 m complex row and column updates (m = 32: 80.6 ms); here A and Z sit in shared
// memory (m <= 64) and one warp carries the chain: it applies a rotation to the few entries
// the next one comes from, a lane per real number, and forms the next rotation while the other
// warps apply this one to everything else, so a rotation costs one barrier and one chain step.
// m = 32: 80.6 -> 3.5 ms (a lane per entry: 4.7 ms).
#pragma once

#include "small_eig.h"

namespace bem {
namespace small {

constexpr int kEigSmemMax = 64;   // largest m whose matrices sit in shared memory

// leading dimension: odd, so that threads across columns hit different banks
__host__ __device__ inline int eig_ld(int m) { return m <= kEigSmemMax ? m + 1 - (m & 1) : m; }
__host__ inline size_t eig_smem(int m) {
  return m <= kEigSmemMax ? (size_t)3 * m * eig_ld(m) * sizeof(zc) : 0;
}
// a warp for the chain, the others for the 2 m rows and columns of a rotation
__host__ inline int eig_threads(int m) { return 32 + 2 * (m < 32 ? 32 : (m + 31) / 32 * 32); }

// Givens rotation as small::givens, by reciprocal square roots where the squares are safe.
__device__ inline void givens_fast(zc x, zc y, double& c, zc& s) {
  const double ax2 = abs2(x), ay2 = abs2(y);
  if (!(ax2 > 1e-200 && ax2 < 1e200 && ay2 > 1e-200 && ay2 < 1e200)) {
    givens(x, y, c, s);
    return;
  }
  const double w = rsqrt(ax2) * rsqrt(ax2 + ay2);
  c = ax2 * w;
  s = scl(mul(x, cj(y)), w);
}

// (p, q) <- (c p + s q, c q - conj(s) p)
__device__ __forceinline__ void rotate(zc& p, zc& q, double c, zc s) {
  const zc a = p, b = q;
  p = add(scl(a, c), mul(s, b));
  q = sub(scl(b, c), mul(cj(s), a));
}

// rotate() of the pair p, q by four lanes, each forming a part of it: lane & 2 the q, lane & 1 the
// imaginary part. Returns the lane's part. The pipe takes 16 clocks a warp's operation however many
// lanes take part, so a chain of few numbers is shortened by giving every lane one of them: a
// rotation's 12 operations become 3, and the next one's formation 12 instead of 23.
__device__ __forceinline__ double rotate_lanes(zc* p, zc* q, bool active, double c, zc s) {
  const int lane = threadIdx.x % 32;
  const bool im = lane & 1, second = lane & 2;
  double v = 0.0;
  double* mine = &(second ? q : p)->re + (im ? 1 : 0);
  if (active) {
    const double* other = &(second ? p : q)->re;
    const double o1 = other[im ? 1 : 0], o2 = other[im ? 0 : 1];
    v = fma(im ? s.im : -s.im, o2, fma(second ? -s.re : s.re, o1, c * *mine));
  }
  __syncwarp();
  if (active) *mine = v;
  __syncwarp();
  return v;
}

// givens_fast(x, y) by a warp (x and y in every lane), written by lanes 0 .. 2.
__device__ __forceinline__ void givens_lanes(zc x, zc y, double& c, zc& s) {
  const int lane = threadIdx.x % 32;
  const bool odd = lane & 1;
  const double re = odd ? y.re : x.re, im = odd ? y.im : x.im, a = fma(re, re, im * im);
  const int e = (__double2hiint(a) >> 20) - 1023;   // a within 2^-600 .. 2^600
  if (!__all_sync(0xffffffffu, e > -600 && e < 600)) {
    double cc;
    zc ss;
    givens(x, y, cc, ss);
    if (lane == 0) {
      c = cc;
      s = ss;
    }
    return;
  }
  // even lanes 1 / |x|, odd ones 1 / sqrt(|x|^2 + |y|^2)
  const double sum = a + __shfl_xor_sync(0xffffffffu, a, 1);
  const double r = rsqrt(odd ? sum : a);
  const double w = r * __shfl_xor_sync(0xffffffffu, r, 1);
  // lane 0: c = |x|^2 w, lanes 1, 2: the parts of s = x conj(y) w
  const double u1 = odd ? x.re : x.im, u2 = odd ? x.im : -x.re;
  const double t = fma(u1, y.re, u2 * y.im);
  const double v = (lane == 0 ? a : t) * w;
  if (lane == 0) c = v;
  else if (lane == 1) s.re = v;
  else if (lane == 2) s.im = v;
}

#define SE_A(M, i, j) (M)[(int64_t)(j) * ld + (i)]

// gA (m x m, column-major, destroyed), gw (m), gV (m x m), gZ (m x m work), as small::eig;
// blockDim.x = eig_threads(m), dynamic shared memory eig_smem(m). Every thread returns the
// same status.
__device__ inline int eig_block(int m, zc* gA, zc* gw, zc* gV, zc* gZ) {
  extern __shared__ __align__(16) unsigned char eig_sm[];
  __shared__ double sh_c[2];
  __shared__ zc sh_s[2];
  __shared__ zc sh_v0, sh_alpha, sh_mu;
  __shared__ double sh_beta;
  __shared__ int sh_l, sh_ihi, sh_state;
  const double eps = 2.220446049250313e-16;
  const int tid = threadIdx.x, nt = blockDim.x, half = nt / 2 / 32 * 32;
  const bool first = tid < half;      // Hessenberg step: this thread works on A (else on Z)
  const int t = first ? tid : tid - half;
  const int zt = nt - half;           // threads that work on Z
  const bool in_smem = m <= kEigSmemMax;
  const int ld = eig_ld(m);
  zc* A = in_smem ? reinterpret_cast<zc*>(eig_sm) : gA;
  zc* Z = in_smem ? A + (size_t)m * ld : gZ;
  zc* Y = in_smem ? Z + (size_t)m * ld : gV;
  for (int e = tid; e < m * m; e += nt) {
    const int i = e % m, j = e / m;
    if (in_smem) SE_A(A, i, j) = gA[e];
    SE_A(Z, i, j) = mk(i == j ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();

  // 1. Hessenberg reduction
  for (int k = 0; k + 2 < m; ++k) {
    if (tid == 0) {
      double nrm2 = 0.0;
      for (int i = k + 1; i < m; ++i) nrm2 += abs2(SE_A(A, i, k));
      const double nrm = sqrt(nrm2);
      sh_beta = 0.0;
      if (nrm != 0.0) {
        const zc x0 = SE_A(A, k + 1, k);
        const double ax0 = absz(x0);
        const zc ph = ax0 > 0.0 ? scl(x0, 1.0 / ax0) : mk(1.0, 0.0);
        sh_alpha = scl(ph, -nrm);
        sh_v0 = sub(x0, sh_alpha);
        double vn2 = abs2(sh_v0);
        for (int i = k + 2; i < m; ++i) vn2 += abs2(SE_A(A, i, k));
        if (vn2 != 0.0) sh_beta = 2.0 / vn2;
      }
    }
    __syncthreads();
    const double beta = sh_beta;
    const zc v0 = sh_v0;
    if (beta == 0.0) {
      __syncthreads();
      continue;
    }
    // left: one thread per column; Z from the right at the same time: one thread per row
    if (first) {
      for (int j = k + 1 + t; j < m; j += half) {
        zc s = mul(cj(v0), SE_A(A, k + 1, j));
        for (int i = k + 2; i < m; ++i) s = add(s, mul(cj(SE_A(A, i, k)), SE_A(A, i, j)));
        s = scl(s, beta);
        SE_A(A, k + 1, j) = sub(SE_A(A, k + 1, j), mul(v0, s));
        for (int i = k + 2; i < m; ++i) SE_A(A, i, j) = sub(SE_A(A, i, j), mul(SE_A(A, i, k), s));
      }
    } else {
      for (int i = t; i < m; i += zt) {
        zc s = mul(SE_A(Z, i, k + 1), v0);
        for (int j = k + 2; j < m; ++j) s = add(s, mul(SE_A(Z, i, j), SE_A(A, j, k)));
        s = scl(s, beta);
        SE_A(Z, i, k + 1) = sub(SE_A(Z, i, k + 1), mul(s, cj(v0)));
        for (int j = k + 2; j < m; ++j)
          SE_A(Z, i, j) = sub(SE_A(Z, i, j), mul(s, cj(SE_A(A, j, k))));
      }
    }
    __syncthreads();
    // right on A: one thread per row
    for (int i = tid; i < m; i += nt) {
      zc s = mul(SE_A(A, i, k + 1), v0);
      for (int j = k + 2; j < m; ++j) s = add(s, mul(SE_A(A, i, j), SE_A(A, j, k)));
      s = scl(s, beta);
      SE_A(A, i, k + 1) = sub(SE_A(A, i, k + 1), mul(s, cj(v0)));
      for (int j = k + 2; j < m; ++j)
        SE_A(A, i, j) = sub(SE_A(A, i, j), mul(s, cj(SE_A(A, j, k))));
    }
    __syncthreads();
    for (int i = k + 1 + tid; i < m; i += nt) SE_A(A, i, k) = i == k + 1 ? sh_alpha : mk(0.0, 0.0);
    __syncthreads();
  }

  // 2. shifted QR on the Hessenberg matrix (full Schur form)
  if (tid == 0) {
    sh_ihi = m - 1;
    sh_state = 0;
  }
  int iter = 0;   // thread 0's
  for (;;) {
    __syncthreads();   // the previous sweep's updates are done
    if (tid == 0) {
      int ihi = sh_ihi, l = 0;
      // deflate every converged 1 x 1 block, then the active block l .. ihi
      while (ihi >= 0) {
        l = ihi;
        while (l > 0) {
          const double tst = abs1(SE_A(A, l - 1, l - 1)) + abs1(SE_A(A, l, l));
          if (abs1(SE_A(A, l, l - 1)) <= eps * (tst > 0.0 ? tst : 1.0)) {
            SE_A(A, l, l - 1) = mk(0.0, 0.0);
            break;
          }
          --l;
        }
        if (l != ihi) break;
        gw[ihi] = SE_A(A, ihi, ihi);
        --ihi;
        iter = 0;
      }
      sh_ihi = ihi;
      sh_l = l;
      if (ihi >= 0) {
        zc mu;
        if (++iter % 11 == 10) {
          const double e = abs1(SE_A(A, ihi, ihi - 1));
          mu = add(SE_A(A, ihi, ihi), mk(0.75 * e, -0.4375 * e));   // exceptional shift
        } else {
          const zc a = SE_A(A, ihi - 1, ihi - 1), b = SE_A(A, ihi - 1, ihi);
          const zc c = SE_A(A, ihi, ihi - 1), d = SE_A(A, ihi, ihi);
          const zc tr2 = scl(add(a, d), 0.5);
          const zc hd = scl(sub(a, d), 0.5);
          const zc disc = csqrt_(add(mul(hd, hd), mul(b, c)));
          const zc e1 = add(tr2, disc), e2 = sub(tr2, disc);
          mu = abs2(sub(e1, d)) <= abs2(sub(e2, d)) ? e1 : e2;
        }
        // a non-finite matrix never converges: give up at once
        if (iter > 60 * m || !isfinite(mu.re) || !isfinite(mu.im)) sh_state = ihi + 1;
        givens_fast(sub(SE_A(A, l, l), mu), SE_A(A, l + 1, l), sh_c[l & 1], sh_s[l & 1]);
      }
    }
    __syncthreads();
    const int ihi = sh_ihi, l = sh_l;
    if (ihi < 0 || sh_state != 0) break;
    for (int k = l; k < ihi; ++k) {
      const double c = sh_c[k & 1];
      const zc s = sh_s[k & 1];
      const int rmax = (k + 2 < ihi ? k + 2 : ihi);
      if (tid < 32) {
        // rows k, k+1 of the columns k, k+1 and (the bulge) k-1, then columns k, k+1 of the rows
        // k .. k+2: four lanes an item, a real number each (givens_lanes)
        const int g = tid / 4, j = g < 2 ? k + g : k - 1;
        rotate_lanes(&SE_A(A, k, j), &SE_A(A, k + 1, j), g < (k > l ? 3 : 2), c, s);
        const int i = k + g;
        const double p = rotate_lanes(&SE_A(A, i, k), &SE_A(A, i, k + 1), g < 3 && i <= rmax, c, cj(s));
        // the next rotation zeroes A(k+2, k) against A(k+1, k)
        if (k + 1 < ihi)
          givens_lanes(mk(__shfl_sync(0xffffffffu, p, 4), __shfl_sync(0xffffffffu, p, 5)),
                       mk(__shfl_sync(0xffffffffu, p, 8), __shfl_sync(0xffffffffu, p, 9)),
                       sh_c[(k + 1) & 1], sh_s[(k + 1) & 1]);
      } else {
        // rows k, k+1 of the columns beyond k+1, columns k, k+1 of the rows above k, and of Z
        const int nrow = m - k - 2 > 0 ? m - k - 2 : 0;
        for (int u = tid - 32; u < nrow + k + m; u += nt - 32) {
          zc *p, *q;
          zc su = cj(s);
          if (u < nrow) {
            p = &SE_A(A, k, k + 2 + u);
            q = &SE_A(A, k + 1, k + 2 + u);
            su = s;
          } else {
            const int i = u - nrow;
            zc* M = i < k ? A : Z;
            const int r = i < k ? i : i - k;
            p = &SE_A(M, r, k);
            q = &SE_A(M, r, k + 1);
          }
          zc pv = *p, qv = *q;
          rotate(pv, qv, c, su);
          *p = pv;
          *q = qv;
        }
      }
      __syncthreads();
    }
  }
  if (sh_state != 0) return sh_state;

  // 3. eigenvectors of T by back substitution (one thread each), then Z y
  double tnorm = 0.0;
  for (int j = 0; j < m; ++j)
    for (int i = tid; i <= j; i += nt) tnorm = fmax(tnorm, abs1(SE_A(A, i, j)));
  __shared__ double sh_t[32];
  for (int off = 16; off > 0; off >>= 1) tnorm = fmax(tnorm, __shfl_xor_sync(0xffffffffu, tnorm, off));
  if (tid % 32 == 0) sh_t[tid / 32] = tnorm;
  __syncthreads();
  for (int q = 0; q < nt / 32; ++q) tnorm = fmax(tnorm, sh_t[q]);
  const double small_pivot = eps * (tnorm > 0.0 ? tnorm : 1.0);
  for (int e = tid; e < m; e += nt) {
    zc* y = &SE_A(Y, 0, e);
    for (int i = 0; i < m; ++i) y[i] = mk(0.0, 0.0);
    y[e] = mk(1.0, 0.0);
    const zc lam = SE_A(A, e, e);
    for (int i = e - 1; i >= 0; --i) {
      zc s = mk(0.0, 0.0);
      for (int k = i + 1; k <= e; ++k) s = add(s, mul(SE_A(A, i, k), y[k]));
      zc dnm = sub(SE_A(A, i, i), lam);
      if (abs1(dnm) < small_pivot) dnm = mk(small_pivot, 0.0);
      y[i] = dvd(mk(-s.re, -s.im), dnm);
    }
  }
  __syncthreads();
  // A <- Z Y (y_e has zeros below row e), then normalise into V
  for (int x = tid; x < m * m; x += nt) {
    const int i = x % m, e = x / m;
    zc s = mk(0.0, 0.0);
    for (int k = 0; k <= e; ++k) s = add(s, mul(SE_A(Z, i, k), SE_A(Y, k, e)));
    SE_A(A, i, e) = s;
  }
  __syncthreads();
  for (int e = tid; e < m; e += nt) {
    double n2 = 0.0;
    for (int i = 0; i < m; ++i) n2 += abs2(SE_A(A, i, e));
    const double inv = n2 > 0.0 ? 1.0 / sqrt(n2) : 0.0;
    for (int i = 0; i < m; ++i) gV[(int64_t)e * m + i] = scl(SE_A(A, i, e), inv);
  }
  return 0;
}

#undef SE_A

}  // namespace small
}  // namespace bem
