// The eigen-decomposition of small_eig.h by one block (same algorithm, same deflation rule
// and shifts).
//
// Bound by the serial chain of Givens rotations: about 3 m sweeps of up to m rotations, each
// needing the previous one's result in two entries. On one thread every rotation also paid
// for its ~3 m complex row and column updates (m = 32: 80 ms); here the updates are spread
// over the threads, the rows and columns of A and Z in shared memory (m <= 64), and the
// thread that owns the chain forms the next rotation while the others still update, so a
// rotation costs two barriers and one chain step. m = 32: 80.6 ms -> 6.3 ms.
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
// half the threads update A, the other half Z
__host__ inline int eig_threads(int m) { return 2 * (m < 32 ? 32 : (m + 31) / 32 * 32); }

// Givens rotation as small::givens, by reciprocal square roots where the squares are safe.
__device__ inline void givens_fast(zc x, zc y, double& c, zc& s) {
  const double ax2 = abs2(x), ay2 = abs2(y);
  if (!(ax2 > 1e-200 && ax2 < 1e200 && ay2 > 1e-200 && ay2 < 1e200)) {
    givens(x, y, c, s);
    return;
  }
  const double ix = rsqrt(ax2), in = rsqrt(ax2 + ay2);
  c = ax2 * ix * in;
  s = scl(mul(x, cj(y)), ix * in);
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
  const int tid = threadIdx.x, nt = blockDim.x, half = nt / 2;
  const bool first = tid < half;      // this thread works on A (else on Z)
  const int t = first ? tid : tid - half;
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
      for (int i = t; i < m; i += half) {
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
      if (first) {
        // rows k, k+1: columns from max(l, k-1) to m-1
        for (int j = (k > l ? k - 1 : l) + t; j < m; j += half) {
          const zc t1 = SE_A(A, k, j), t2 = SE_A(A, k + 1, j);
          SE_A(A, k, j) = add(scl(t1, c), mul(s, t2));
          SE_A(A, k + 1, j) = sub(scl(t2, c), mul(cj(s), t1));
        }
      } else {
        for (int i = t; i < m; i += half) {
          const zc t1 = SE_A(Z, i, k), t2 = SE_A(Z, i, k + 1);
          SE_A(Z, i, k) = add(scl(t1, c), mul(cj(s), t2));
          SE_A(Z, i, k + 1) = sub(scl(t2, c), mul(s, t1));
        }
      }
      __syncthreads();
      // columns k, k+1: rows 0 .. min(k+2, ihi); thread 0 takes rows k+1 and k+2, whose new
      // entries of column k are the next rotation's, and forms it
      const int rmax = (k + 2 < ihi ? k + 2 : ihi);
      auto col = [&](int i) {
        const zc t1 = SE_A(A, i, k), t2 = SE_A(A, i, k + 1);
        const zc a = add(scl(t1, c), mul(cj(s), t2));
        SE_A(A, i, k) = a;
        SE_A(A, i, k + 1) = sub(scl(t2, c), mul(s, t1));
        return a;
      };
      if (tid == 0) {
        const zc x = col(k + 1);
        if (k + 2 <= rmax) {
          const zc y = col(k + 2);
          givens_fast(x, y, sh_c[(k + 1) & 1], sh_s[(k + 1) & 1]);
        }
      } else {
        for (int i = tid - 1; i <= k; i += nt - 1) col(i);
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
