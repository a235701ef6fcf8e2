// Residuals of approximate eigenpairs, matrix-free in FP64 (Section 4: the accuracy of an
// eigenpair (lambda, u) is ||T(lambda) u||_2 / ||u||_2).
//
// residual_kernel: r = A(lambda_c) x_c, one thread per row, columns of A streamed through
// shared memory in chunks; norms_kernel: ||r_c||^2 and ||x_c||^2 by a fixed-order block
// reduction (deterministic).
#include <math.h>

#include <algorithm>
#include <string>
#include <vector>

#include "expand64.h"
#include "internal.h"

namespace bem {
namespace {

constexpr int kRowsPerBlock = 128;
constexpr int kChunk = 128;

// kDeriv: the k-derivative of the off-diagonal entries, sum_q W_lq i exp(i k r) / (4 pi).
template <bool kDeriv>
__global__ void __launch_bounds__(kRowsPerBlock)
residual_kernel(Geometry g, const double* __restrict__ lam, const double* __restrict__ X,
                int64_t ldx, double* __restrict__ R, OpCoef op) {
  __shared__ double sQ[4][7][kChunk];
  __shared__ double sN[3][kChunk];
  const bool general = !op_single(op);
  __shared__ double2 sX[kChunk];
  const int64_t n = g.n;
  const int c = blockIdx.y;
  const int64_t i = (int64_t)blockIdx.x * kRowsPerBlock + threadIdx.x;
  const double kr = lam[2 * c], ki = lam[2 * c + 1];
  const double2* x = reinterpret_cast<const double2*>(X) + (int64_t)c * ldx;
  double xi = 0, yi = 0, zi = 0;
  if (i < n) {
    xi = g.cx[i]; yi = g.cx[n + i]; zi = g.cx[2 * n + i];
  }
  double2 acc = make_double2(0.0, 0.0);
  double2 self_x = make_double2(0.0, 0.0);   // x_i, multiplied by the self term below
  for (int64_t l0 = 0; l0 < n; l0 += kChunk) {
    __syncthreads();
    for (int t = threadIdx.x; t < 7 * kChunk; t += blockDim.x) {
      const int q = t / kChunk, lc = t % kChunk;
      const int64_t l = l0 + lc;
      const bool ok = l < n;
      sQ[0][q][lc] = ok ? g.qp[q * n + l] : 0.0;
      sQ[1][q][lc] = ok ? g.qp[(7 + q) * n + l] : 0.0;
      sQ[2][q][lc] = ok ? g.qp[(14 + q) * n + l] : 0.0;
      sQ[3][q][lc] = ok ? g.qw[q * n + l] : 0.0;
    }
    for (int t = threadIdx.x; t < kChunk; t += blockDim.x) {
      const int64_t l = l0 + t;
      sX[t] = (l < n) ? x[l] : make_double2(0.0, 0.0);
      if (general)
        for (int c2 = 0; c2 < 3; ++c2) sN[c2][t] = (l < n) ? g.nrm[c2 * n + l] : 0.0;
    }
    __syncthreads();
    if (i < n) {
      const int lim = (int)((n - l0) < kChunk ? (n - l0) : kChunk);
      for (int lc = 0; lc < lim; ++lc) {
        const int64_t l = l0 + lc;
        if (l == i) {
          self_x = sX[lc];
          continue;
        }
        double2 a = make_double2(0.0, 0.0);
        if (general) {   // T = c_G G + c_H (1/2 I + K), or its k-derivative
          for (int q = 0; q < 7; ++q)
            op_point64(a, op, sQ[3][q][lc], sQ[0][q][lc] - xi, sQ[1][q][lc] - yi,
                       sQ[2][q][lc] - zi, sN[0][lc], sN[1][lc], sN[2][lc], kr, ki, kDeriv);
        } else
        for (int q = 0; q < 7; ++q) {
          const double dx = xi - sQ[0][q][lc], dy = yi - sQ[1][q][lc], dz = zi - sQ[2][q][lc];
          const double r = sqrt(dx * dx + dy * dy + dz * dz);
          double s, co;
          sincos(kr * r, &s, &co);
          const double amp = kDeriv ? sQ[3][q][lc] * exp(-ki * r) : sQ[3][q][lc] * exp(-ki * r) / r;
          if (kDeriv) {   // i * amp * (co + i s)
            a.x -= amp * s;
            a.y += amp * co;
          } else {
            a.x += amp * co;
            a.y += amp * s;
          }
        }
        const double2 v = sX[lc];
        acc.x += a.x * v.x - a.y * v.y;
        acc.y += a.x * v.y + a.y * v.x;
      }
    }
  }
  if (i < n) {
    // R holds A_ii(lambda_c), written by launch_self_at before this kernel runs
    double2* Rc = reinterpret_cast<double2*>(R) + (int64_t)c * n;
    const double2 sd = Rc[i];
    acc.x += sd.x * self_x.x - sd.y * self_x.y;
    acc.y += sd.x * self_x.y + sd.y * self_x.x;
    Rc[i] = acc;
  }
}

__global__ void norms_kernel(const double* __restrict__ R, const double* __restrict__ X,
                             int64_t ldx, int64_t n, double* __restrict__ out) {
  __shared__ double sr[256], sx[256];
  const int c = blockIdx.x;
  const double2* r = reinterpret_cast<const double2*>(R) + (int64_t)c * n;
  const double2* x = reinterpret_cast<const double2*>(X) + (int64_t)c * ldx;
  double ar = 0.0, ax = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    ar += r[i].x * r[i].x + r[i].y * r[i].y;
    ax += x[i].x * x[i].x + x[i].y * x[i].y;
  }
  sr[threadIdx.x] = ar;
  sx[threadIdx.x] = ax;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      sr[threadIdx.x] += sr[threadIdx.x + w];
      sx[threadIdx.x] += sx[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[2 * c] = sr[0];
    out[2 * c + 1] = sx[0];
  }
}

}  // namespace

cudaError_t launch_apply_percol64(bem_ctx* ctx, int m, const double* lam_dev, const double* X,
                                  int64_t ldx, double* R, bool deriv, cudaStream_t s) {
  const int64_t n = ctx->geo.n;
  const cudaError_t e = launch_self_at(ctx, m, lam_dev, R, deriv, s);
  if (e != cudaSuccess) return e;
  dim3 g2((unsigned)((n + kRowsPerBlock - 1) / kRowsPerBlock), (unsigned)m);
  if (deriv)
    residual_kernel<true><<<g2, kRowsPerBlock, 0, s>>>(ctx->geo, lam_dev, X, ldx, R, ctx->op);
  else
    residual_kernel<false><<<g2, kRowsPerBlock, 0, s>>>(ctx->geo, lam_dev, X, ldx, R, ctx->op);
  ctx->launches++;
  if (near_active(ctx)) return launch_near_percol64(ctx, m, lam_dev, X, ldx, R, deriv, s);
  return cudaGetLastError();
}

cudaError_t launch_colnorms(bem_ctx* ctx, const double* R, int64_t ldr, const double* X,
                            int64_t ldx, int64_t n, int m, double* out, cudaStream_t s) {
  (void)ldr;
  norms_kernel<<<m, 256, 0, s>>>(R, X, ldx, n, out);
  ctx->launches++;
  return cudaGetLastError();
}

}  // namespace bem

using namespace bem;

namespace {

// Whether the FP64 expansion is faster than the double-FP32 kernel (its time depends on the
// columns, the expansion's hardly does), in us, both with the self terms:
//   12 panels 217 / 155, 32 227 / 208, 48 232 / 249, 64 235 / 292, 108 259 / 407;
//   4800 panels: 16.9 ms for any number of columns against 7.8 ms at 4, 22.8 ms at 12; 768 panels
//   0.76 ms against 0.61 at 8, 0.79 at 12; the near pairs 15 ns once against 23 ns a column (4800
//   panels with near field, 12 columns: 19.4 against 67.8 ms).
bool expand_beats_ff(const bem_ctx* ctx, const ExpandPlan& ex, int m, bool deriv) {
  const double n2 = (double)ctx->geo.n * (double)ctx->geo.n;
  const double pairs = near_active(ctx) ? (double)ctx->near_nnz : 0.0;
  const double expand = 240.0 + n2 * ex.cost / 5.3e5 + pairs * 0.015;
  const double few = std::min(450.0, 125.0 + 2.6 * (double)ctx->geo.n);
  const double ff = std::max(few, 200.0 + n2 * m * 0.082e-3) + pairs * m * 0.023;
  return ex.use && (deriv ? 2.0 : 1.0) * expand < 0.9 * ff;
}

bem_status residual_impl(bem_ctx* ctx, int m, const double* lam_host, const double* X_dev,
                         int64_t ldx, double* R_dev, double* Rd_dev, double* relres_host,
                         int arith, void* stream, const char* name) {
  if (!ctx) return BEM_EINVAL;
  if (ctx->geo.n == 0) return fail(ctx, BEM_ESTATE, std::string(name) + ": no mesh set");
  const int64_t n = ctx->geo.n;
  if (m < 1 || m > 65535 || !lam_host || !X_dev || !relres_host || ldx < n ||
      (arith != 0 && arith != 1))
    return fail(ctx, BEM_EINVAL, std::string(name) +
                                     ": need 1 <= m <= 65535, lam, X, relres, ldx >= n, arith 0/1");
  for (int c = 0; c < 2 * m; ++c)
    if (!isfinite(lam_host[c])) return fail(ctx, BEM_EINVAL, std::string(name) + ": non-finite lambda");
  cudaSetDevice(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  bem_status st = ensure_near(ctx, s);
  if (st != BEM_OK) return st;
  // workspace: lambda (2m) + norms (2m) [+ R if the caller passes none]
  const size_t small = (size_t)4 * m * sizeof(double);
  st = ensure_small(ctx, small);
  if (st != BEM_OK) return st;
  // One FP64 evaluation expanded about the middle of the given values for all columns, where that
  // costs less than one per column (in FP64, or in double-FP32 if asked for: single layer only)
  // and its workspace can be had
  st = ensure_scratch(ctx, R_dev ? 0 : (size_t)2 * n * m * sizeof(double));
  if (st != BEM_OK) return st;
  ExpandUse ws(ctx, s);
  ExpandPlan ex, exd;   // of A, and of A' if it is asked for
  {
    double lo[2] = {lam_host[0], lam_host[1]}, hi[2] = {lam_host[0], lam_host[1]};
    for (int c = 0; c < 2 * m; ++c) {
      lo[c % 2] = std::min(lo[c % 2], lam_host[c]);
      hi[c % 2] = std::max(hi[c % 2], lam_host[c]);
    }
    const double cr = 0.5 * (lo[0] + hi[0]), ci = 0.5 * (lo[1] + hi[1]);
    const int ar = op_single(ctx->op) ? arith : 0;
    ex = expand_plan(ctx, m, lam_host, cr, ci, m, false, false, ar);
    if (Rd_dev) {
      exd = expand_plan(ctx, m, lam_host, cr, ci, m, false, true, ar);
      ex.use = ex.use && exd.use;
    }
    if (arith == 1 && op_single(ctx->op) && !expand_beats_ff(ctx, ex, m, Rd_dev != nullptr)) ex.use = false;
    ex.use = ex.use && ws.get(std::max(ex.bytes, exd.bytes));
  }
  double* R = R_dev ? R_dev : ctx->d_scratch;
  double* dlam = ctx->d_small;
  double* dnorm = ctx->d_small + 2 * m;
  st = cuda_check(ctx, cudaMemcpyAsync(dlam, lam_host, 2 * m * sizeof(double),
                                       cudaMemcpyHostToDevice, s), name);
  if (st != BEM_OK) return st;
  cudaError_t e = cudaSuccess;
  if (arith == 1 && !ex.use) {
    e = launch_apply_ff(ctx, m, dlam, X_dev, ldx, R, Rd_dev, s);
  } else if (ex.use) {
    st = expand_apply_columns(ctx, ex, m, dlam, X_dev, ldx, R, ws.work, s);
    if (st == BEM_OK && Rd_dev)
      st = expand_apply_columns(ctx, exd, m, dlam, X_dev, ldx, Rd_dev, ws.work, s);
    if (st != BEM_OK) return st;
  } else {
    e = launch_apply_percol64(ctx, m, dlam, X_dev, ldx, R, false, s);
    if (e == cudaSuccess && Rd_dev) e = launch_apply_percol64(ctx, m, dlam, X_dev, ldx, Rd_dev, true, s);
  }
  st = cuda_check(ctx, e, name);
  if (st != BEM_OK) return st;
  st = cuda_check(ctx, launch_colnorms(ctx, R, n, X_dev, ldx, n, m, dnorm, s), name);
  if (st != BEM_OK) return st;
  std::vector<double> h(2 * m);
  const bool waits = ex.use && (ex.split || exd.split);
  int flags = 0;
  st = cuda_check(ctx, cudaMemcpyAsync(h.data(), dnorm, 2 * m * sizeof(double),
                                       cudaMemcpyDeviceToHost, s), name);
  if (st == BEM_OK && waits)
    st = cuda_check(ctx, cudaMemcpyAsync(&flags, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, s), name);
  if (st == BEM_OK) st = cuda_check(ctx, cudaStreamSynchronize(s), name);
  if (st != BEM_OK) return st;
  // the split products' waits are bounded: norms of products that gave up are no result. (What other
  // calls recorded is left to bem_check, as ever, where this one has no such wait.)
  if (flags & kStatusTimeout) return take_status(ctx, s, name);
  for (int c = 0; c < m; ++c)
    relres_host[c] = h[2 * c + 1] > 0.0 ? sqrt(h[2 * c]) / sqrt(h[2 * c + 1]) : INFINITY;
  return BEM_OK;
}

}  // namespace

extern "C" bem_status bem_residual(bem_ctx* ctx, int m, const double* lam_host, const double* X_dev,
                                   int64_t ldx, double* R_dev, double* relres_host, void* stream) {
  return residual_impl(ctx, m, lam_host, X_dev, ldx, R_dev, nullptr, relres_host, 0, stream,
                       "bem_residual");
}

extern "C" bem_status bem_residual_arith(bem_ctx* ctx, int m, const double* lam_host,
                                         const double* X_dev, int64_t ldx, double* R_dev,
                                         double* Rd_dev, double* relres_host, int arith,
                                         void* stream) {
  return residual_impl(ctx, m, lam_host, X_dev, ldx, R_dev, Rd_dev, relres_host, arith, stream,
                       "bem_residual_arith");
}
