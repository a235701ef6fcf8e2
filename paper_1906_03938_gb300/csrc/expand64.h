// FP64 products with the operator at many wavenumbers from one evaluation (expand64.cu).
#pragma once

#include "internal.h"
#include "split64.h"

namespace bem {

constexpr int kMaxTerms = 32;   // longest series the kernels are built for

struct FixedPhase {
  double inv_R;   // rho = r inv_R
  long long K;    // turns per unit of rho, times 2^(62 - kb)
  int kb;
};

struct ExpandPlan {
  bool use = false;        // the expansion applies and costs less than the direct form
  int M = 0;               // series terms
  bool hasG = false;       // a family for the single layer
  int nh = 0, fams = 0;    // families for the double layer; all of them
  bool deriv = false;      // the k-derivative's families
  int S = 0;               // slots, fams M
  int kc = 0;              // columns evaluated at a time
  int splits = 1;          // shares of those columns in the products
  double R = 0.0;          // largest distance
  double cost = 0.0;       // time per entry, in FP64 operations
  double2 c{};             // centre
  FixedPhase phase{};
  bool split = false;      // products on the tensor core (split64.cu)
  SplitBatch batch;
  size_t coef_off = 0, mom_off = 0, y_off = 0, batch_off = 0, near_off = 0, bytes = 0;
};

// Weights of the moments, by their first family.
enum MomentKind { kSingle, kSingleDeriv, kDouble, kDoubleDeriv };

// Plan for the nk wavenumbers k (re, im on the host), expanded about (c_re, c_im), and ncols columns:
// every wavenumber times every column (nodes), or wavenumber c times column c; of A, or (deriv) of A'.
// arith 1: in the place of double-FP32 products.
ExpandPlan expand_plan(bem_ctx* ctx, int nk, const double* k, double c_re, double c_im, int ncols,
                       bool nodes, bool deriv, int arith = 0);
// Y_j = A(z_j) V for all nodes of the contour (its FP64 self-term table filled), near field
// included; Y as launch_apply_fp64's. work: plan's bytes.
bem_status expand_apply_nodes(bem_ctx* ctx, const ExpandPlan& p, const double* V, int64_t ldv,
                              int nu, double* Y, void* work, cudaStream_t s);
// As launch_apply_percol64 (A' for a plan of the derivative), near field included.
bem_status expand_apply_columns(bem_ctx* ctx, const ExpandPlan& p, int m, const double* lam_dev,
                                const double* X, int64_t ldx, double* R, void* work, cudaStream_t s);
// Near pairs (near.cu): Y_s += C_s X for every slot, C_s the moments of the corrections
// (A_near - A_7), in near_expand_bytes of workspace.
size_t near_expand_bytes(const bem_ctx* ctx, const ExpandPlan& p, int ncols);
bem_status near_expand64(bem_ctx* ctx, const ExpandPlan& p, const int4* angles, const double* X,
                         int64_t ldx, int ncols, double2* Ys, void* work, cudaStream_t s);

}  // namespace bem
