// FP64-accurate products of tall matrices on the tensor core (split64.cu).
#pragma once

#include "internal.h"

namespace bem {

// Workspace of the split products of an n x nu basis (Gram matrix and multiplication).
struct Split64 {
  bool use = false;
  int64_t n = 0, ldv = 0;
  int nu = 0;
  int kbn = 0, kbu = 0;      // 16-deep K-blocks along the rows, along the columns
  int mtu = 0, ntu = 0;      // 128-wide and 32-wide tiles of the columns
  int64_t mtn = 0;           // 128-row tiles
  int parts = 0;             // row ranges of the Gram matrix (its partial sums)
  unsigned char *a = nullptr, *b = nullptr;   // digit planes of the two operands
  unsigned* hcol = nullptr;                   // largest high words of the columns
  int *erow = nullptr, *ez = nullptr;         // exponents of the rows and of the factor
};

// Workspace of the split products of an n x nu basis (0: the FP64 kernels are the better choice).
size_t split64_bytes(const bem_ctx* ctx, int64_t n, int nu);
// Fills sp for an n x nu basis of leading dimension ldv, in mem (split64_bytes); use is false where the
// FP64 kernels are the better choice.
void split64_plan(bem_ctx* ctx, int64_t ldv, int64_t n, int nu, void* mem, Split64& sp);
// Row ranges of the Gram matrix of an n x nu basis (partial sums to provide for).
int split64_parts(const bem_ctx* ctx, int64_t n, int nu);
// part[r][b nu + a] = sum over row range r of conj(V[i][a]) V[i][b] for the upper 32 x 32 tiles
// (sp.parts ranges). Skipped on the device when gate is given and *gate == 0.
bem_status split64_gram(bem_ctx* ctx, const Split64& sp, const double2* V, double2* part,
                        const int* gate, cudaStream_t s);
// V <- V Z, Z nu x nu upper triangular. same: V is unchanged since split64_gram (its scales are
// there). Skipped when (gate and *gate == 0) or (skip and *skip != 0).
bem_status split64_multiply(bem_ctx* ctx, const Split64& sp, bool same, double2* V,
                            const double2* Z, const int* gate, const int* skip, cudaStream_t s);

// Products A_s X, s < S, of n x kc matrices A_s (column-major, ld n) with the rows of X, in
// `bytes` of workspace; X is taken kc rows at a time.
struct SplitBatch {
  int64_t n = 0, mtn = 0;   // rows and their 128-row tiles
  int S = 0, nu = 0, ntu = 0, kc = 0;
  size_t b_off = 0, e_off = 0, bytes = 0;
};
SplitBatch split64_batch_plan(int64_t n, int kc, int S, int ncols);
// The scales of X's columns (all n rows), once before the products.
bem_status split64_batch_scales(bem_ctx* ctx, const SplitBatch& b, char* work, const double2* X,
                                int64_t ldx, cudaStream_t s);
// out_s (n x nu, ld n, one after the other) (+)= A_s X for kc <= b.kc columns of the A_s (astep
// elements apart) and rows of X.
bem_status split64_batch(bem_ctx* ctx, const SplitBatch& b, char* work, const double2* A,
                         int64_t astep, int kc, const double2* X, int64_t ldx, bool add,
                         double2* out, cudaStream_t s);

// C_j = scale_j X^H Y_j, j < nb (as launch_xhy_fp64, Y contiguous with ld n).
struct SplitCross {
  bool use = false;         // large enough to pay, and its workspace within bounds
  int64_t n = 0;
  int p = 0, q = 0, nb = 0;
  int mtp = 0, nt = 0, parts = 1;   // 128-row and 32-column tiles of the outputs, row ranges
  size_t b_off = 0, part_off = 0, h_off = 0, bytes = 0;
};
SplitCross split64_cross_plan(const bem_ctx* ctx, int64_t n, int p, int q, int nb);
bem_status split64_cross(bem_ctx* ctx, const SplitCross& c, void* work, const double2* X,
                         int64_t ldx, const double2* Y, const double2* scale, double2* C,
                         cudaStream_t s);

}  // namespace bem
