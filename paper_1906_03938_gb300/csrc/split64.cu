// FP64-accurate Gram matrix V^H V and product V Z of a tall complex basis on the tensor core.
//
// FP64 runs at 1/64 of the FP32 rate on this part (1.06e12 flop/s), BF16 products at 1.9e15.
// Each operand is scaled by powers of two (its columns, its rows) to |x| < 1 and cut into
// seven signed 8-bit digits, x = 2^-7 sum_s d_s 2^(-8 s), |d_s| <= 128, |rest| <= 2^-56: the
// error-free splitting of Ozaki, Ogita, Oishi and Rump (2012). A digit is exact in BF16 and a
// product of two an integer up to 2^14, so the FP32 accumulators sum exactly up to 2^24. The
// digit pairs s + t <= 7 go into eight accumulators by d = s + t; those left out are below
// 2^-61 of the scales' product a term. The accumulators are added to 64-bit integers in
// registers (d >= 4 every 64 rows, d < 4, which collect fewer pairs, every 128), so a whole sum
// is exact until its single conversion to FP64: the errors are the digits' cut and that
// rounding. The cut is one of the whole column (or row): a sum of K terms is off by up to
// 2.1 K 2^-53 max|a| max|b|, the bound of an FP64 sum of entries that are all as large. Entries far
// below their column's largest keep fewer bits (2^-20 of it: 36), so this bound holds normwise where
// an FP64 sum's holds term by term; for Gaussian columns the sums are more exact than FP64's
// (X^H Y_j at 768 x 64 1e-16 against 1.2e-15).
//
// split_gemm_kernel: a block owns 128 x 32 complex outputs, [Re | Im] of the 32 columns as the
// 64 columns of each accumulator (8 x 64 = all 512 TMEM columns). Per 16-deep K-block two bulk
// copies bring the left operand's digit planes (re, im) and the right operand's in the two
// arrangements the complex product needs; one thread issues the MMAs, eight warps empty the
// accumulators. The right operand's digits t follow one another in shared memory as the
// accumulators s + t do in TMEM, so one MMA takes a left digit s against up to four digits t
// (N = 256): 11 MMAs for the 34 pairs. An MMA reads its 128 x 16 left operand in 128 cycles
// whatever N, so a pair to itself (N = 64) cost four times as much.
//
// Measured at 98304 x 256, a Gram matrix or a product: 1.03 ms (0.62 ms of it MMA cycles, the
// rest waits for the accumulators' reads) and 0.4 ms for scales and digits, against 24 ms on the
// FP64 pipe; a whole CholeskyQR2 101 -> 6.4 ms with ||Q^H Q - I|| 7.4e-16 -> 6.5e-16. One
// MMA (N = 64) per pair took 2.3 ms; eight 7-bit digits with 36 pairs left 1.5e-15.
#include <cuda_bf16.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "sm100.cuh"
#include "split64.h"

namespace bem {
namespace {

using namespace sm100;

constexpr int kDigits = 7, kOrders = 8;      // digits, accumulators d = s + t
constexpr int kTileM = 128, kTileN = 32;      // outputs of a block (complex columns of N)
constexpr uint32_t kABytes = kDigits * 2 * 4096;   // digit planes of a 128 x 16 block
constexpr uint32_t kBHalf = kDigits * 2048;  // [first | second part] planes of a 32 x 16 block
constexpr uint32_t kBBytes = 2 * kBHalf;     // for the real, then the imaginary left digits
constexpr int kStagesG = 2;
constexpr int kFlush = 4;                     // K-blocks between two flushes of d >= 4 (64 rows)
constexpr int kFlushWarps = 8;
constexpr int kThreadsG = 32 * (2 + kFlushWarps);
constexpr uint32_t kDrainWait = kStageWaitDefault;   // of the waits before a block leaves
constexpr int kNotFinite = INT_MIN;           // exponent of a scale over non-finite values
constexpr int kZero = -4000;                  // of one over zeros
constexpr size_t kMaxSplitBytes = (size_t)8 << 30;
// n nu^2 from which the split products pay (more launches, less work). A CholeskyQR2, split
// against FP64 products, in us: 4096 x 32 209 / 169, 20000 x 16 285 / 270, 1452 x 64 248 / 233
// below it; 600 x 128 424 / 498, 12000 x 32 248 / 282, 3072 x 64 260 / 308, 6000 x 48 271 / 418,
// 50000 x 16 406 / 528, 8192 x 256 1909 / 7171 above.
constexpr int64_t kMinWork = (int64_t)1 << 23;

// n p q nb from which X^H Y_j by splitting pays. FP64 projections whose last step it is, split
// against FP64, in us: 192 panels, 16 columns, 16 nodes (2^19.6) 492 / 491; 300 x 10 x 24 457 / 535,
// 588 x 30 x 16 700 / 833, 972 x 100 x 16 1814 / 3654. Its error against 128-bit sums at 768 x 64
// is 1e-16, the FP64 kernel's 1.2e-15.
constexpr int64_t kMinCross = (int64_t)1 << 19;

__device__ __forceinline__ bool skipped(const int* gate, const int* skip) {
  return (gate && *gate == 0) || (skip && *skip != 0);
}

// |x|'s exponent e with |x| < 2^e, from the high word of the largest |x|
__device__ __forceinline__ int exponent_of(unsigned hi) {
  const int be = (int)(hi >> 20);
  if (be == 2047) return kNotFinite;
  if (be == 0) return hi == 0 ? kZero : -1021;   // (a zero high word: below 2^-1042, cut)
  return be - 1022;
}

// round(x 2^(55 - e)), |x| < 2^e
__device__ __forceinline__ long long fixed55(double x, int e) {
  const long long bits = __double_as_longlong(x);
  const int be = (int)((bits >> 52) & 2047);
  long long m = (bits & 0xFFFFFFFFFFFFFll) | (be ? 0x10000000000000ll : 0ll);
  const int k = (be ? be : 1) - 1020 - e;   // x = m 2^(be - 1075)
  if (k >= 0) m <<= k;
  else if (k > -56) m = (m + (1ll << (-k - 1))) >> -k;
  else m = 0;
  return bits < 0 ? -m : m;
}

// The digits of q = fixed55(x) for eight values, as rows of BF16: out[s] holds digit s of the
// eight. neg: of -x. With 128 added to every digit but the first they are the bytes of q, which
// become numbers as the low mantissa byte of 2^23 (no conversions, which run at an eighth of the
// rate).
__device__ __forceinline__ void digits8(const long long (&q)[8], uint4 (&out)[kDigits], bool neg) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const long long r = (neg ? -q[j] : q[j]) + 0x0000808080808080ll;
    lo[j] = (uint32_t)r;
    hi[j] = (uint32_t)(r >> 32);
  }
#pragma unroll
  for (int s = 0; s < kDigits; ++s) {
    uint32_t h[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      uint32_t m;   // 2^23 + 128 + digit
      if (s == 0) m = 0x4B000000u + (uint32_t)(((int)hi[j] >> 16) + 128);
      else if (s < 3) m = __byte_perm(hi[j], 0x4B000000u, 0x7440u | (2 - s));
      else m = __byte_perm(lo[j], 0x4B000000u, 0x7440u | (6 - s));
      h[j] = __float_as_uint(__uint_as_float(m) - 8388736.f);
    }
    out[s] = make_uint4(__byte_perm(h[0], h[1], 0x7632), __byte_perm(h[2], h[3], 0x7632),
                        __byte_perm(h[4], h[5], 0x7632), __byte_perm(h[6], h[7], 0x7632));
  }
}

// Largest high word of |re|, |im| per column (hi zeroed before).
__global__ void __launch_bounds__(256)
split_colmax_kernel(const double2* __restrict__ V, int64_t ldv, int64_t n, unsigned* hi,
                    const int* gate, const int* skip) {
  if (skipped(gate, skip)) return;
  const double2* v = V + (int64_t)blockIdx.x * ldv;
  unsigned m = 0;
  for (int64_t i = blockIdx.y * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.y * blockDim.x) {
    const double2 x = v[i];
    m = max(m, max((unsigned)__double2hiint(x.x) & 0x7FFFFFFFu, (unsigned)__double2hiint(x.y) & 0x7FFFFFFFu));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (threadIdx.x % 32 == 0 && m) atomicMax(hi + blockIdx.x, m);
}

__device__ __forceinline__ int scale_exp(int e) { return (e == kNotFinite || e == kZero) ? 0 : e; }
__device__ __forceinline__ int col_exp(const unsigned* hi, int c) { return scale_exp(exponent_of(hi[c])); }

// Digit planes of V's columns with the rows as K: a[kb][tile of 128 columns][digit][re, im] and
// b[kb][tile of 32 columns]{[digit][re | im], [digit][im | -re]} (b null: not written), in K-major
// core matrices. One thread per column and 8 rows.
__global__ void __launch_bounds__(128)
split_columns_kernel(const double2* __restrict__ V, int64_t ldv, int64_t n, int nu, int kbn,
                     int mtu, int ntu, const unsigned* __restrict__ hc, unsigned char* __restrict__ a,
                     unsigned char* __restrict__ b, const int* gate) {
  if (skipped(gate, nullptr)) return;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t groups = 2 * (int64_t)kbn;
  const int cols = mtu * kTileM;
  if (t >= groups * cols) return;
  // eight consecutive threads take one group of 8 rows in 8 columns: their 16-byte rows of a
  // core matrix are contiguous
  const int c = (int)(t % 8 + t / (8 * groups) * 8);
  const int64_t gr = t / 8 % groups;
  const int64_t kb = gr / 2;
  const int kh = (int)(gr % 2);
  long long re[8], im[8];
  const int e = c < nu ? col_exp(hc, c) : 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int64_t i = gr * 8 + j;
    const double2 v = (c < nu && i < n) ? V[(int64_t)c * ldv + i] : make_double2(0.0, 0.0);
    re[j] = fixed55(v.x, e);
    im[j] = fixed55(v.y, e);
  }
  uint4 d[kDigits];
  const int m = c % kTileM, r = c % kTileN;
  unsigned char* ap = a + ((size_t)kb * mtu + c / kTileM) * kABytes + (m / 8) * 256 + kh * 128 + (m % 8) * 16;
  unsigned char* bp = b + ((size_t)kb * ntu + c / kTileN) * kBBytes + (r / 8) * 256 + kh * 128 + (r % 8) * 16;
  const bool inb = b && c / kTileN < ntu;
  // part h of half w of the right operand: rows 32 h + r of the digit's 64
  auto put_b = [&](int w, int h) {
    if (!inb) return;
#pragma unroll
    for (int s = 0; s < kDigits; ++s)
      *reinterpret_cast<uint4*>(bp + w * kBHalf + s * 2048 + h * 1024) = d[s];
  };
  digits8(re, d, false);
#pragma unroll
  for (int s = 0; s < kDigits; ++s) *reinterpret_cast<uint4*>(ap + (2 * s) * 4096) = d[s];
  put_b(0, 0);
  digits8(im, d, false);
#pragma unroll
  for (int s = 0; s < kDigits; ++s) *reinterpret_cast<uint4*>(ap + (2 * s + 1) * 4096) = d[s];
  put_b(0, 1);
  put_b(1, 0);
  digits8(re, d, true);
  put_b(1, 1);
}

// Exponents of the rows of V D^-1, D the columns' scales (hc null: 1), and their digit planes with
// the columns as K: a[kb][matrix][tile of 128 rows][digit][re, im], blockIdx.y of gridDim.y
// matrices vstep apart. 32 rows a block, eight threads a row; the second pass over the block's
// rows comes from the caches.
__global__ void __launch_bounds__(256)
split_rows_kernel(const double2* __restrict__ V, int64_t ldv, int64_t vstep, int64_t n, int nu,
                  int kbu, int64_t mtn, const unsigned* __restrict__ hc, int* __restrict__ er,
                  unsigned char* __restrict__ a, const int* gate, const int* skip) {
  if (skipped(gate, skip)) return;
  __shared__ int ec[kMaxNu], se[8][32], sbad;
  V += blockIdx.y * vstep;
  er += blockIdx.y * n;
  a += blockIdx.y * (size_t)mtn * kABytes;
  const int lane = threadIdx.x % 32, q = threadIdx.x / 32;
  const int64_t i = blockIdx.x * (int64_t)32 + lane;
  if (threadIdx.x == 0) sbad = 0;
  __syncthreads();
  if (hc)
    for (int c = threadIdx.x; c < nu; c += 256) {
      const int e = exponent_of(hc[c]);
      if (e == kNotFinite) sbad = 1;
      ec[c] = scale_exp(e);
    }
  __syncthreads();
  int e = kZero;
  if (i < n)
#pragma unroll 4
    for (int c = q; c < nu; c += 8) {
      const double2 v = V[(int64_t)c * ldv + i];
      const int x = exponent_of(max((unsigned)__double2hiint(v.x) & 0x7FFFFFFFu,
                                    (unsigned)__double2hiint(v.y) & 0x7FFFFFFFu));
      if (x == kNotFinite) e = INT_MAX;
      else if (x != kZero) e = max(e, x - (hc ? ec[c] : 0));
    }
  se[q][lane] = e;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k) e = max(e, se[k][lane]);
  if (sbad || e == INT_MAX) e = kNotFinite;
  if (q == 0 && i < n) er[i] = e;
  e = scale_exp(e);
  const int m = (int)(i % kTileM);
  for (int gr = q; gr < 2 * kbu; gr += 8) {
    const int kb = gr / 2, kh = gr % 2;
    long long re[8], im[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = gr * 8 + j;
      const bool in = i < n && c < nu;
      const double2 v = in ? V[(int64_t)c * ldv + i] : make_double2(0.0, 0.0);
      const int ej = in ? e + (hc ? ec[c] : 0) : 0;
      re[j] = fixed55(v.x, ej);
      im[j] = fixed55(v.y, ej);
    }
    unsigned char* ap = a + ((size_t)kb * gridDim.y * mtn + i / kTileM) * kABytes + (m / 8) * 256 + kh * 128 + (m % 8) * 16;
    uint4 d[kDigits];
    digits8(re, d, false);
#pragma unroll
    for (int s = 0; s < kDigits; ++s) *reinterpret_cast<uint4*>(ap + (2 * s) * 4096) = d[s];
    digits8(im, d, false);
#pragma unroll
    for (int s = 0; s < kDigits; ++s) *reinterpret_cast<uint4*>(ap + (2 * s + 1) * 4096) = d[s];
  }
}

// Digit planes of the columns of D Z (Z upper triangular) with the rows as K:
// b[kb][tile of 32 columns]{[digit][re | im], [digit][-im | re]}; one block per column, and its
// exponent.
__global__ void __launch_bounds__(64)
split_factor_kernel(const double2* __restrict__ Z, int nu, int kbu, int ntu,
                    const unsigned* __restrict__ hc, int* __restrict__ ez, unsigned char* __restrict__ b,
                    const int* gate, const int* skip) {
  if (skipped(gate, skip)) return;
  __shared__ int se[2], sbad;
  const int c = blockIdx.x, tid = threadIdx.x;
  if (tid == 0) sbad = 0;
  __syncthreads();
  int e = kZero;
  if (c < nu)
    for (int k = tid; k <= c; k += 64) {
      const double2 z = Z[(int64_t)c * nu + k];
      const int x = exponent_of(max((unsigned)__double2hiint(z.x) & 0x7FFFFFFFu,
                                    (unsigned)__double2hiint(z.y) & 0x7FFFFFFFu));
      if (x == kNotFinite) sbad = 1;
      else if (x != kZero) e = max(e, x + col_exp(hc, k));
    }
  for (int off = 16; off > 0; off >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
  if (tid % 32 == 0) se[tid / 32] = e;
  __syncthreads();
  e = max(se[0], se[1]);
  if (tid == 0 && c < nu) ez[c] = sbad ? kNotFinite : e;
  e = scale_exp(e);
  const int r = c % kTileN;
  for (int gr = tid; gr < 2 * kbu; gr += 64) {
    const int kb = gr / 2, kh = gr % 2;
    long long re[8], im[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = gr * 8 + j;
      double2 z = make_double2(0.0, 0.0);
      int ej = 0;
      if (c < nu && k <= c && !sbad) {
        z = Z[(int64_t)c * nu + k];
        ej = e - col_exp(hc, k);
      }
      re[j] = fixed55(z.x, ej);
      im[j] = fixed55(z.y, ej);
    }
    unsigned char* bp = b + ((size_t)kb * ntu + c / kTileN) * kBBytes + (r / 8) * 256 + kh * 128 + (r % 8) * 16;
    uint4 d[kDigits];
    auto put_b = [&](int w, int h) {
#pragma unroll
      for (int s = 0; s < kDigits; ++s)
        *reinterpret_cast<uint4*>(bp + w * kBHalf + s * 2048 + h * 1024) = d[s];
    };
    digits8(re, d, false);
    put_b(0, 0);
    put_b(1, 1);
    digits8(im, d, false);
    put_b(0, 1);
    digits8(im, d, true);
    put_b(1, 0);
  }
}

// Digit planes of the columns of X with the rows [0, n) as K: b[kb][tile of 32 columns]
// {[digit][re | im], [digit][-im | re]} for a plain product, {.., [digit][im | -re]} (kConj) for
// one with a conjugated left operand. A thread per column and 8 rows.
template <bool kConj>
__global__ void __launch_bounds__(128)
split_rhs_kernel(const double2* __restrict__ X, int64_t ldx, int64_t n, int nu, int kbn, int ntu,
                 const unsigned* __restrict__ hc, unsigned char* __restrict__ b) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t gr = t % (2 * kbn);
  const int c = (int)(t / (2 * kbn));
  if (c >= ntu * kTileN) return;
  long long re[8], im[8];
  const int e = c < nu ? col_exp(hc, c) : 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int64_t i = gr * 8 + j;
    const double2 v = (c < nu && i < n) ? X[(int64_t)c * ldx + i] : make_double2(0.0, 0.0);
    re[j] = fixed55(v.x, e);
    im[j] = fixed55(v.y, e);
  }
  const int r = c % kTileN;
  unsigned char* bp = b + ((size_t)(gr / 2) * ntu + c / kTileN) * kBBytes + (r / 8) * 256 + (gr % 2) * 128 + (r % 8) * 16;
  uint4 d[kDigits];
  auto put_b = [&](int w, int h) {
#pragma unroll
    for (int s = 0; s < kDigits; ++s)
      *reinterpret_cast<uint4*>(bp + w * kBHalf + s * 2048 + h * 1024) = d[s];
  };
  digits8(re, d, false);
  put_b(0, 0);
  if (!kConj) put_b(1, 1);
  digits8(im, d, false);
  put_b(0, 1);
  if (kConj) put_b(1, 0);
  digits8(kConj ? re : im, d, true);
  put_b(1, kConj ? 1 : 0);
}

struct GemmArgs {
  const unsigned char *a, *b;
  int64_t ta, tb;      // tiles per K-block of a and b
  int64_t mtn;         // batch: row tiles of one matrix (ta / mtn matrices)
  bool add;            // batch: add to out
  int nu;
  int64_t n, ldv;
  int kb_total, parts; // Gram: K-blocks and row ranges
  const int *ea, *eb;  // exponents of the output's rows and columns (Gram, and the columns of a
                       // batch: largest high words)
  double2* out;        // Gram partial sums, V, or the products of a batch
  int* status;
  const int *gate, *skip;
  uint32_t wait_limit;   // polls of a pipeline wait
};

struct GemmSmem {
  static constexpr uint32_t a = 0, b = kStagesG * kABytes, bar = b + kStagesG * kBBytes,
                            misc = bar + 10 * 8, total = misc + 16;
};

__device__ __forceinline__ bool wait_flag(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          const GemmArgs& p) {
  for (uint32_t it = 0; it < p.wait_limit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (it > 64) __nanosleep(64);
  }
  atomicOr(p.status, kStatusTimeout);
  *abort_flag = 1;
  return false;
}

// One output tile: its row tile, column tile and K-blocks.
struct Tile {
  int64_t ta;
  int tb, kb0, kb1;
};

// Tile i of this block (false: no more).
enum { kGramSum = 0, kTriangle = 1, kBatch = 2, kCross = 3 };

// Gram: one tile per block, the upper ones only, counted along b within a; blockIdx.y the row
// range. Cross: likewise, all tiles. Products: whole rows of tiles per block (the row tile's planes stay in L2), widest
// first; the rows left over after the last full round are dealt tile by tile.
template <int kMode>
__device__ __forceinline__ bool tile_of(const GemmArgs& p, int i, Tile& t) {
  const int nt = (int)p.tb;
  if (kMode == kCross) {
    if (i > 0) return false;
    t.ta = blockIdx.x % p.ta;
    t.tb = (int)(blockIdx.x / p.ta);
    t.kb0 = (int)((int64_t)p.kb_total * blockIdx.y / p.parts);
    t.kb1 = (int)((int64_t)p.kb_total * (blockIdx.y + 1) / p.parts);
    return true;
  }
  if (kMode == kGramSum) {
    if (i > 0) return false;
    int rest = blockIdx.x, at = 0;
    while (rest >= nt - at * (kTileM / kTileN)) {
      rest -= nt - at * (kTileM / kTileN);
      ++at;
    }
    t.ta = at;
    t.tb = at * (kTileM / kTileN) + rest;
    t.kb0 = (int)((int64_t)p.kb_total * blockIdx.y / p.parts);
    t.kb1 = (int)((int64_t)p.kb_total * (blockIdx.y + 1) / p.parts);
    return true;
  }
  const int64_t rounds = p.ta / gridDim.x, left = p.ta - rounds * gridDim.x;
  if (i < rounds * nt) {
    t.ta = (int64_t)(i / nt) * gridDim.x + blockIdx.x;
    t.tb = nt - 1 - i % nt;
  } else {
    const int64_t w = (int64_t)(i - rounds * nt) * gridDim.x + blockIdx.x;
    if (w >= left * nt) return false;
    t.ta = rounds * gridDim.x + w % left;
    t.tb = nt - 1 - (int)(w / left);
  }
  t.kb0 = 0;
  t.kb1 = kMode == kTriangle ? min(p.kb_total, (t.tb + 1) * (kTileN / 16)) : p.kb_total;
  return true;
}

// kGramSum: out[part][b nu + a] = sum of the rows of part blockIdx.y, with [re | im] and
// [im | -re] for conj(V)^T V. kTriangle: V[i][c] = sum_k V[i][k] Z[k][c], with [re | im] and
// [-im | re]; the K-blocks of the upper triangle only. kBatch: out_s (+)= A_s X likewise, all
// K-blocks, the row tiles of the matrices one after the other. kCross: as kGramSum with another
// right operand, out[part][c n + a], a < n, c < nu.
template <int kMode>
__global__ void __launch_bounds__(kThreadsG, 1) split_gemm_kernel(GemmArgs p) {
  if (skipped(p.gate, p.skip)) return;
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + GemmSmem::bar);
  uint64_t* full = bars;         // [2] a stage's copies landed
  uint64_t* empty = bars + 2;    // [2] the MMAs are done with it
  uint64_t* accfull = bars + 4;  // [2] the accumulators d < 4, d >= 4 hold a finished chunk
  uint64_t* accfree = bars + 6;  // [2] they have been read
  uint64_t* drained = bars + 8;  // every MMA is done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + GemmSmem::misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + GemmSmem::misc + 4);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStagesG; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int g = 0; g < 2; ++g) {
      mbar_init(&accfull[g], 1);
      mbar_init(&accfree[g], 32 * kFlushWarps);
    }
    mbar_init(drained, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  Tile t;
  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;   // K-blocks over all tiles
      bool ok = true;
      for (int i = 0; ok && tile_of<kMode>(p, i, t); ++i)
        for (int kb = t.kb0; kb < t.kb1; ++kb, ++issued) {
          const int s = issued % kStagesG;
          ok = wait_flag(&empty[s], ((issued / kStagesG) & 1) ^ 1, abort_flag, p);
          if (!ok) break;
          mbar_arrive_expect_tx(&full[s], kABytes + kBBytes);
          bulk_g2s(smem + GemmSmem::a + s * kABytes, p.a + ((size_t)kb * p.ta + t.ta) * kABytes,
                   kABytes, &full[s]);
          bulk_g2s(smem + GemmSmem::b + s * kBBytes, p.b + ((size_t)kb * p.tb + t.tb) * kBBytes,
                   kBBytes, &full[s]);
        }
      // no copy may be in flight when the block leaves, also if the others gave up without it
      for (int it = max(0, issued - kStagesG); it < issued; ++it)
        mbar_wait(&full[it % kStagesG], (it / kStagesG) & 1, kDrainWait);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int it = 0;               // K-blocks over all tiles
      int done[2] = {0, 0};     // chunks of the two groups handed over
      bool ok = true;
      for (int i = 0; ok && tile_of<kMode>(p, i, t); ++i)
        for (int kb = t.kb0; ok && kb < t.kb1; ++kb, ++it) {
          const int s = it % kStagesG, at = kb - t.kb0;
          const bool end = kb + 1 == t.kb1;
          bool fresh[2], last[2];
          for (int g = 0; g < 2; ++g) {   // group 0: d < 4, every second flush
            const int every = g ? kFlush : 2 * kFlush;
            fresh[g] = at % every == 0;
            last[g] = end || at % every == every - 1;
          }
          ok = wait_flag(&full[s], (it / kStagesG) & 1, abort_flag, p);
          for (int g = 0; ok && g < 2; ++g)
            if (fresh[g] && done[g] > 0) ok = wait_flag(&accfree[g], (done[g] - 1) & 1, abort_flag, p);
          if (!ok) break;
          tc_fence_after();
          const uint32_t ab = smem_u32(smem + GemmSmem::a + s * kABytes);
          const uint32_t bb = smem_u32(smem + GemmSmem::b + s * kBBytes);
          // left digit q against the digits t0 .. t0 + count - 1, into the accumulators q + t
          auto mma = [&](int q, int part, int t0, int count, bool accumulate) {
            mma_bf16(tmem + (q + t0) * 64, smem_desc(ab + (2 * q + part) * 4096, 128, 256),
                     smem_desc(bb + part * kBHalf + t0 * 2048, 128, 256),
                     idesc_bf16(kTileM, 64 * count), accumulate ? 1u : 0u);
          };
#pragma unroll
          for (int q = 0; q < kDigits; ++q)
#pragma unroll
            for (int part = 0; part < 2; ++part) {
              const int tn = min(kDigits, kOrders - q);   // digits t of this q
              mma(q, part, 0, min(4, tn), !(q + part == 0 && fresh[0]));
              if (q == 1 && part == 0 && fresh[1]) {   // d = 7 is met here first
                mma(q, part, 4, 2, true);
                mma(q, part, 6, 1, false);
              } else if (tn > 4) {
                mma(q, part, 4, tn - 4, !(q + part == 0 && fresh[1]));
              }
            }
          mma_commit(&empty[s]);
          for (int g = 0; g < 2; ++g)
            if (last[g]) {
              mma_commit(&accfull[g]);
              ++done[g];
            }
        }
      mma_commit(drained);   // also after an abort: arrives once every MMA issued is done
    }
  } else {
    // flush warps: lanes of TMEM quarter warp % 4, 32 of the 64 columns: side 0 the real
    // parts, side 1 the imaginary ones
    const int quarter = warp % 4, side = (warp - 2) / 4;
    const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + side * 32;
    int done[2] = {0, 0};
    bool ok = true;
    for (int i = 0; ok && tile_of<kMode>(p, i, t); ++i) {
      const int nkb = t.kb1 - t.kb0;
      long long hi[32], lo[32];   // sums of d < 4 and d >= 4
#pragma unroll
      for (int k = 0; k < 32; ++k) hi[k] = lo[k] = 0;
      for (int at = kFlush; ok && at - kFlush < nkb; at += kFlush) {   // chunks end at K-block at
#pragma unroll
        for (int g = 1; g >= 0; --g) {
          if (g == 0 && at % (2 * kFlush) != 0 && at < nkb) continue;
          if (ok) ok = __all_sync(0xffffffffu, wait_flag(&accfull[g], done[g] & 1, abort_flag, p));
          if (!ok) continue;
          tc_fence_after();
#pragma unroll
          for (int d4 = 0; d4 < 4; ++d4) {
#pragma unroll
            for (int half = 0; half < 32; half += 16) {
              float v[16];
              tmem_ld16(base + (4 * g + d4) * 64 + half, v);
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                const long long x = (long long)__float2int_rn(v[k]) * (1 << (8 * (3 - d4)));
                if (g == 0) hi[half + k] += x;
                else lo[half + k] += x;
              }
            }
          }
          tc_fence_before();
          mbar_arrive(&accfree[g]);
          ++done[g];
        }
      }
      if (!ok) break;
      // value = (hi 2^32 + lo) 2^(ea + eb - 70)
      const int64_t slot = kMode == kBatch ? t.ta / p.mtn : 0;
      const int64_t row = (t.ta - slot * p.mtn) * kTileM + quarter * 32 + lane;
      const int64_t rows = kMode == kGramSum ? p.nu : p.n;
      int er = row < rows ? p.ea[slot * p.n + row] : 0;
      if (kMode == kGramSum || kMode == kCross) er = exponent_of((unsigned)er);
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        const int col = t.tb * kTileN + k;
        if (row >= rows || col >= p.nu) continue;
        const int ec = kMode == kTriangle ? p.eb[col] : exponent_of((unsigned)p.eb[col]);
        const int e = scale_exp(er) + scale_exp(ec) - 70;
        double v = fma((double)hi[k], 4294967296.0, (double)lo[k]);
        v = e > -1022 && e < 1023 ? v * __longlong_as_double((long long)(e + 1023) << 52) : ldexp(v, e);
        if (er == kNotFinite || ec == kNotFinite) v = NAN;
        double* o = reinterpret_cast<double*>(
            kMode == kGramSum || kMode == kCross ? p.out + ((int64_t)blockIdx.y * p.nu + col) * rows + row
                              : p.out + (slot * p.nu + col) * p.ldv + row);
        o[side] = kMode == kBatch && p.add ? o[side] + v : v;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    if (lane == 0) mbar_wait(drained, 0, kDrainWait);   // before the accumulators are released
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

bem_status set_gemm_smem(bem_ctx* ctx) {
  for (const void* f : {(const void*)split_gemm_kernel<kGramSum>, (const void*)split_gemm_kernel<kTriangle>,
                        (const void*)split_gemm_kernel<kBatch>, (const void*)split_gemm_kernel<kCross>}) {
    const bem_status st = cuda_check(
        ctx, cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GemmSmem::total),
        "split product attribute");
    if (st != BEM_OK) return st;
  }
  return BEM_OK;
}

}  // namespace

int split64_parts(const bem_ctx* ctx, int64_t n, int nu) {
  int sms = 0, tiles = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  const int ntu = (nu + kTileN - 1) / kTileN;
  for (int a = 0; a * kTileM < nu; ++a) tiles += ntu - a * (kTileM / kTileN);
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 15) / 16 / kFlush, std::max(1, sms) / tiles));
}

namespace {

struct SplitSizes {
  size_t a, b, total;   // the operands' planes, all with the scales
};

// The split products' workspace for n x nu (total 0: the FP64 kernels).
SplitSizes split_sizes(const bem_ctx* ctx, int64_t n, int nu) {
  SplitSizes z{};
  if (n * (int64_t)nu * nu < kMinWork) return z;
  const size_t kbn = (size_t)(n + 15) / 16, kbu = (size_t)(nu + 15) / 16;
  const size_t mtu = (nu + kTileM - 1) / kTileM, ntu = (nu + kTileN - 1) / kTileN;
  const size_t mtn = (size_t)(n + kTileM - 1) / kTileM;
  if ((int64_t)kbn / split64_parts(ctx, n, nu) / kFlush > 2000) return z;   // the 64-bit sums' range
  auto up = [](size_t b) { return (b + 1023) / 1024 * 1024; };
  z.a = up(std::max(kbn * mtu, kbu * mtn) * kABytes);
  z.b = up(std::max(kbn * ntu, kbu * ntu) * kBBytes);
  const size_t total = z.a + z.b + up((size_t)(2 * nu + n) * sizeof(int));
  if (total <= kMaxSplitBytes) z.total = total;
  return z;
}

}  // namespace

size_t split64_bytes(const bem_ctx* ctx, int64_t n, int nu) { return split_sizes(ctx, n, nu).total; }

void split64_plan(bem_ctx* ctx, int64_t ldv, int64_t n, int nu, void* mem, Split64& sp) {
  sp = Split64();
  const SplitSizes z = split_sizes(ctx, n, nu);
  if (z.total == 0) return;
  sp.n = n;
  sp.ldv = ldv;
  sp.nu = nu;
  sp.kbn = (int)((n + 15) / 16);
  sp.kbu = (nu + 15) / 16;
  sp.mtu = (nu + kTileM - 1) / kTileM;
  sp.ntu = (nu + kTileN - 1) / kTileN;
  sp.mtn = (n + kTileM - 1) / kTileM;
  sp.parts = split64_parts(ctx, n, nu);
  unsigned char* base = static_cast<unsigned char*>(mem);
  sp.a = base;
  sp.b = base + z.a;
  sp.hcol = reinterpret_cast<unsigned*>(base + z.a + z.b);
  sp.ez = reinterpret_cast<int*>(sp.hcol + nu);
  sp.erow = sp.ez + nu;
  sp.use = set_gemm_smem(ctx) == BEM_OK;
}

namespace {

bem_status column_maxima(bem_ctx* ctx, unsigned* hcol, const double2* V, int64_t ldv, int64_t n,
                         int nu, const int* gate, const int* skip, cudaStream_t s) {
  const bem_status st = cuda_check(ctx, cudaMemsetAsync(hcol, 0, nu * sizeof(int), s), "split scales");
  if (st != BEM_OK) return st;
  const unsigned ys = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 2047) / 2048, 64));
  split_colmax_kernel<<<dim3((unsigned)nu, ys), 256, 0, s>>>(V, ldv, n, hcol, gate, skip);
  ctx->launches++;
  return BEM_OK;
}

}  // namespace

bem_status split64_gram(bem_ctx* ctx, const Split64& sp, const double2* V, double2* part,
                        const int* gate, cudaStream_t s) {
  bem_status st = column_maxima(ctx, sp.hcol, V, sp.ldv, sp.n, sp.nu, gate, nullptr, s);
  if (st != BEM_OK) return st;
  const int64_t threads = 2 * (int64_t)sp.kbn * sp.mtu * kTileM;
  split_columns_kernel<<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(
      V, sp.ldv, sp.n, sp.nu, sp.kbn, sp.mtu, sp.ntu, sp.hcol, sp.a, sp.b, gate);
  int tiles = 0;
  for (int a = 0; a < sp.mtu; ++a) tiles += sp.ntu - a * (kTileM / kTileN);
  GemmArgs g{sp.a, sp.b, sp.mtu, sp.ntu, 0, false, sp.nu, sp.n, sp.ldv, sp.kbn, sp.parts,
             reinterpret_cast<const int*>(sp.hcol), reinterpret_cast<const int*>(sp.hcol), part, ctx->d_status, gate, nullptr, ctx->stage_wait_limit};
  split_gemm_kernel<kGramSum><<<dim3((unsigned)tiles, (unsigned)sp.parts), kThreadsG, GemmSmem::total, s>>>(g);
  ctx->launches += 2;
  return cuda_check(ctx, cudaGetLastError(), "split Gram matrix");
}

bem_status split64_multiply(bem_ctx* ctx, const Split64& sp, bool same, double2* V,
                            const double2* Z, const int* gate, const int* skip, cudaStream_t s) {
  if (!same) {
    const bem_status st = column_maxima(ctx, sp.hcol, V, sp.ldv, sp.n, sp.nu, gate, skip, s);
    if (st != BEM_OK) return st;
  }
  split_rows_kernel<<<(unsigned)(sp.mtn * (kTileM / 32)), 256, 0, s>>>(
      V, sp.ldv, 0, sp.n, sp.nu, sp.kbu, sp.mtn, sp.hcol, sp.erow, sp.a, gate, skip);
  split_factor_kernel<<<(unsigned)(sp.ntu * kTileN), 64, 0, s>>>(Z, sp.nu, sp.kbu, sp.ntu, sp.hcol,
                                                                sp.ez, sp.b, gate, skip);
  GemmArgs g{sp.a, sp.b, sp.mtn, sp.ntu, sp.mtn, false, sp.nu, sp.n, sp.ldv, sp.kbu, 1, sp.erow, sp.ez, V,
             ctx->d_status, gate, skip, ctx->stage_wait_limit};
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  const unsigned grid = (unsigned)std::min<int64_t>(std::max(1, sms), sp.mtn * sp.ntu);
  split_gemm_kernel<kTriangle><<<grid, kThreadsG, GemmSmem::total, s>>>(g);
  ctx->launches += 3;
  return cuda_check(ctx, cudaGetLastError(), "split product");
}

SplitBatch split64_batch_plan(int64_t n, int kc, int S, int ncols) {
  SplitBatch b;
  b.n = n;
  b.S = S;
  b.nu = ncols;
  b.kc = kc;
  b.mtn = (n + kTileM - 1) / kTileM;
  b.ntu = (ncols + kTileN - 1) / kTileN;
  const size_t kb = (size_t)(kc + 15) / 16;
  auto up = [](size_t x) { return (x + 1023) / 1024 * 1024; };
  b.b_off = up(kb * S * (size_t)b.mtn * kABytes);
  b.e_off = b.b_off + up(kb * b.ntu * kBBytes);
  b.bytes = b.e_off + up(((size_t)ncols + (size_t)S * n) * sizeof(int));
  return b;
}

bem_status split64_batch_scales(bem_ctx* ctx, const SplitBatch& b, char* work, const double2* X,
                                int64_t ldx, cudaStream_t s) {
  const bem_status st = set_gemm_smem(ctx);
  if (st != BEM_OK) return st;
  return column_maxima(ctx, reinterpret_cast<unsigned*>(work + b.e_off), X, ldx, b.n, b.nu, nullptr, nullptr, s);
}

bem_status split64_batch(bem_ctx* ctx, const SplitBatch& b, char* work, const double2* A,
                         int64_t astep, int kc, const double2* X, int64_t ldx, bool add,
                         double2* out, cudaStream_t s) {
  unsigned char* ap = reinterpret_cast<unsigned char*>(work);
  unsigned char* bp = ap + b.b_off;
  unsigned* hcol = reinterpret_cast<unsigned*>(work + b.e_off);
  int* er = reinterpret_cast<int*>(hcol + b.nu);
  const int kb = (kc + 15) / 16;
  split_rows_kernel<<<dim3((unsigned)(b.mtn * (kTileM / 32)), (unsigned)b.S), 256, 0, s>>>(
      A, b.n, astep, b.n, kc, kb, b.mtn, nullptr, er, ap, nullptr, nullptr);
  const int64_t threads = 2 * (int64_t)kb * b.ntu * kTileN;
  split_rhs_kernel<false><<<(unsigned)((threads + 127) / 128), 128, 0, s>>>(X, ldx, kc, b.nu, kb, b.ntu, hcol, bp);
  GemmArgs g{ap, bp, b.S * b.mtn, b.ntu, b.mtn, add, b.nu, b.n, b.n, kb, 1, er,
             reinterpret_cast<const int*>(hcol), out, ctx->d_status, nullptr, nullptr, ctx->stage_wait_limit};
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  const unsigned grid = (unsigned)std::min<int64_t>(std::max(1, sms), g.ta * g.tb);
  split_gemm_kernel<kBatch><<<grid, kThreadsG, GemmSmem::total, s>>>(g);
  ctx->launches += 3;
  return cuda_check(ctx, cudaGetLastError(), "split products");
}

namespace {

// C_j = scale_j * sum of the partial products of its columns.
__global__ void __launch_bounds__(256)
split_cross_sum_kernel(const double2* __restrict__ part, int parts, int64_t block, int64_t count,
                       const double2* __restrict__ scale, double2* __restrict__ C) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= count) return;
  double2 v = part[t];
  for (int r = 1; r < parts; ++r) {
    const double2 u = part[r * count + t];
    v.x += u.x;
    v.y += u.y;
  }
  if (scale) {
    const double2 s = scale[t / block];
    v = make_double2(s.x * v.x - s.y * v.y, s.x * v.y + s.y * v.x);
  }
  C[t] = v;
}

}  // namespace

SplitCross split64_cross_plan(const bem_ctx* ctx, int64_t n, int p, int q, int nb) {
  SplitCross c;
  const int64_t cols = (int64_t)q * nb;
  if (n * p * cols < kMinCross || cols > INT_MAX / 2) return c;
  c.n = n;
  c.p = p;
  c.q = q;
  c.nb = nb;
  c.mtp = (p + kTileM - 1) / kTileM;
  c.nt = (int)((cols + kTileN - 1) / kTileN);
  const int64_t kb = (n + 15) / 16;
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  c.parts = (int)std::max<int64_t>(1, std::min<int64_t>(kb / (2 * kFlush), std::max(1, sms) / (c.mtp * c.nt)));
  if (kb / c.parts / kFlush > 2000) return c;   // the 64-bit sums' range
  auto up = [](size_t x) { return (x + 1023) / 1024 * 1024; };
  c.b_off = up((size_t)kb * c.mtp * kABytes);
  c.part_off = c.b_off + up((size_t)kb * c.nt * kBBytes);
  c.h_off = c.part_off + up((size_t)c.parts * p * cols * sizeof(double2));
  c.bytes = c.h_off + up(((size_t)p + cols) * sizeof(unsigned));
  c.use = c.bytes <= kMaxSplitBytes;
  return c;
}

bem_status split64_cross(bem_ctx* ctx, const SplitCross& c, void* work, const double2* X,
                         int64_t ldx, const double2* Y, const double2* scale, double2* C,
                         cudaStream_t s) {
  unsigned char* ap = static_cast<unsigned char*>(work);
  unsigned char* bp = ap + c.b_off;
  double2* part = reinterpret_cast<double2*>(ap + c.part_off);
  unsigned* hx = reinterpret_cast<unsigned*>(ap + c.h_off);
  unsigned* hy = hx + c.p;
  const int cols = c.q * c.nb, kb = (int)((c.n + 15) / 16);
  bem_status st = set_gemm_smem(ctx);
  if (st == BEM_OK) st = column_maxima(ctx, hx, X, ldx, c.n, c.p, nullptr, nullptr, s);
  if (st == BEM_OK) st = column_maxima(ctx, hy, Y, c.n, c.n, cols, nullptr, nullptr, s);
  if (st != BEM_OK) return st;
  const int64_t tx = 2 * (int64_t)kb * c.mtp * kTileM, ty = 2 * (int64_t)kb * c.nt * kTileN;
  split_columns_kernel<<<(unsigned)((tx + 127) / 128), 128, 0, s>>>(X, ldx, c.n, c.p, kb, c.mtp, 0, hx, ap,
                                                                   nullptr, nullptr);
  split_rhs_kernel<true><<<(unsigned)((ty + 127) / 128), 128, 0, s>>>(Y, c.n, c.n, cols, kb, c.nt, hy, bp);
  GemmArgs g{ap, bp, c.mtp, c.nt, c.mtp, false, cols, c.p, c.p, kb, c.parts,
             reinterpret_cast<const int*>(hx), reinterpret_cast<const int*>(hy), part, ctx->d_status,
             nullptr, nullptr, ctx->stage_wait_limit};
  split_gemm_kernel<kCross><<<dim3((unsigned)(c.mtp * c.nt), (unsigned)c.parts), kThreadsG, GemmSmem::total, s>>>(g);
  const int64_t count = (int64_t)c.p * cols;
  split_cross_sum_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(
      part, c.parts, (int64_t)c.p * c.q, count, scale, C);
  ctx->launches += 4;
  return cuda_check(ctx, cudaGetLastError(), "split projection");
}

}  // namespace bem
