// Double-precision products on the integer tensor cores.
//
// The FP64 pipe of an SM does 64 multiply-adds a clock, tcgen05.mma kind::i8 does 8192 exact ones.  Operands
// are fixed-point numbers: a row of A (or a column of B) is scaled by a power of two so that its largest
// entry is just below 1, rounded to 54 fractional bits and written as seven signed base-256 digits,
//   a = 2^Ea sum_i a_i 256^-(i+1) 2^2,   a_i in [-128, 127].
// The product of two digits is exact in int32 and so are the sums; digit products of equal weight,
// i + j = s, share an accumulator, s = 0 .. 6 are kept (28 digit products).  What is left out or rounded is
// below 2^-51 of (largest |a| of the row) (largest |b| of the column) per contraction step at worst and
// 2^-54 on the average, as the roundings of a double product whose terms are of that size.  Measured on
// random operands, rms error over sum |a||b|: 1.3e-17 at 256 steps and 1.1e-17 at 4096, the FP64 pipe
// 4.4e-17 and 7.6e-17.  The one thing a caller has to see to is that a small entry of a row that also has a
// large one keeps fewer digits: operands whose rows (A) and columns (B) are of one size, as triangular
// factors of an equilibrated matrix are, lose nothing.
// A row of A or a column of B with an entry that is no finite number (and that no mask takes out) makes all of that
// row or column of C no number.
// 170 TFLOP/s of double-precision products is what the issue rate allows at 1965 MHz (37 on the FP64 pipe).
#pragma once

#include "tb_gemm.cuh"
#include "tb_tma.cuh"

namespace tb {

// A matrix of digits: blocks of 64 rows x 32 contraction steps, [row block][k block][2 x 16 k][7 digits][64 rows][16 k].
// That order is, box by box, the shared-memory image of both operands (K-major, no swizzle), and one TMA box
// loads a block with all its digits.
enum { I8_DIGITS = 7, I8_RB = 64, I8_KB = 32, I8_BLOCK = I8_DIGITS * I8_RB * I8_KB };
// the longest contraction (16384 steps): the int32 sums hold 7 digit products of 2^14 a step
enum { I8_MAX_K_BLOCKS = 512 };
struct I8Mat {
  unsigned char* data;
  long long row_blocks;  // of the whole allocation (all matrices of a batch)
  int k_blocks;
};
inline size_t i8_bytes(long long row_blocks, int k_blocks) { return (size_t)row_blocks * k_blocks * I8_BLOCK; }

// Rounds the rows (k_contig: X(row, k) = X[row ld + k]) or the columns (X(row, k) = X[k ld + row]) of a matrix to
// digits, row blocks rb0 .. and k blocks kb0 .. of dst.  max_bits: per row the bit pattern of the largest
// magnitude (i8_row_max), or nullptr: every entry is below 2^fixed_exp.
// bad (with a fixed exponent): bad[max_batch matrix + row] becomes 1 where an entry is not below the bound (or is
// no number).  mask 1: entries with k > row are taken as zero; 2: entries with k < row; 3: entries with k <= row.
// k_exp: entries are multiplied by 2^(k_sign k_exp[k]) (one vector for all matrices), which takes out scales that
// the contraction steps of both operands have in opposite directions.
struct I8Src {
  const void* X;
  long long ld, batch;  // element strides
  int rows, K, n_batch;
  bool is_float, k_contig;
  int mask;
  const int* k_exp;  // or nullptr
  int k_sign;
};
// exps[k] = exponent of the diagonal entry U_kk of an upper factor: the scale of row k of U, column k of H^{-1/2}
tb_status i8_diag_exp(const float* U, int* exps, int d, cudaStream_t st);
tb_status i8_row_max(const I8Src& s, unsigned long long* max_bits, long long max_batch, cudaStream_t st);
tb_status i8_slice(const I8Src& s, const unsigned long long* max_bits, long long max_batch, int fixed_exp,
                   const I8Mat& dst, long long rb0, long long rb_batch, int kb0, cudaStream_t st, int* bad = nullptr);

// C = alpha A B^T + beta C over k blocks [0, k_blocks) of two digit matrices (alpha = 1 or -1, beta = 0 or 1).
struct I8Gemm {
  I8Mat A, B;
  long long a_rb, b_rb, a_rb_batch, b_rb_batch;  // first row block, and its step from one matrix of a batch to the next
  int a_kb, b_kb, k_blocks;
  const unsigned long long *a_max, *b_max;  // or nullptr: fixed exponents
  long long a_max_batch, b_max_batch;
  int a_exp, b_exp;
  double* C;
  float* Cf;  // instead of C: the result rounded to float (beta = 0)
  long long ldc, c_batch;
  int M, N, n_batch;
  double alpha, beta;
  // known zeros: 1: A(m, k) = 0 for k > m;  2: B(k, n) = 0 for k < n;  4: only tiles on or below the diagonal;
  // 8: B(k, n) = 0 for k > n;  16: A(m, k) = 0 for k < m
  int zeros;
  int tiles_per_cta;  // 0: as few CTAs as fill the SMs; else at most that many tiles per CTA
  int order;  // 0: tiles row by row; 1: columns ascending, slowest index; 2: rows descending, slowest index
};
inline I8Gemm i8_gemm_params() {
  I8Gemm g = {};
  g.n_batch = 1;
  g.alpha = 1.0;
  return g;
}
tb_status i8_gemm(const I8Gemm& g, cudaStream_t st);

}  // namespace tb
