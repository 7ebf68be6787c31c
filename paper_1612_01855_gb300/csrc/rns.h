// FP64-class matrix products on the BF16 tensor cores in a residue number
// system: the products of the sliced schedule of the FP64 solve and the
// residual of the mixed-precision solve.
//
// Method (K. Ozaki, Y. Uchino, T. Imamura, "Ozaki Scheme II: a GEMM-oriented
// emulation of floating-point matrix multiplication using an integer modular
// technique", 2025), restated for this hardware:
//   * every row of A and of B^T is cut along K into chunks of at most 2048
//     values; a (row, chunk) gets a power-of-two exponent e with max|a| <
//     2^e, and its values become integers round(a 2^(bits - e)), |.| <=
//     2^bits;
//   * the integers' residues modulo kModuli pairwise coprime moduli p <= 179
//     (symmetric: at most 90 in absolute value) are stored as bf16, exact;
//   * one bf16 tensor-core product per modulus sums residue products over a
//     chunk: at most 2048 * 90 * 90 = 16,588,800 < 2^24, exact in FP32;
//   * reduced modulo p again, the sums are the residues of the integer
//     product, whose absolute value is at most 2^(11 + bitsA + bitsB), below
//     half the product M of the moduli: the Chinese remainder theorem gives
//     it back, and it is scaled and applied in FP64.
// The errors are the roundings of the factors to `bits` bits, the integer
// product's to 3.2 M 2^-64 at most (about 2^-49 of the product of the two
// maxima, to either side alike) and the final FP64 operations.  Short factors,
// nine 6-bit digits a pair from their maxima down (24 and 30 bits, say, or
// integers below 2^24 both), are not rounded and give the double next to their
// product: integer and dyadic systems keep their exact results.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace trsm {

constexpr int kModuli = 15;
constexpr int kChunk = 2048;   // longest K range summed exactly in FP32 (the default chunk)
constexpr int kBitsFull = 48;  // integer bits of the plan's operands and of an eight-plane product

// Residue planes of a rows x K operand, in blocks of 64 values along K: block
// (m, q) holds the residues modulo the m-th modulus of k = 64 q .. 64 q + 63
// of every row, row after row (128 bytes each), so that a 128-row tile's step
// of 64 along K is one contiguous 16 KB read.  (With whole rows contiguous a
// tile read 128 bytes of each of 128 rows 2 K bytes apart, and the products
// that stream A from HBM ran at 4.4 TB/s.)  Values past K are zeros.  One
// int16 exponent per (row, chunk of kc along K); kc is at most kChunk and a
// multiple of 64 when there is more than one chunk (a step of 64 must not
// straddle two exponents).
//
// A triangular operand (tri; K = rows, the plan's factors) keeps of chunk c
// only the rows from c kc on, chunk after chunk, each chunk laid out as above
// on its own: rns_chunk gives one as an operand of K = kc.
struct RnsOperand {
  __nv_bfloat16* res = nullptr;  // [kModuli][kb][rows][64]
  int16_t* ex = nullptr;         // exponent of (row, chunk) at ex[row ex_ld + chunk]
  int8_t* zeros = nullptr;       // in the same places: 6-bit digits (0 to 7) that end all its integers in zeros
  int* zmax = nullptr;           // at least the largest of them; zero before the first residues are made
  int64_t rows = 0, K = 0, kb = 0, nch = 0, kc = kChunk, ex_ld = 0;  // kb: blocks of 64 along K
  bool tri = false;
};

size_t rns_operand_bytes(int64_t rows, int64_t K, int64_t kc = kChunk, bool tri = false);
RnsOperand rns_operand_view(void* base, int64_t rows, int64_t K, int64_t kc = kChunk, bool tri = false);
RnsOperand rns_chunk(const RnsOperand& o, int64_t c);

// How many of the moduli, and how many integer bits of the right factor, a
// product of the accuracy class of P 6-bit digits takes (P = 5 .. 8; the
// left factor, the plan's, always has kBitsFull bits).  M / 2 has to exceed
// 2^(11 + 48 + bits): 13, 14 and 15 moduli make 2^83.5, 2^90.6 and 2^97.6 of
// 2^(bitsA + bitsB): six digits are one bit too many for 13 moduli.
struct RnsClass {
  int moduli, bits;
};
inline RnsClass rns_class(int planes) {
  return planes <= 5 ? RnsClass{13, 35} : planes <= 7 ? RnsClass{14, 42} : RnsClass{15, kBitsFull};
}

// Residues of `rows` rows of FP64 values (row r contiguous from src + r ld)
// in the given class; only the first K (<= o.K) values of each row are read,
// the rest are zeros (K < o.K needs a single chunk).
cudaError_t rns_rows(const double* src, int64_t ld, int64_t K, const RnsOperand& o, RnsClass c, cudaStream_t s);

// Residues of the rows of the strictly lower triangle of a column-major
// n x n L (through a row-major copy in tmp_rowmajor, n*n doubles); o is
// triangular.
cudaError_t rns_lower_rows(const double* L, int64_t ldl, int64_t n, const RnsOperand& o, double* tmp_rowmajor,
                           cudaStream_t s);

// The two operands of the sliced schedule, from a plan's L~ (column-major,
// ldt; diagonal blocks of order n0 hold the inverses):
//   off: the rows of L~ with every diagonal block (and the upper triangle)
//        zeroed, rows n x K n, triangular, chunks of n0 (one exponent per
//        row and block column), for the trailing updates;
//   inv: row r holds the inverted diagonal block's row below its diagonal,
//        L~(r, b n0 + c) for c < r - b n0 with b = r / n0 (zeros elsewhere),
//        rows n x K n0, one chunk, for the diagonal multiplies; the diagonal
//        L~(r, r) goes to diag (n doubles) and is applied in FP64.
// tmp_rowmajor holds n*n doubles of scratch.
cudaError_t rns_offdiag_block_rows(const double* Lt, int64_t ldt, int64_t n, int64_t n0, const RnsOperand& off,
                                   double* tmp_rowmajor, cudaStream_t s);
cudaError_t rns_inverse_block_rows(const double* Lt, int64_t ldt, int64_t n, int64_t n0, const RnsOperand& inv,
                                   double* diag, double* tmp_rowmajor, cudaStream_t s);

// One product P(r, c) = sum_{t < K} A(a_row0 + r, a_k0 + t) B(c, b_k0 + t),
// r < M, c < N, applied in FP64 to Y(r, c) = Y[c * ldy + r]:
//   kRnsDiag     Y = dg[r] S(r, c) + P       (the diagonal multiply)
//   kRnsUpdate   Y = S - P                   (S may be Y)
//   kRnsResidual Y = S - dg[r] X(r, c) - P
// [a_k0, a_k0 + K) and [b_k0, b_k0 + K) each lie in one chunk and start at a
// multiple of 64.  lower:
// A(a_row0 + r, a_k0 + t) = 0 for t > r (the sums of row tile q stop at
// 128 (q + 1)).
enum RnsMode { kRnsDiag = 0, kRnsUpdate = 1, kRnsResidual = 2 };
struct RnsProduct {
  RnsOperand A, B;
  int64_t a_row0 = 0, a_k0 = 0, b_row0 = 0, b_k0 = 0;
  int64_t M = 0, N = 0, K = 0;
  RnsClass cls{kModuli, kBitsFull};  // of B
  bool lower = false;
  int mode = kRnsUpdate;
  double* Y = nullptr;
  int64_t ldy = 0;
  const double* S = nullptr;
  int64_t lds = 0;
  const double* dg = nullptr;
  const double* X = nullptr;
  int64_t ldx = 0;
};

// Scratch of the products of at most M rows and exactly N columns: control
// words and the residues of the sums.  The control words must be zero before
// the first product (rns_scratch_clear); every product leaves them zero (zmax
// as it is).
// Products that may overlap need scratch of their own.
struct RnsScratch {
  int* ctrl = nullptr;
  int* zmax = nullptr;  // a word for the zmax of an operand made again and again; rns_scratch_clear zeroes it
  void* resid = nullptr;
  int64_t tiles = 0;  // output tiles it holds
};
size_t rns_scratch_bytes(int64_t M, int64_t N);
RnsScratch rns_scratch_view(void* base, int64_t M, int64_t N);
cudaError_t rns_scratch_clear(const RnsScratch& sc, cudaStream_t s);
cudaError_t rns_product(const RnsProduct& p, const RnsScratch& sc, int* err, cudaStream_t s);

// R = B - L X with the strictly lower part of L given by its residue rows
// (Ls: n x n), its diagonal as a vector, and X by its residue rows (Xs: k
// rows of length n, made in the class of `planes`) and by itself; R, B, X
// column-major n x k.  `planes` (5 to 8) sets the accuracy: X to 35, 42, 42
// or 48 bits of each (column, chunk) maximum.
cudaError_t rns_residual(const RnsOperand& Ls, const double* diag, const RnsOperand& Xs, const double* X, int64_t ldx,
                         const double* B, int64_t ldb, double* R, int64_t ldr, int planes, const RnsScratch& sc,
                         int* err, cudaStream_t s);

}  // namespace trsm
