// Float64 contractions on the tcgen05 tensor cores (internal header).
//
// GB300 runs float64 at ~1.2 TFLOP/s, so every dense contraction of the float64
// path is bound by that pipe.  Here an operand row is held as a fixed-point
// number of 57 bits relative to a power of two above its largest element,
//   x = 2^(e - 56) X,  X = sum_i v_i 2^(49 - 7 i),  i = 0 .. 7,
// |v_0| <= 128 and |v_i| <= 64: integers that BF16 holds exactly (the error-free
// splitting of K. Ozaki, T. Ogita, S. Oishi, S. M. Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59 (2012), with digits of a common
// exponent per row).  A product of two rows is then
//   sum_k a b = 2^(ea + eb - 63) sum_t D_t 2^(7 (7 - t)),
//   D_t = sum_{i + j = t} sum_k v_i w_j,
// each D_t an integer below 2^24 over kOzSegK values of k, so the FP32
// accumulators hold it exactly; the segments are added as 64-bit integers and
// the result is rounded to float64 once.
//
// What is lost, against the row maxima (2^(ea - 1) <= max |a| < 2^ea, or ea =
// -1021 in a row of subnormals): an element more than three binades below its
// row's largest is rounded to 2^(e - 57), the products with i + j > 7 are left out
// (7.1 2^-58 per term at most, of either sign), and so
//   |C - A B^T| <= 2^-53 |C| + 2.8 K 2^(ea + eb - 56),
// at most 1.4 K 2^-53 max |a| max |b| beside the rounding of C.  A float64 FMA
// chain's bound is K 2^-53 sum |a b|: the same kind where a sum is of the size of
// its largest elements' product, as in a step's, in which one operand's elements
// are of a size (the fields, Theta's and the orbitals' rows; orbitals against each
// other are made so by a power of two each, oz_row_exps).  A sum whose large
// elements meet only small ones loses what the chain would keep.  A row that holds
// an infinity or a NaN gives NaN.
#pragma once

#include "kernels.cuh"

namespace afq {

constexpr int kOzSlices = 8;
constexpr int kOzSegBlk = 25;             // K blocks of 16 between two drains of the accumulators
constexpr int kOzSegK = 16 * kOzSegBlk;   // 400: 40960 * 400 < 2^24 (D_7: 2 * 2^13 + 6 * 2^12 per k)
constexpr int kOzZeroExp = -30000;        // exponent of a row of zeros
constexpr int kOzNanExp = 100000;         // a row holding an infinity or a NaN: its results are NaN

// Slices of `rows` operand rows as the kernel's shared-memory tiles: row tile
// rt = r / rows_per_tile holds RT rows (a multiple of 8, >= rows_per_tile), K
// in blocks of 16.  Tile (rt, kb) is 8 slices x RT rows x 16 BF16, 256 bytes
// per 8 rows (two 8 x 8 core matrices); rows past rows_per_tile are not
// written (they only meet output rows or columns that are dropped).
struct OzOperand {
  void* data = nullptr;
  int* exps = nullptr;  // [tiles * rows_per_tile] row exponents e
  int RT = 128, rows_per_tile = 128;
  int nkb = 0;          // K blocks of 16
  long batch_stride = 0;      // bytes between the operands of a batch (0: shared)
  long batch_exp_stride = 0;  // row exponents between them
};
inline size_t oz_tiles(size_t rows, int rows_per_tile) { return (rows + rows_per_tile - 1) / rows_per_tile; }
inline size_t oz_bytes(size_t rows, int rows_per_tile, int RT, size_t k) {
  return oz_tiles(rows, rows_per_tile) * ((k + 15) / 16) * (size_t)kOzSlices * RT * 32;
}

// Rows of a row-major float64 matrix (pitch ld) into an operand.
int oz_slice_rows(const double* src, long rows, int k, long ld, const OzOperand& o, cudaStream_t st);
// Taylor operands of W walkers (see oz.cu): the rows of V / sqrt(dt) from the
// packed Y, and the term's rows.
int oz_slice_v(const double* Y, long ldy, int W, int M, int Mp, const OzOperand& o, cudaStream_t st);
int oz_slice_term(const double* t, int W, int N, int M, int Mp, const OzOperand& o, cudaStream_t st);

// C[m][n] = 2^alpha_log2 sum_k A[m][k] B[n][k] (float64, pitch ldc); rows of
// dead walkers (mask, mask_rows rows each) are not stored.  A batch of them
// with the operands' strides and C c_batch values apart.
struct OzGemm {
  int m = 0, n = 0, batch = 1;
  long c_batch = 0;
  OzOperand A, B;  // B: RT = 64
  double* C = nullptr;
  long ldc = 0;
  int alpha_log2 = 0;
  const double* mask = nullptr;
  int mask_rows = 1;
  int* err = nullptr;
};
int oz_gemm_store(const OzGemm& g, cudaStream_t st);

// One Taylor term of W walkers: tout = scale (V tin), acc (k == 1: tin) += tout.
struct OzTerm {
  int W = 0, M = 0, N = 0, k = 0;
  double scale = 0.0;  // sqrt(dt) / k
  bool last = false;  // tout is not needed
  OzOperand V, T;     // T: RT = oz_term_width(N)
  const double* tin = nullptr;
  double* tout = nullptr;
  double* acc = nullptr;
  int* err = nullptr;
};
int oz_term_width(int N);
int oz_taylor_term(const OzTerm& t, cudaStream_t st);

// Theta = Phi S^-1 of nds inverses per walker (see oz.cu for the operands):
// theta[ds][w][2][N][M]; rows p < N are the identity when unit.  A walker with
// weight 0 or without an inverse (log det -inf, at ld[w ld_w + ds ld_ds])
// keeps its rows, or gets zeros (zero_singular, live walkers only).
struct OzTheta {
  int W = 0, M = 0, N = 0, nds = 1;
  int w0 = 0, nw = 0;   // walkers [w0, w0 + nw) of the operands
  OzOperand A, B;
  double* theta = nullptr;
  const double* ld = nullptr;
  int ld_w = 2, ld_ds = 2;
  const double* wt = nullptr;
  const int* flag = nullptr;  // instead of ld: walkers with flag 0 keep their rows
  int unit = 0, zero_singular = 0;
  void* th_lo = nullptr;  // BF16/TF32 copy of the rows, pitch Mp
  int lo_kind = 0, Mp = 0;
  int* err = nullptr;
};
// Row exponents of n rows of M values, as oz_slice_rows gives them.  Those of the
// planes (w, c, i) of Phi scale the rows over the orbitals by a power of two per
// orbital (down in Phi, up in the inverse: exactly), so that a result does not
// depend on the orbitals' norms.
int oz_row_exps(const double* src, long n, int M, int* exps, cudaStream_t st);
// operand rows p = [Re Phi_p | Im Phi_p] (2 N values, N <= 64) of W walkers
int oz_slice_cols(const double* phi, int W, int N, int M, const int* planes, const OzOperand& o, cudaStream_t st);
// Operands of sum_k conj(Phi_k[p]) Th_k[q] over the rows k = (w, i) of nz
// groups of cw walkers from walker w0 on (the last may be short), a batch entry
// each, K = 2 N cw: A rows p = [Re Phi_p | Im Phi_p] and M + p =
// [-Im Phi_p | Re Phi_p] per walker (sums with [Re Th | Im Th]: the real and the
// imaginary part), B rows q of thA and M + q of thB, orbitals scaled as above
// (planes: room for 2 N exponents of nz cw walkers).
int oz_slice_densities(const double* phi, const double* thA, const double* thB, int W, int N, int M, int w0,
                       int nz, int cw, int* planes, const OzOperand& A, const OzOperand& B, cudaStream_t st);
// operand rows (re, j) = [Re S^-1_j | -Im S^-1_j], (im, j) = [Im | Re] of the
// inverses sinv[ds W + w0 + w], batch ds nw + w
int oz_slice_inverse(const double2* sinv, int W, int w0, int nw, int nds, int N, const int* planes,
                     const OzOperand& o, cudaStream_t st);
int oz_theta(const OzTheta& t, cudaStream_t st);

// gram[w][r][c] = sum_k of rows r and c of each walker's 2 N rows (A and B the
// same operand, one tile per walker, RT = oz_term_width(N), N <= 32).
int oz_gram(const OzOperand& rows, int W, int N, double* gram, int* err, cudaStream_t st);

// Exchange: part[w][c][2] = sum over the vectors of row tile c of
// sum_ij T_ij T_ji, T_g = Lh_g Theta_w (same-spin pairs).  A: rows (g, i),
// rows_per_tile a multiple of N; B: rows (w, c, j), rows_per_tile a multiple
// of 2 N.
struct OzExchange {
  int W = 0, N = 0, G = 0, nup = 0, nchunk = 0;
  OzOperand A, B;
  double* part = nullptr;
  int* err = nullptr;
};
int oz_exchange_vectors(int N);  // vectors per row tile
int oz_exchange_walkers(int N);  // walkers per column tile
int oz_exchange(const OzExchange& x, cudaStream_t st);

}  // namespace afq
