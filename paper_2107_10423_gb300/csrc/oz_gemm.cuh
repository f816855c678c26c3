// FP64 products on the BF16 tensor cores by exact integer digits (oz_gemm.cu).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstddef>

namespace gw {

constexpr int OZ_S = 8;              // digits per operand element

// Digit operand: dig [batch][OZ_S][rows][ld] BF16 and sc [batch][rows] (the power of two of each row).
struct OzOperand {
  const __nv_bfloat16* dig;
  const double* sc;
  int batched;                       // 0: one matrix for every entry
};

enum { OZ_EPI_STORE = 0, OZ_EPI_SUMSQ = 1, OZ_EPI_SUB2 = 2 };
struct OzEpi {
  int kind;
  // OZ_EPI_STORE: out_b[m][n] = f(v) (f: 0 v, 1 delta_mn - v, 2 -v; even / odd entries), added to what is there when
  // accumulate; lower != 0 computes the lower tiles and mirrors them
  int mode_even, mode_odd, lower, accumulate;
  double* out;
  long out_bstride;
  int ldo;
  // OZ_EPI_SUMSQ: part[b][column tile][m] = sum of v[m][n]^2 over a tile's 32 columns (oz_sumsq_tiles(N) tiles of M values
  // an entry; oz_sumsq_add sums them); the B rows are lower triangular (row n ends at column n)
  double* part;
  // OZ_EPI_SUB2: out_b[m][n] -= v for m < half, out_b[plane + (m - half) ldo + n] -= v below (ldo, out_bstride as above)
  long plane;
  int half;
};

int oz_sumsq_tiles(int N);
// W[m * ldw + gidx[b]] += sum over the column tiles t of part[b][t][m], t ascending, for b < batch and m < M.
cudaError_t oz_sumsq_add(const double* part, int batch, int tiles, int M, double* W, int ldw, const int* gidx,
                         cudaStream_t s);
int oz_ld(int K);                    // row length of the digit arrays
size_t oz_elems(int rows, int K);    // BF16 elements of one matrix's digits
// out_b[m][n] = f(sum_k A_b[m][k] B_b[n][k]) for b < batch.  *err receives a code if a bounded wait ran out.
cudaError_t oz_gemm(const OzOperand& A, const OzOperand& B, int batch, int M, int N, int K, const OzEpi& ep, int* err,
                    cudaStream_t s);

// Row scales sc[r] = 2^e >= max_k |x[r][k]| (NaN for a row with a NaN or infinity); rows of `cols` at stride ld.
cudaError_t oz_row_scale(const double* x, int rows, long cols, long ld, double* sc, cudaStream_t s);
// Digits of rows x_b[r][k0 .. k0 + cols) (stride ld, matrices b < nb at stride xbs) with the rows' scales sc [nb][rows].
cudaError_t oz_split(const double* x, long xbs, int rows, int k0, int cols, long ld, const double* sc, int nb,
                     __nv_bfloat16* dig, cudaStream_t s);
// Digits of the transpose: row c of the operand is column c of x [rows][ld] (cols operand rows of length rows).
cudaError_t oz_split_transpose(const double* x, int rows, int cols, long ld, const double* sc, __nv_bfloat16* dig,
                               cudaStream_t s);
cudaError_t oz_col_scale(const double* x, int rows, int cols, long ld, double* sc, cudaStream_t s);
// Digits and scales of x[r][k] f[b][k] (digA, scA [nb][rows]) and, unless h is null, of x[r][k] 2^h[b][k] (digB, scB) for
// the columns [k0, k0 + cols) and nb rows of weights.
cudaError_t oz_split_weighted(const double* x, int rows, int k0, int cols, long ld, const double* f, const int* h,
                              long ldw, int nb, __nv_bfloat16* digA, double* scA, __nv_bfloat16* digB, double* scB,
                              cudaStream_t s);
// FP64 weights w[b][k] of tc_pair_weights' kinds (row length K) as f 2^h, 4^h ~ |w|.
cudaError_t oz_pair_weights(const double* Dk, int K, const int* kinds, const double* params, double eta, int nb,
                            double* f, int* h, cudaStream_t s);
// flags[b][t] = 1 for the lower 64 x 64 tiles t of entry b that hold an element whose sum of |terms| is below an eighth of
// its two scales' product, or of a row with a NaN or an infinity (others are left as they are); batched operands of n rows
// and `cols` columns, oz_cover_tiles(n) tiles an entry.
int oz_cover_tiles(int n);
cudaError_t oz_cover(const OzOperand& A, const OzOperand& B, int n, int cols, int nb, int* flags, cudaStream_t s);

// Row scales and digits of x [rows][cols] (row length ld) in one launch.
cudaError_t oz_row_digits(const double* x, int rows, int cols, long ld, double* sc, __nv_bfloat16* dig,
                          cudaStream_t s);
// dw[j] = sum_k Re(c'_k(x_j) t_k^2), t_k = T[2j][k] - i T[2j + 1][k].
cudaError_t oz_pole_derivative(const double* T, int K, const double* Dk, const double* xs, double eta, int nr,
                               double* dw, cudaStream_t s);

}  // namespace gw
