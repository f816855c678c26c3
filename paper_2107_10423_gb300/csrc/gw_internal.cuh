// Internal declarations of libgw: kernel launchers shared between translation units.
// Not part of the public ABI (include/gw.h).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <atomic>
#include <cstdint>
#include <vector>

namespace gw {

// Runs a set-up that belongs to a device (kernel attributes) once on each, again where it failed; any thread may call it.
class PerDevice {
  std::atomic<unsigned long long> done_[2] = {};

 public:
  template <typename F>
  cudaError_t run(int dev, F set_up) {
    if (dev < 0 || dev >= 128) return set_up();
    const unsigned long long bit = 1ull << (dev & 63);
    if (done_[dev >> 6].load(std::memory_order_acquire) & bit) return cudaSuccess;
    const cudaError_t e = set_up();              // threads that meet here each run it
    if (e == cudaSuccess) done_[dev >> 6].fetch_or(bit, std::memory_order_release);
    return e;
  }
  template <typename F>
  cudaError_t run(F set_up) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e == cudaSuccess ? run(dev, set_up) : e;
  }
};

// Lets a kernel take all the dynamic shared memory its device has, once per device.  The limit is a property of the kernel
// that every thread shares: set to each launch's own size, a plan's smaller one between another's call and launch makes
// that launch fail.
template <auto Kernel>
cudaError_t allow_smem() {
  static PerDevice once;
  return once.run([] {
    cudaFuncAttributes a;
    int dev = 0, most = 0;
    cudaError_t e = cudaFuncGetAttributes(&a, (const void*)Kernel);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute((const void*)Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               most - (int)a.sharedSizeBytes);
    return e;
  });
}

// ---------------------------------------------------------------- dense kernels (kernels_dense.cu)
// Every kernel below takes the pair energies D_k (k < n_ov, the columns of B) as an array Dk.
// In-place lower Cholesky of `batch` SPD matrices A[b] = base + b*stride (row-major n x n).
// info[b] = 0 on success, j+1 if pivot j was not positive.
template <typename T>
void launch_cholesky(T* base, int n, long stride, int batch, int* info, cudaStream_t s);

// out_g = Pi(i xi_g) (mode 0) or 1 - Pi(i xi_g) (mode 1), g < n_xi, n_aux x n_aux, on the FP64 pipe; flags: only the
// lower 64 x 64 tiles whose flag [g][tile] is set (oz_cover's).
void launch_pi_syrk(const double* B, const double* Dk, long n_ov, int n_aux, const double* xi, int n_xi, double* out,
                    int mode, cudaStream_t s, const int* flags = nullptr);

// X_b = L_b^-1 (full n x n, zeros above the diagonal) from lower factors L_b at stride `stride`.
cudaError_t launch_tri_inv(const double* L, long stride, int n, int batch, double* X, long xstride, cudaStream_t s);
// W[r][c] = -|Bn_r|^2 for c < n_cols.
cudaError_t launch_w_minus_norm(const double* Bn, int n, long R, int n_cols, double* W, cudaStream_t s);

// W table from Cholesky factors (gw_w_table_noalloc, small FP64 plans): for matrices g in [0, n_g): y = L_g^-1 b_r for rows r of Bn [R][n],
// W[r*w_ld + g_out[g]] = |y|^2 - |b|^2 = b^T(eps^-1 - 1)b.  scratch: [n_cta][n][64] elements of T.
template <typename T>
cudaError_t launch_trsm_w(const T* Lbase, long Lstride, int n, int n_g, const int* g_out, const T* Bn, int R,
                          double* W, int w_ld, T* scratch, int n_cta, cudaStream_t s);
template <typename T>
size_t trsm_w_scratch_elems(int n, int n_cta);
int trsm_w_default_ctas();

// Matrix-free FP64 operator of the residue systems (MINRES), for a batch of nr right-hand sides.
// V: [2nr][n_aux] pairs (u, v) encoding z = u - i v.
// gemm1: U[2j..2j+1][k] = c_k(x_j) * t_k, t = B^T z, with c_k(x) = 2[1/(x-D_k+i eta) + 1/(-x-D_k+i eta)].
// gemm2: S[r][P] = sum_k U[r][k] B[P][k]; mode 0 writes S (= [Re; Im] of Pi z),
//   mode 1 writes the real embedding [u - S_re; -v - S_im] of (1 - Pi) z.
// run_if: device flag, the launch does nothing if *run_if == 0.
void launch_op_gemm1(const double* V, const double* B, const double* Dk, long n_ov, int n_aux, const double* x,
                     double eta, int nr, double* U, cudaStream_t s, const int* run_if = nullptr);
void launch_op_gemm2(const double* U, const double* B, int n_aux, long n_ov, int nr, const double* V, double* out,
                     int mode, cudaStream_t s, const int* run_if = nullptr);
// Both products in FP32 for up to kSkinnyRhs right-hand sides: B FP32 [n_aux][ldb] (rows 16-byte aligned, zero padded),
// U [2 nr][ldb] work space, S as in gemm2.
constexpr int kSkinnyRhs = 4;
void launch_op_skinny(const float* V, const float* B, long ldb, const double* Dk, int n_ov, int n_aux, const double* x,
                      float eta, int nr, float* U, float* S, int mode, cudaStream_t s, const int* run_if);
// dw[j] += sum_k Re(c'_k(x_j) t_k^2) in FP64, c' the x-derivative (dw zeroed by the caller), skipping the pairs with
// |x_j - D_k| < cut or |-x_j - D_k| < cut (added by launch_deriv_resonant); ldb: row length of B.
template <typename T>
void launch_deriv(const T* V, const T* B, const double* Dk, long n_ov, int n_aux, const double* x, double eta, int nr,
                  double* dw, double cut, long ldb, cudaStream_t s);
// Double-float (FP32 pair, 48-bit) versions of op_gemm1 and op_gemm2 mode 1 for the refinement residual:
// V, U, out FP64; B as its split Bh + Bl (launch_df_split of the FP64 B_ia): Bh [n_aux][ldh] is the FP32 rounding
// of B (the plan's FP32 copy), Bl [n_aux][n_ov] the rounding of the remainder.  launch_df_split writes h only if it
// is not NULL.
void launch_df_split(const double* x, long n, float* h, float* l, cudaStream_t s);
void launch_op_gemm1_df(const double* V, const float* Bh, const float* Bl, long ldh, const double* Dk, long n_ov,
                        int n_aux, const double* x, double eta, int nr, double* U, cudaStream_t s);
// part: op_gemm2_df_ranges x 2 nr x n_aux work space where that is more than one range (at most kDfPartTiles 64 x 64 tiles).
constexpr long kDfPartTiles = 1520;
int op_gemm2_df_ranges(int n_aux, long n_ov, int nr);
void launch_op_gemm2_df(const double* U, const float* Bh, const float* Bl, long ldh, int n_aux, int n_ov, int nr,
                        const double* V, double* out, double* part, cudaStream_t s);
// The pairs that launch_deriv skips, in FP64: dw[j] += Re(c'_k(x_j) t_k^2) with t from the FP64 rows of V64 and the FP64
// B_ia [n_aux][n_ov]; Dsort ascending pair energies with their pair indices kidx.
void launch_deriv_resonant(const double* V64, const double* B, long n_ov, int n_aux, const double* Dsort,
                           const int* kidx, const double* xs, int nr, double eta, double cut, double* dw,
                           cudaStream_t s);
// ---------------------------------------------------------------- CD kernels (kernels_cd.cu)
// Sigma_x of each target; occ_t (device [n_t], or NULL for n_occ everywhere): occupied states of its spin.
void launch_sigma_x(const double* B_nm, int n_t, int n_bas, int n_aux, int n_occ, double* sx, cudaStream_t s,
                    const int* occ_t = nullptr);

// I term (eq. "inn") with optional static subtraction, per target t at omega[t].
// n_t evaluation points; point t reads the W rows of target tmap[t] (t itself when tmap is NULL) and the G energies
// eps + spin[target] * n_bas (eps [n_spin][n_bas]; spin NULL: one set).
void launch_sigma_imag(const double* W, int n_t, int n_bas, int n_g, const double* eps, const double* xi,
                       const double* wt, const double* omega, int static_sub, double* I, double* dI,
                       const unsigned char* active, cudaStream_t s, const int* tmap = nullptr,
                       const int* spin = nullptr);

struct MinresState {
  double beta, c2, s2, c1, s1, phibar, beta1, pad;
  int iters, done, pad0, pad1;
};

// Gather b_j = B_nm[t_j][m_j] into V as (u, v) = (b, 0); T is the operator precision.
template <typename T>
void launch_gather_rhs(const double* B_nm, int n_bas, int n_aux, const int* rhs_t, const int* rhs_m, int nr, T* V,
                       cudaStream_t s);
// From S = [Re; Im](Pi b): initialise MINRES (v_1 = rhs/|rhs|) and write v_1 into V.
template <typename T>
void launch_minres_init(const T* S, int nr, int n_aux, double* vprev, double* v, double* d1, double* d2, double* x,
                        MinresState* st, T* V, cudaStream_t s);
// One MINRES step given P = E v (embedding matvec output).  Writes the next Lanczos vector into V.
template <typename T>
void launch_minres_step(const T* P, int nr, int n_aux, double tol, double* vprev, double* v, double* d1, double* d2,
                        double* x, MinresState* st, T* V, int* n_active, cudaStream_t s);
// After MINRES: W = b^T delta; y = b + delta written into V as (u, v) = (y_r, -y_i) for the derivative pass
// (and into V64 in FP64 when given).
template <typename T>
void launch_minres_finish(const double* B_nm, int n_bas, int n_aux, const int* rhs_t, const int* rhs_m, int nr,
                          const double* x, const MinresState* st, double* w_re, double* w_im, int* iters,
                          double* resnorm, T* V, cudaStream_t s, double* V64 = nullptr);

// Spectral-decomposition route (kernels_sd.cu): the Casida matrix M = D^1/2 (D + 4 B^T B) D^1/2 [Np][Np] (Np = N
// rounded up to even, identity padding) and T = I; one cyclic Jacobi sweep of M (rotations accumulated in T, cs [Np]
// work space); off[0] / off[1] = squared off-diagonal / diagonal Frobenius norms; Omega [N], V = 2 B D^1/2 T
// [n_aux][N] and the pole weights w2[r][s] = (Bn_r . V_s)^2 / (2 Omega_s) for the R rows of Bn; Sigma_c and its
// derivative at evaluation points (target tmap[p] at omega[p]) from those weights.
cudaError_t sd_casida_matrix(const double* B, const double* Dk, int n_aux, int N, int Np, double* M, double* T,
                             cudaStream_t s);
cudaError_t sd_jacobi_sweep(double* M, double* T, int Np, double* cs, cudaStream_t s);
cudaError_t sd_offdiag(const double* M, int Np, double* off, cudaStream_t s);
cudaError_t sd_weights(const double* B, const double* Dk, const double* M, const double* T, const double* Bn,
                       int n_aux, int N, int Np, int R, double* Om, double* V, double* w2, cudaStream_t s);
// part [npts][sd_sigma_parts][2] is work space.
int sd_sigma_parts(int n_bas, int N);
cudaError_t sd_sigma(const double* w2, const double* Om, int N, int n_bas, const double* eps, const int* tmap,
                     const int* spin, const int* occ_t, int n_occ, const double* omega, int npts, double eta,
                     double* part, double* S, double* dS, cudaStream_t s);
// Direct route (N <= sd_direct_max()): A [N][ld] (overwritten) = Q T Q^T with reflectors H [N][ld], beta, d, e [N]
// (p_buf [4 N], bar one counter, *err set if a wait ran out); then eigenvectors Z (rows, length ld) of A from T by
// bisection (lam), twisted factorisations (W1, W2 [N][ldw]) and the reflectors; nrm [N] work space.
int sd_direct_max();
cudaError_t sd_tridiagonal(double* A, int N, long ld, double* H, double* beta, double* d, double* e, double* p_buf,
                           unsigned* bar, int* err, cudaStream_t s);
cudaError_t sd_tridiagonal_vectors(const double* d, const double* e, int N, double* lam, double* W1, double* W2, long ldw,
                                   const double* H, const double* beta, long ld, double* nrm, double* Z,
                                   cudaStream_t s);
// Refinement step on rows V with S = V M V^T and G = V V^T ([N][N]): norms [3] (off-diagonal and diagonal squares of S,
// squares of I - G), and C = I + E^T, the factor of the next rows C V.
cudaError_t sd_eig_norms(const double* S, const double* G, int N, double* norms, cudaStream_t s);
cudaError_t sd_eig_update(const double* S, double* G, int N, double* C, const double* norms, cudaStream_t s);
cudaError_t sd_pack_rows(const double* X, int rows, int N, long ld, double* Y, cudaStream_t s);
cudaError_t sd_twice_sqrt(const double* Dk, int N, double* w, cudaStream_t s);
// Omega from S and G, and the pole weights from V = 2 B D^1/2 T [n_aux][N].
cudaError_t sd_rows_weights(const double* S, const double* G, const double* V, const double* Bn, int n_aux, int N, int R,
                            double* Om, double* w2, cudaStream_t s);
// Blocked LU of `batch` complex matrices (planes A and A + plane, matrix stride `stride`, FP32 or FP64) with partial
// pivoting, in place, trailing updates on the tensor cores.  perm [batch][n]: the row order as launch_zlu_solve reads it
// (the original row at each row of the factors; the sequential swaps for n > 16384, FP64 8192); info[b]: 0, or the first zero pivot's column + 1.  Work space: work of work_elems BF16 (at least
// zlu_operand_elems(n, 1, fp64); the batch runs in sub-batches that fit it), idx zlu_index_ints, linv zlu_linv_elems,
// scales zlu_scale_elems (FP64 only).
size_t zlu_operand_elems(int n, int batch, bool fp64);
size_t zlu_index_ints(int batch);
size_t zlu_linv_elems(int batch);
size_t zlu_scale_elems(int n, int batch);
template <typename T>
cudaError_t launch_zlu(T* A, long stride, long plane, int n, int batch, int* perm, int* info, __nv_bfloat16* work,
                       size_t work_elems, int* idx, T* linv, double* scales, int* err, cudaStream_t s);
template <typename T>
cudaError_t launch_zlu_solve(const T* Ar, const T* Ai, long stride, int n, int batch, const int* perm, T* yr, T* yi,
                             long ystride, cudaStream_t s);
// Fallback bookkeeping: for k < nf with slot index idx[k] (into the MINRES batch), set y planes = (b, 0) before
// the solve (stage 0), or after it write W = b^T y - b^T b, resnorm 0 and the (u, v) = (y_r, -y_i) rows of V.
template <typename T>
void launch_fallback_rhs(const double* B_nm, int n_bas, int n_aux, const int* rt, const int* rm, const int* idx,
                         int nf, T* y, cudaStream_t s);
template <typename T>
void launch_fallback_finish(const double* B_nm, int n_bas, int n_aux, const int* rt, const int* rm, const int* idx,
                            int nf, const T* y, double* w_re, double* w_im, double* resnorm, T* V, cudaStream_t s);

// Iterative refinement of fallback solves (k < nf; y32 planes [nf][2][n], y64 the same in FP64):
//   stage 0: y64 = y32;            V32 rows (2k, 2k+1) = (Re y, -Im y)
//   stage 1: y32 = [b; 0] - S      (residual, next right-hand side; S = S32 rows (2k, 2k+1), or, if S64 is given,
//                                   S64 rows (2q, 2q+1) with q = pos[k] (q = k without pos; q < 0: y32 = 0))
//   stage 2: y64 += y32;           V32 rows = (Re y, -Im y); rho[k] = |y32| / |y64| if rho is given
void launch_refine(int stage, const double* B_nm, int n_bas, int n_aux, const int* rt, const int* rm, const int* idx,
                   int nf, float* y32, double* y64, float* V32, const float* S32, cudaStream_t s,
                   const double* S64 = nullptr, const int* pos = nullptr, double* rho = nullptr);
// V64 rows (2q, 2q+1) = (Re y, -Im y) of the FP64 solution sel[q] (q without sel) of y64 [.][2][n], q < m.
void launch_refine_v64(int m, int n_aux, const int* sel, const double* y64, double* V64, cudaStream_t s);
// W = b^T y - b^T b from FP64 solutions; V (operator precision) rows of slot idx[k] = (Re y, -Im y); resnorm 0.
template <typename T>
void launch_fallback_finish64(const double* B_nm, int n_bas, int n_aux, const int* rt, const int* rm, const int* idx,
                              int nf, const double* y64, double* w_re, double* w_im, double* resnorm, T* V,
                              cudaStream_t s, double* V64 = nullptr);

// Nodes of the imaginary-axis stage (freq_nodes.cu): the positions at which it is computed and the matrix that gives
// every grid column of W from them.
struct FreqNodes {
  std::vector<int> col;       // W column per position: position 0 is the static point (column n_g), then grid columns
  int n_diff = 0;             // positions 1 .. n_diff hold W_g - W_0 (difference form)
  std::vector<double> C;      // [positions][n_g]: W[r][g] = sum_p C[p][g] value_p
};
// Nodes for the ascending positive grid xi whose first n_diff points are difference columns, for poles in
// [D_min, inf); false where the nodes would save less than a quarter of the n_g + 1 points or the grid is not
// ascending and positive (the stage then runs at every point).
bool freq_nodes(const std::vector<double>& xi, int n_diff, double D_min, FreqNodes& out);
// Every grid column of W [R][n_g + 1] from the node columns (col, C: device copies of FreqNodes).
cudaError_t launch_w_expand(double* W, long R, int n_g, int n_pos, const int* col, const double* C, cudaStream_t s);

// R term reduction per target over its right-hand sides [start[t], start[t+1]).
// W[r][g] += W[r][n_g] for g < n_cols (table [R][n_g + 1]): columns held as differences from the static one.
void launch_w_add_static(double* W, long R, int n_g, int n_cols, cudaStream_t s);
// W[r][c] = 0 outside the processing positions [p0, p1) (position 0 = column n_g, position p > 0 = column p - 1).
void launch_w_keep_positions(double* W, long R, int n_g, int p0, int p1, cudaStream_t s);
void launch_residue_reduce(const int* start, int n_t, const double* coef, const double* w_re, const double* dw_re,
                           double* R, double* dR, cudaStream_t s);

struct QPState {
  double omega, f_prev, omega_prev, Z;
  double a, fa, b, fb, x, fx;
  double sigma, dsigma;
  int br_kind, has_prev, iter, status;   // status: 0 running, 1 converged, 2 not converged
};
void launch_qp_init(QPState* st, const double* omega0, int n, cudaStream_t s);   // omega0: starting points
// sigma = R - I, dsigma = dR - dI for active states, then one step-tree step.
void launch_qp_step(QPState* st, const double* R, const double* dR, const double* I, const double* dI,
                    const double* e_n, const double* shift, double tol, int maxit, int n, int linearised,
                    cudaStream_t s);

}  // namespace gw
