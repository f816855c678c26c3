// Dense kernels of the CD-G0W0 path (SIMT, templated on the arithmetic type):
//  * Pi(i xi) of small FP64 plans;
//  * batched in-place Cholesky of eps(i xi) = 1 - Pi (SPD, Sec. 3.3 text after "inn");
//  * triangular solves that turn the factors into the table W^c_nm(i xi) (Algorithm 1, imaginary-grid loop);
//  * the two skinny products of the FP64 matrix-free residue operator 1 - Pi(x) (Sec. 3.3, MINRES paragraph) and the
//    derivative pass.
#include "gw_internal.cuh"
#include "gw.h"

#include <cstdio>
#include <mutex>

namespace gw {

namespace {

constexpr int TM = 64;     // tile rows
constexpr int TN = 64;     // tile cols
constexpr int TK = 16;     // k step
constexpr int NT = 256;    // threads per CTA (16 x 16, 4 x 4 outputs each)

// ------------------------------------------------------------------ Pi(i xi) SYRK
// Pi(i xi) on the FP64 pipe: 1 - Pi of FP64 plans of at most one 128-row digit tile (screening_T), and the tiles of a
// digit product that oz_cover flagged (flags: one per tile and frequency, the others are left alone).
// grid.x: lower-triangular tile index (bi >= bj), grid.y: frequency index.
__global__ void __launch_bounds__(NT) pi_syrk_kernel(const double* __restrict__ B, const double* __restrict__ Dk,
                                                     long n_ov, int n_aux,
                                                     const double* __restrict__ xi, double* __restrict__ out, int mode,
                                                     const int* __restrict__ flags) {
  if (flags && flags[(long)blockIdx.y * gridDim.x + blockIdx.x] == 0) return;
  __shared__ double As[TK][TM + 4];
  __shared__ double Bs[TK][TN + 4];
  // decode lower tile (bi, bj) from linear index t = bi*(bi+1)/2 + bj
  int t = blockIdx.x;
  int bi = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
  while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
  while (bi * (bi + 1) / 2 > t) --bi;
  int bj = t - bi * (bi + 1) / 2;
  const int g = blockIdx.y;
  const double x2 = xi[g] * xi[g];
  const int p0 = bi * TM, q0 = bj * TN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  const int lr = tid >> 2, lk = (tid & 3) * 4;
  for (long k0 = 0; k0 < n_ov; k0 += TK) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      long k = k0 + lk + u;
      double wa = 0.0, va = 0.0, vb = 0.0;
      if (k < n_ov) {
        const double D = Dk[k];
        wa = (-4.0 * D / (D * D + x2));
        if (p0 + lr < n_aux) va = B[(long)(p0 + lr) * n_ov + k];
        if (q0 + lr < n_aux) vb = B[(long)(q0 + lr) * n_ov + k];
      }
      As[lk + u][lr] = va * wa;
      Bs[lk + u][lr] = vb;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  double* o = out + (long)g * n_aux * n_aux;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int p = p0 + ty + 16 * i;
    if (p >= n_aux) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int q = q0 + tx + 16 * j;
      if (q >= n_aux || q > p) continue;
      double v = acc[i][j];
      if (mode == 1) v = (p == q ? 1.0 : 0.0) - v;
      o[(long)p * n_aux + q] = v;
      o[(long)q * n_aux + p] = v;
    }
  }
}

// ------------------------------------------------------------------ batched Cholesky, one CTA per matrix
constexpr int CH_NB = 32;
constexpr int CH_THREADS = 512;

template <typename T>
__global__ void __launch_bounds__(CH_THREADS) cholesky_kernel(T* base, int n, long stride, int* info) {
  __shared__ T Ld[CH_NB][CH_NB + 1];
  __shared__ T Pi_[64][CH_NB + 1];
  __shared__ T Pj_[64][CH_NB + 1];
  __shared__ int bad;
  T* A = base + (long)blockIdx.x * stride;
  const int tid = threadIdx.x;
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int j0 = 0; j0 < n; j0 += CH_NB) {
    const int nb = min(CH_NB, n - j0);
    // (1) diagonal block
    for (int idx = tid; idx < nb * nb; idx += CH_THREADS) {
      int r = idx / nb, c = idx % nb;
      Ld[r][c] = A[(long)(j0 + r) * n + j0 + c];
    }
    __syncthreads();
    for (int c = 0; c < nb; ++c) {
      if (tid == 0) {
        T d = Ld[c][c];
        if (!(d > T(0))) { bad = j0 + c + 1; d = T(1); }
        Ld[c][c] = sqrt(d);
      }
      __syncthreads();
      for (int r = c + 1 + tid; r < nb; r += CH_THREADS) Ld[r][c] /= Ld[c][c];
      __syncthreads();
      for (int idx = tid; idx < (nb - c - 1) * (nb - c - 1); idx += CH_THREADS) {
        int r = c + 1 + idx / (nb - c - 1), s = c + 1 + idx % (nb - c - 1);
        if (s <= r) Ld[r][s] -= Ld[r][c] * Ld[s][c];
      }
      __syncthreads();
    }
    for (int idx = tid; idx < nb * nb; idx += CH_THREADS) {
      int r = idx / nb, c = idx % nb;
      if (c <= r) A[(long)(j0 + r) * n + j0 + c] = Ld[r][c];
    }
    // (2) panel rows below: x L^T = a
    for (int i = j0 + nb + tid; i < n; i += CH_THREADS) {
      T xr[CH_NB];
      for (int c = 0; c < nb; ++c) {
        T v = A[(long)i * n + j0 + c];
        for (int s = 0; s < c; ++s) v -= xr[s] * Ld[c][s];
        xr[c] = v / Ld[c][c];
      }
      for (int c = 0; c < nb; ++c) A[(long)i * n + j0 + c] = xr[c];
    }
    __threadfence_block();
    __syncthreads();
    // (3) trailing lower update A[i][j] -= sum_c P[i][c] P[j][c], i >= j >= j0+nb
    const int t0 = j0 + nb;
    const int nt = (n - t0 + 63) / 64;
    for (int ti = 0; ti < nt; ++ti) {
      for (int tj = 0; tj <= ti; ++tj) {
        const int r0 = t0 + ti * 64, c0 = t0 + tj * 64;
        for (int idx = tid; idx < 64 * CH_NB; idx += CH_THREADS) {
          int r = idx / CH_NB, c = idx % CH_NB;
          Pi_[r][c] = (r0 + r < n && c < nb) ? A[(long)(r0 + r) * n + j0 + c] : T(0);
          Pj_[r][c] = (c0 + r < n && c < nb) ? A[(long)(c0 + r) * n + j0 + c] : T(0);
        }
        __syncthreads();
        const int r = tid >> 3;             // 0..63
        const int cb = tid & 7;             // cols cb + 8*jj
        T acc[8];
        for (int jj = 0; jj < 8; ++jj) acc[jj] = T(0);
        for (int c = 0; c < nb; ++c) {
          T a = Pi_[r][c];
          for (int jj = 0; jj < 8; ++jj) acc[jj] = fma(a, Pj_[cb + 8 * jj][c], acc[jj]);
        }
        const int gi = r0 + r;
        if (gi < n) {
          for (int jj = 0; jj < 8; ++jj) {
            int gj = c0 + cb + 8 * jj;
            if (gj < n && gj <= gi) A[(long)gi * n + gj] -= acc[jj];
          }
        }
        __syncthreads();
      }
    }
    __threadfence_block();
    __syncthreads();
  }
  if (tid == 0) info[blockIdx.x] = bad;
}

// ------------------------------------------------------------------ inverse of the Cholesky factors
// X = L^-1 (lower, zeros above the diagonal) for a batch of factors.  CTA (J, b) builds the 64 columns of block J:
//   X_JJ = L_JJ^-1,  X_IJ = -L_II^-1 sum_{J <= K < I} L_IK X_KJ,
// every column block on its own, so (n / 64) CTAs a matrix; n^3/6 FP64 FMAs a matrix, bound by the FP64 pipe.
__global__ void __launch_bounds__(NT) tri_inv_kernel(const double* __restrict__ Lb, long stride, int n,
                                                     double* __restrict__ Xb, long xstride) {
  __shared__ double As[TK][TM + 4];
  __shared__ double Bs[TK][TN + 4];
  extern __shared__ double tri_sm[];
  double* Ts = tri_sm;                  // [64][65]
  double* Ls = tri_sm + 64 * 65;        // [64][65]
  const double* L = Lb + (long)blockIdx.y * stride;
  double* X = Xb + (long)blockIdx.y * xstride;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int J = blockIdx.x, nJ = (n + 63) / 64, c0 = J * 64;
  for (int i = tid; i < c0 * 64; i += NT) {          // zeros above the diagonal block
    const int r = i >> 6, c = c0 + (i & 63);
    if (c < n) X[(long)r * n + c] = 0.0;
  }
  for (int I = J; I < nJ; ++I) {
    const int r0 = I * 64, nr = min(64, n - r0);
    double acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = (I == J && ty + 16 * i == tx + 16 * j) ? 1.0 : 0.0;
    for (int k0 = c0; k0 < r0; k0 += TK) {
      {
        const int r = tid >> 2, k4 = (tid & 3) * 4, kr = tid >> 4, c4 = (tid & 15) * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          As[k4 + u][r] = r0 + r < n ? L[(long)(r0 + r) * n + k0 + k4 + u] : 0.0;
          Bs[kr][c4 + u] = c0 + c4 + u < n ? X[(long)(k0 + kr) * n + c0 + c4 + u] : 0.0;
        }
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < TK; ++kk) {
        double a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
        for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fma(-a[i], b[j], acc[i][j]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) Ts[(ty + 16 * i) * 65 + tx + 16 * j] = acc[i][j];
    for (int idx = tid; idx < 64 * 64; idx += NT) {
      const int r = idx >> 6, c = idx & 63;
      Ls[r * 65 + c] = (r < nr && c <= r) ? L[(long)(r0 + r) * n + r0 + c] : 0.0;
    }
    __syncthreads();
    if (tid < 64)
      for (int p = 0; p < nr; ++p) {
        double v = Ts[p * 65 + tid];
        for (int q = 0; q < p; ++q) v = fma(-Ls[p * 65 + q], Ts[q * 65 + tid], v);
        Ts[p * 65 + tid] = v / Ls[p * 65 + p];
      }
    __syncthreads();
    for (int idx = tid; idx < 64 * 64; idx += NT) {
      const int r = idx >> 6, c = idx & 63;
      if (r < nr && c0 + c < n) X[(long)(r0 + r) * n + c0 + c] = (I == J && c > r) ? 0.0 : Ts[r * 65 + c];
    }
    __threadfence_block();
    __syncthreads();
  }
}

// W[r][col] = -|b_r|^2 for every column of the table (the sums of squares of L^-1 b_r are then added).
__global__ void __launch_bounds__(128) w_minus_norm_kernel(const double* __restrict__ Bn, int n, long R, int n_cols,
                                                           double* __restrict__ W) {
  const int lane = threadIdx.x & 31;
  for (long r = blockIdx.x * 4L + (threadIdx.x >> 5); r < R; r += gridDim.x * 4L) {
    double s = 0.0;
    for (int p = lane; p < n; p += 32) s = fma(Bn[r * n + p], Bn[r * n + p], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    for (int c = lane; c < n_cols; c += 32) W[r * n_cols + c] = -s;
  }
}

// ------------------------------------------------------------------ TRSM -> W table
// Work item = (matrix g, tile of 64 right-hand sides).  Y for the tile lives in this CTA's scratch slice.
template <typename T>
__global__ void __launch_bounds__(NT) trsm_w_kernel(const T* __restrict__ Lbase, long Lstride, int n, int n_g,
                                                    const int* __restrict__ g_out, const T* __restrict__ Bn, int R,
                                                    double* __restrict__ W, int w_ld, T* __restrict__ scratch) {
  extern __shared__ unsigned char smem_raw[];
  T* As = reinterpret_cast<T*>(smem_raw);             // [TK][TM+4]
  T* Bs = As + TK * (TM + 4);                          // [TK][TN+4]
  T* Ts = Bs + TK * (TN + 4);                          // [64][65]
  T* Ls = Ts + 64 * 65;                                // [64][65]
  double* red = reinterpret_cast<double*>(Ls + 64 * 65);  // [2][16][64]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int n_ct = (R + 63) / 64;
  const int nJ = (n + 63) / 64;
  // per-CTA slice of [nJ*64][64]: the last row block is written in full (zeros past n)
  T* Y = scratch + (long)blockIdx.x * nJ * 64 * 64;
  const long n_items = (long)n_g * n_ct;
  for (long item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int g = (int)(item / n_ct);
    const int r0 = (int)(item % n_ct) * 64;
    const T* L = Lbase + (long)g * Lstride;
    double ws[4] = {0, 0, 0, 0}, bs[4] = {0, 0, 0, 0};
    for (int J = 0; J < nJ; ++J) {
      const int P0 = J * 64;
      const int nr = min(64, n - P0);
      T acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          int P = P0 + ty + 16 * i, c = r0 + tx + 16 * j;
          T v = (P < n && c < R) ? Bn[(long)c * n + P] : T(0);
          acc[i][j] = v;
          bs[j] += (double)v * (double)v;
        }
      for (int K = 0; K < J; ++K) {
        for (int kk0 = 0; kk0 < 64; kk0 += TK) {
          {
            // As[kk][r] = L[P0+r][K*64+kk0+kk]; Bs[kk][c] = Y[(K*64+kk0+kk)*64 + c]
            int r = tid >> 2, k4 = (tid & 3) * 4;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              int kk = k4 + u;
              int col = K * 64 + kk0 + kk;
              As[kk * (TM + 4) + r] = (P0 + r < n) ? L[(long)(P0 + r) * n + col] : T(0);
            }
            int kr = tid >> 4, c4 = (tid & 15) * 4;
#pragma unroll
            for (int u = 0; u < 4; ++u) Bs[kr * (TN + 4) + c4 + u] = Y[(long)(K * 64 + kk0 + kr) * 64 + c4 + u];
          }
          __syncthreads();
#pragma unroll
          for (int kk = 0; kk < TK; ++kk) {
            T a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk * (TM + 4) + ty + 16 * i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk * (TN + 4) + tx + 16 * j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j) acc[i][j] = fma(-a[i], b[j], acc[i][j]);
          }
          __syncthreads();
        }
      }
      // stage the right-hand side block and the diagonal factor block
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) Ts[(ty + 16 * i) * 65 + tx + 16 * j] = acc[i][j];
      for (int idx = tid; idx < 64 * 64; idx += NT) {
        int r = idx >> 6, c = idx & 63;
        Ls[r * 65 + c] = (r < nr && c <= r) ? L[(long)(P0 + r) * n + P0 + c] : (r == c ? T(1) : T(0));
      }
      __syncthreads();
      if (tid < 64) {
        const int c = tid;
        for (int p = 0; p < nr; ++p) {
          T v = Ts[p * 65 + c];
          for (int q = 0; q < p; ++q) v = fma(-Ls[p * 65 + q], Ts[q * 65 + c], v);
          Ts[p * 65 + c] = v / Ls[p * 65 + p];
        }
      }
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          int p = ty + 16 * i, c = tx + 16 * j;
          T v = (p < nr) ? Ts[p * 65 + c] : T(0);
          Y[(long)(P0 + p) * 64 + c] = v;   // rows beyond n are never read
          ws[j] += (double)v * (double)v;
        }
      __threadfence_block();
      __syncthreads();
    }
    // reduce per column over ty
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      red[(0 * 16 + ty) * 64 + tx + 16 * j] = ws[j];
      red[(1 * 16 + ty) * 64 + tx + 16 * j] = bs[j];
    }
    __syncthreads();
    if (tid < 64) {
      double w = 0, b = 0;
      for (int y = 0; y < 16; ++y) { w += red[(0 * 16 + y) * 64 + tid]; b += red[(1 * 16 + y) * 64 + tid]; }
      int r = r0 + tid;
      if (r < R) W[(long)r * w_ld + g_out[g]] = w - b;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ derivative pass
// dw[j] += sum_k Re(c'_k(x_j) t_k^2) in FP64, t = V B over rows r in [0, 2nr) and the columns k (B is N-contiguous), the
// reduction fused into the product's epilogue (no N_ov-sized output); pairs within `cut` of resonance left out.
template <typename T>
__global__ void __launch_bounds__(NT) deriv_kernel(const T* __restrict__ V, const T* __restrict__ B,
                                                   const double* __restrict__ Dk, long n_ov, int n_aux,
                                                   const double* __restrict__ xs, double eta, int nr,
                                                   double* __restrict__ dw, double cut, long ldb) {
  __shared__ T As[TK][TM + 4];
  __shared__ T Bs[TK][TN + 4];
  const int M = 2 * nr;
  const int m0 = blockIdx.y * TM;
  const long k0c = (long)blockIdx.x * TN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
  for (int p0 = 0; p0 < n_aux; p0 += TK) {
    {
      int r = tid >> 2, k4 = (tid & 3) * 4;       // A: V rows, K (=P) contiguous
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        int P = p0 + k4 + u;
        As[k4 + u][r] = (m0 + r < M && P < n_aux) ? V[(long)(m0 + r) * n_aux + P] : T(0);
      }
      int kr = tid >> 4, c4 = (tid & 15) * 4;     // B: rows P, cols k contiguous
      int P = p0 + kr;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        long k = k0c + c4 + u;
        Bs[kr][c4 + u] = (P < n_aux && k < n_ov) ? B[(long)P * ldb + k] : T(0);
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][2 * ty + (i & 1) + 32 * (i >> 1)];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  const double e2 = eta * eta;
  // c' = 2[-(a1 - i eta)^2/d1^2 + (a2 - i eta)^2/d2^2]
#pragma unroll
  for (int ip = 0; ip < 2; ++ip) {
    const int r = m0 + 2 * ty + 32 * ip;
    double sum = 0.0;
    if (r < M) {
      const double x = xs[r >> 1];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long k = k0c + tx + 16 * j;
        if (k >= n_ov) continue;
        const double tr = (double)acc[2 * ip][j], ti = -(double)acc[2 * ip + 1][j];
        const double D = Dk[k];
        const double a1 = x - D, a2 = -x - D;
        if (fabs(a1) < cut || fabs(a2) < cut) continue;   // near resonance: FP64 pass (deriv_resonant)
        const double d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
        const double q1r = (a1 * a1 - e2) / (d1 * d1), q1i = -2.0 * a1 * eta / (d1 * d1);
        const double q2r = (a2 * a2 - e2) / (d2 * d2), q2i = -2.0 * a2 * eta / (d2 * d2);
        const double cr = 2.0 * (-q1r + q2r), ci = 2.0 * (-q1i + q2i);
        sum += cr * (tr * tr - ti * ti) - ci * (2.0 * tr * ti);
      }
    }
    // the 16 lanes tx of one ty hold the same row: reduce within each half warp
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (tx == 0 && r < M) atomicAdd(dw + (r >> 1), sum);
  }
}

// First index q of the ascending array with a[q] >= v.
__device__ __forceinline__ long lower_index(const double* a, long n, double v) {
  long lo = 0, hi = n;
  while (lo < hi) {
    const long mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// FP64 part of the fused derivative pass: the pairs k near resonance with x_j (|x_j - D_k| < cut or
// |-x_j - D_k| < cut, the same test in the same arithmetic as the FP32 pass, which skips them).  One CTA per right-hand
// side; candidate windows come from the ascending pair energies Dsort (pair index kidx), widened by cut on each side
// and then filtered by the exact test, so every pair is counted once.  One warp per pair:
// t_k = sum_P B[P][k] (u_P - i v_P) from the FP64 rows (u, v) = V64 rows (2j, 2j+1); dw[j] += Re(c'_k(x_j) t_k^2).
__global__ void __launch_bounds__(256) deriv_resonant_kernel(const double* __restrict__ V64,
                                                             const double* __restrict__ B, long n_ov, int n_aux,
                                                             const double* __restrict__ Dsort,
                                                             const int* __restrict__ kidx,
                                                             const double* __restrict__ xs, double eta, double cut,
                                                             double* __restrict__ dw) {
  __shared__ long rng[4];
  __shared__ double red[8];
  const int j = blockIdx.x;
  const double x = xs[j], e2 = eta * eta;
  if (threadIdx.x == 0) {
    long l1 = lower_index(Dsort, n_ov, x - 2.0 * cut), h1 = lower_index(Dsort, n_ov, x + 2.0 * cut);
    long l2 = lower_index(Dsort, n_ov, -x - 2.0 * cut), h2 = lower_index(Dsort, n_ov, -x + 2.0 * cut);
    if (l2 < h1 && l1 < h2) {   // overlapping windows: one merged window
      l1 = l1 < l2 ? l1 : l2;
      h1 = h1 > h2 ? h1 : h2;
      l2 = h2 = 0;
    }
    rng[0] = l1; rng[1] = h1; rng[2] = l2; rng[3] = h2;
  }
  __syncthreads();
  const double* u = V64 + (long)(2 * j) * n_aux;
  const double* v = u + n_aux;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double sum = 0.0;
  for (int w = 0; w < 2; ++w) {
    for (long q = rng[2 * w] + warp; q < rng[2 * w + 1]; q += nw) {
      const double D = Dsort[q];
      const double a1 = x - D, a2 = -x - D;
      if (!(fabs(a1) < cut || fabs(a2) < cut)) continue;   // warp-uniform
      const long k = kidx[q];
      double tr = 0.0, tv = 0.0;
      for (int P = lane; P < n_aux; P += 32) {
        const double b = B[(long)P * n_ov + k];
        tr += b * u[P];
        tv += b * v[P];
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        tr += __shfl_xor_sync(0xffffffffu, tr, o);
        tv += __shfl_xor_sync(0xffffffffu, tv, o);
      }
      const double ti = -tv;
      const double d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
      const double q1r = (a1 * a1 - e2) / (d1 * d1), q1i = -2.0 * a1 * eta / (d1 * d1);
      const double q2r = (a2 * a2 - e2) / (d2 * d2), q2i = -2.0 * a2 * eta / (d2 * d2);
      const double cr = 2.0 * (-q1r + q2r), ci = 2.0 * (-q1i + q2i);
      if (lane == 0) sum += cr * (tr * tr - ti * ti) - ci * (2.0 * tr * ti);
    }
  }
  if (lane == 0) red[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += red[w];
    atomicAdd(dw + j, t);
  }
}

// ------------------------------------------------------------------ FP64 residue operator
// One output a thread, one row a warp: a CTA takes CR rows x 32 columns, its warps without a row do nothing.  FP64 runs
// at two multiply-adds a clock and SM (16 clocks a warp instruction), so a tile must not pad: 64 x 64 tiles spent 91 us
// on a product of 2 rows, 84 and 95 long, and 3.2 ms on one of 382 rows, 504 and 3040 long on 48 CTAs (here 4 us and
// 1.1 ms, the FP64 pipe's own time).  Every output is one chain of FMAs in ascending order, as in those tiles: MINRES
// amplifies a last-bit difference of its operator to 1e-2 of a residual norm within 25 steps near a resonance, so the
// order is kept (products by exact digits take a sixth of the time, but round differently).
constexpr int CR = 8, CK = 32;

// gemm1: t = V B, then U[2j], U[2j + 1] = Re, Im of c_k(x_j) (t[2j] - i t[2j + 1]).
__global__ void __launch_bounds__(256) op_chain1_kernel(const double* __restrict__ V, const double* __restrict__ B,
                                                        const double* __restrict__ Dk, long n_ov, int n_aux,
                                                        const double* __restrict__ xs, double eta, int M,
                                                        double* __restrict__ U, const int* __restrict__ run_if) {
  if (run_if && *run_if == 0) return;
  __shared__ double As[CR][CK];
  __shared__ double Bs[CK][32];
  __shared__ double Ts[CR][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, m0 = blockIdx.y * CR, r = m0 + w;
  const long k = blockIdx.x * 32L + lane;
  double acc = 0.0;
  for (int p0 = 0; p0 < n_aux; p0 += CK) {
    As[w][lane] = (r < M && p0 + lane < n_aux) ? V[(long)r * n_aux + p0 + lane] : 0.0;
#pragma unroll
    for (int u = 0; u < CK / 8; ++u) {
      const int P = p0 + w + 8 * u;
      Bs[w + 8 * u][lane] = (P < n_aux && k < n_ov) ? B[(long)P * n_ov + k] : 0.0;
    }
    __syncthreads();
    if (r < M)
#pragma unroll
      for (int kk = 0; kk < CK; ++kk) acc = fma(As[w][kk], Bs[kk][lane], acc);
    __syncthreads();
  }
  Ts[w][lane] = acc;
  __syncthreads();
  if ((w & 1) || r >= M || k >= n_ov) return;
  const double tr = acc, ti = -Ts[w + 1][lane];
  // every rounding spelled out, for the same reason
  const double x = xs[r >> 1], e2 = __dmul_rn(eta, eta);
  const double D = Dk[k];
  const double a1 = x - D, a2 = -x - D;
  const double d1 = fma(a1, a1, e2), d2 = fma(a2, a2, e2);
  const double cr = 2.0 * __dadd_rn(a1 / d1, a2 / d2);
  const double ci = -2.0 * eta * __dadd_rn(1.0 / d1, 1.0 / d2);
  const double outr = fma(cr, tr, -__dmul_rn(ci, ti));
  const double outi = fma(ci, tr, __dmul_rn(cr, ti));
  U[(long)r * n_ov + k] = outr;
  U[(long)(r + 1) * n_ov + k] = outi;
}

// gemm2: out[r][P] = sum_k U[r][k] B[P][k] (mode 0), or the embedding [u - acc; -v - acc] (mode 1).
__global__ void __launch_bounds__(256) op_chain2_kernel(const double* __restrict__ U, const double* __restrict__ B,
                                                        int n_aux, long n_ov, int M, const double* __restrict__ V,
                                                        double* __restrict__ out, int mode,
                                                        const int* __restrict__ run_if) {
  if (run_if && *run_if == 0) return;
  __shared__ double As[CR][CK];
  __shared__ double Bs[32][CK + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, m0 = blockIdx.y * CR, r = m0 + w;
  const int q0 = blockIdx.x * 32, P = q0 + lane;
  double acc = 0.0;
  for (long k0 = 0; k0 < n_ov; k0 += CK) {
    const long k = k0 + lane;
    As[w][lane] = (r < M && k < n_ov) ? U[(long)r * n_ov + k] : 0.0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = w + 8 * u;
      Bs[q][lane] = (q0 + q < n_aux && k < n_ov) ? B[(long)(q0 + q) * n_ov + k] : 0.0;
    }
    __syncthreads();
    if (r < M)
#pragma unroll
      for (int kk = 0; kk < CK; ++kk) acc = fma(As[w][kk], Bs[lane][kk], acc);
    __syncthreads();
  }
  if (r >= M || P >= n_aux) return;
  if (mode == 1) {
    const double vin = V[(long)r * n_aux + P];
    acc = ((r & 1) ? -vin : vin) - acc;
  }
  out[(long)r * n_aux + P] = acc;
}

// ------------------------------------------------------------------ FP32 residue operator for few rows
// Mixed plans, up to eight rows (four right-hand sides: HOMO and LUMO jobs), where a 128-row tensor tile is padding.
// A MINRES iteration (operator and recurrences) of 1, 2, 3, 4 right-hand sides here, and of 3, 4, 5 in the tensor tiles:
//   126 x 190       23   23    24    25 us     34   35   34
//   629 x 4675      38   40    43    45        52   53   53
//   1259 x 18950    97  107   116   130        96   93   93
//   3024 x 109440  598  766  1135  1338       527  527  548
// So the line is right up to some 10 thousand pairs.  Beyond, the first product reads B at 6 TB/s and the second, whose
// rows of U come from L2 once per four rows of B, does not keep up with the tensor tiles (they took 1.6 ms a product
// before theirs was split in K); it stays for its FP32 operands, where the tiles hold 16 bits.
// Sums run in chains of 64 (gemm2) or one slice's 1/8 of the contraction (gemm1) before they are added.
constexpr int SKC = 128;             // gemm1 columns a CTA: 32 lanes x 4
template <int RM>
__global__ void __launch_bounds__(256) op_skinny1_kernel(const float* __restrict__ V, const float* __restrict__ B,
                                                         long ldb, const double* __restrict__ Dk, int n_ov, int n_aux,
                                                         const double* __restrict__ xs, float eta, int M,
                                                         float* __restrict__ U, const int* __restrict__ run_if) {
  if (run_if && *run_if == 0) return;
  __shared__ float Vs[256][RM];
  __shared__ float red[8][RM][SKC];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const long k = blockIdx.x * (long)SKC + 4 * lane;
  float tot[RM][4];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) tot[i][c] = 0.f;
  for (int p0 = 0; p0 < n_aux; p0 += 256) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RM; ++i)
      Vs[threadIdx.x][i] = (i < M && p0 + (int)threadIdx.x < n_aux) ? V[(long)i * n_aux + p0 + threadIdx.x] : 0.f;
    __syncthreads();
    const int pe = min(32, n_aux - p0 - 32 * sl);
    float acc[RM][4];
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][c] = 0.f;
    if (k < ldb)
#pragma unroll 8
      for (int t = 0; t < pe; ++t) {
        const float4 b = *reinterpret_cast<const float4*>(B + (long)(p0 + 32 * sl + t) * ldb + k);
#pragma unroll
        for (int i = 0; i < RM; ++i) {
          const float v = Vs[32 * sl + t][i];
          acc[i][0] = fmaf(v, b.x, acc[i][0]);
          acc[i][1] = fmaf(v, b.y, acc[i][1]);
          acc[i][2] = fmaf(v, b.z, acc[i][2]);
          acc[i][3] = fmaf(v, b.w, acc[i][3]);
        }
      }
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) tot[i][c] += acc[i][c];
  }
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) red[sl][i][4 * lane + c] = tot[i][c];
  __syncthreads();
  const float e2 = eta * eta;
  for (int it = threadIdx.x; it < SKC * (RM / 2); it += 256) {
    const int c = it % SKC, pr = it / SKC;
    const long kk = blockIdx.x * (long)SKC + c;
    if (2 * pr >= M || kk >= ldb) continue;
    float tr = 0.f, ti = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      tr += red[q][2 * pr][c];
      ti -= red[q][2 * pr + 1][c];
    }
    float ur = 0.f, ui = 0.f;                      // zero in the rows' padding
    if (kk < n_ov) {
      const double x = xs[pr], D = Dk[kk];
      const float a1 = (float)(x - D), a2 = (float)(-x - D);
      const float d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
      const float cr = 2.f * (a1 / d1 + a2 / d2);
      const float ci = -2.f * eta * (1.f / d1 + 1.f / d2);
      ur = cr * tr - ci * ti;
      ui = cr * ti + ci * tr;
    }
    U[(long)(2 * pr) * ldb + kk] = ur;
    U[(long)(2 * pr + 1) * ldb + kk] = ui;
  }
}

// Four rows P of B a CTA, its eight warps over the contraction.
template <int RM>
__global__ void __launch_bounds__(256) op_skinny2_kernel(const float* __restrict__ U, const float* __restrict__ B,
                                                         long ldb, int n_aux, int M, const float* __restrict__ V,
                                                         float* __restrict__ out, int mode,
                                                         const int* __restrict__ run_if) {
  if (run_if && *run_if == 0) return;
  __shared__ float red[8][4][RM];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, P0 = blockIdx.x * 4;
  float tot[4][RM];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int i = 0; i < RM; ++i) tot[p][i] = 0.f;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (long k0 = 4L * threadIdx.x; k0 < ldb; k0 += 1024 * 16) {
    float acc[4][RM];
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int i = 0; i < RM; ++i) acc[p][i] = 0.f;
#pragma unroll 2
    for (int t = 0; t < 16; ++t) {
      const long k = k0 + 1024L * t;
      if (k >= ldb) break;
      float4 b[4];
#pragma unroll
      for (int p = 0; p < 4; ++p)
        b[p] = P0 + p < n_aux ? *reinterpret_cast<const float4*>(B + (long)(P0 + p) * ldb + k) : zero;
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        if (i >= M) break;
        const float4 u = *reinterpret_cast<const float4*>(U + (long)i * ldb + k);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          acc[p][i] = fmaf(u.x, b[p].x, acc[p][i]);
          acc[p][i] = fmaf(u.y, b[p].y, acc[p][i]);
          acc[p][i] = fmaf(u.z, b[p].z, acc[p][i]);
          acc[p][i] = fmaf(u.w, b[p].w, acc[p][i]);
        }
      }
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int i = 0; i < RM; ++i) tot[p][i] += acc[p][i];
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int i = 0; i < RM; ++i) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) tot[p][i] += __shfl_xor_sync(0xffffffffu, tot[p][i], o);
      if (lane == 0) red[w][p][i] = tot[p][i];
    }
  __syncthreads();
  if (threadIdx.x < 4 * RM) {
    const int p = threadIdx.x / RM, i = threadIdx.x % RM;
    if (i < M && P0 + p < n_aux) {
      float s = 0.f;
      for (int q = 0; q < 8; ++q) s += red[q][p][i];
      const long at = (long)i * n_aux + P0 + p;
      out[at] = mode == 1 ? ((i & 1) ? -V[at] : V[at]) - s : s;
    }
  }
}

// ------------------------------------------------------------------ double-float GEMMs (refinement residual)
// A double x is carried as the FP32 pair (h, l), h = fl(x), l = fl(x - h): 48 significant bits.  A multiply-add
// s += a b takes the product exactly to FP32 pair precision (h*h by an FMA error term, plus the two cross terms)
// and adds it with Knuth's TwoSum; the low word collects every rounding error and is folded in once at the end.
// The _rn intrinsics keep the compiler from contracting the error-free steps into FMAs.
__device__ __forceinline__ void df_split(double x, float& h, float& l) {
  h = __double2float_rn(x);
  l = __double2float_rn(x - (double)h);
}

__device__ __forceinline__ void df_mac(float ah, float al, float bh, float bl, float& sh, float& sl) {
  const float ph = __fmul_rn(ah, bh);
  float pe = __fmaf_rn(ah, bh, -ph);
  pe = __fmaf_rn(ah, bl, pe);
  pe = __fmaf_rn(al, bh, pe);
  const float t = __fadd_rn(sh, ph);
  const float v = __fsub_rn(t, sh);
  const float e = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, v)), __fsub_rn(ph, v));
  sl = __fadd_rn(sl, __fadd_rn(e, pe));
  sh = t;
}

// df gemm1: U[r][k] for rows r of V [2nr][n_aux] (FP64) against B = Bh + Bl [n_aux][n_ov], then the complex
// weights c_k(x_j) of the pair (2j, 2j+1) as in op_gemm1 mode 0; U in FP64.
__global__ void __launch_bounds__(NT) op_gemm1_df_kernel(const double* __restrict__ V, const float* __restrict__ Bh,
                                                         const float* __restrict__ Bl, long ldh,
                                                         const double* __restrict__ Dk,
                                                         long n_ov, int n_aux,
                                                         const double* __restrict__ xs, double eta, int nr,
                                                         double* __restrict__ U) {
  __shared__ float Ah_s[TK][TM + 4], Al_s[TK][TM + 4];
  __shared__ float Bh_s[TK][TN + 4], Bl_s[TK][TN + 4];
  const int M = 2 * nr;
  const int m0 = blockIdx.y * TM;
  const long k0c = (long)blockIdx.x * TN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float ah_[4][4], al_[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) ah_[i][j] = al_[i][j] = 0.f;
  for (int p0 = 0; p0 < n_aux; p0 += TK) {
    {
      const int r = tid >> 2, k4 = (tid & 3) * 4;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int P = p0 + k4 + u;
        float h = 0.f, l = 0.f;
        if (m0 + r < M && P < n_aux) df_split(V[(long)(m0 + r) * n_aux + P], h, l);
        Ah_s[k4 + u][r] = h;
        Al_s[k4 + u][r] = l;
      }
      const int kr = tid >> 4, c4 = (tid & 15) * 4;
      const int P = p0 + kr;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const long k = k0c + c4 + u;
        const bool in = P < n_aux && k < n_ov;
        Bh_s[kr][c4 + u] = in ? Bh[(long)P * ldh + k] : 0.f;
        Bl_s[kr][c4 + u] = in ? Bl[(long)P * n_ov + k] : 0.f;
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < TK; ++kk) {
      float a_h[4], a_l[4], b_h[4], b_l[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = 2 * ty + (i & 1) + 32 * (i >> 1);
        a_h[i] = Ah_s[kk][c];
        a_l[i] = Al_s[kk][c];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        b_h[j] = Bh_s[kk][tx + 16 * j];
        b_l[j] = Bl_s[kk][tx + 16 * j];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) df_mac(a_h[i], a_l[i], b_h[j], b_l[j], ah_[i][j], al_[i][j]);
    }
    __syncthreads();
  }
  const double e2 = eta * eta;
#pragma unroll
  for (int ip = 0; ip < 2; ++ip) {
    const int r = m0 + 2 * ty + 32 * ip;
    if (r >= M) continue;
    const double x = xs[r >> 1];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const long k = k0c + tx + 16 * j;
      if (k >= n_ov) continue;
      const double tr = (double)ah_[2 * ip][j] + (double)al_[2 * ip][j];
      const double ti = -((double)ah_[2 * ip + 1][j] + (double)al_[2 * ip + 1][j]);
      const double D = Dk[k];
      const double a1 = x - D, a2 = -x - D;
      const double d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
      const double cr = 2.0 * (a1 / d1 + a2 / d2);
      const double ci = -2.0 * eta * (1.0 / d1 + 1.0 / d2);
      U[(long)r * n_ov + k] = cr * tr - ci * ti;
      U[(long)(r + 1) * n_ov + k] = cr * ti + ci * tr;
    }
  }
}

// df gemm2: acc[r][P] = sum_k U[r][k] B[P][k]; out = the real embedding [u - acc_re; -v - acc_im] (op_gemm2 mode 1), or,
// with grid.z > 1 K ranges of `range` columns, the range's sums in FP64 to part [grid.z][M][n_aux] (df_part_kernel).
// Bound by the FP32 pipes, 12 instructions a multiply-add; the next tile's loads run under a tile's arithmetic.  One range
// and loads before each tile: 1.55 ms for 25 right-hand sides at N_aux 630, K 4750 (20 CTAs), 4.3 for 231 at 1008 and
// 12160, 15.8 for 226 at 1800 and 26496; now 0.17, 3.0 and 12.3.
__global__ void __launch_bounds__(NT) op_gemm2_df_kernel(const double* __restrict__ U, const float* __restrict__ Bh,
                                                         const float* __restrict__ Bl, long ldh, int n_aux, long n_ov,
                                                         int nr,
                                                         const double* __restrict__ V, double* __restrict__ out,
                                                         int range, double* __restrict__ part) {
  __shared__ float Ah_s[TK][TM + 4], Al_s[TK][TM + 4];
  __shared__ float Bh_s[TK][TN + 4], Bl_s[TK][TN + 4];
  const int M = 2 * nr;
  const int m0 = blockIdx.y * TM;
  const int q0 = blockIdx.x * TN;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float ah_[4][4], al_[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) ah_[i][j] = al_[i][j] = 0.f;
  const int lr = tid >> 2, lk = (tid & 3) * 4;
  const long kbeg = (long)blockIdx.z * range, kend = kbeg + range < n_ov ? kbeg + range : n_ov;
  double av[4];
  float bh[4], bl[4];
  auto load = [&](long k0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long k = k0 + lk + u;
      const bool in = q0 + lr < n_aux && k < kend;
      av[u] = m0 + lr < M && k < kend ? U[(long)(m0 + lr) * n_ov + k] : 0.0;
      bh[u] = in ? Bh[(long)(q0 + lr) * ldh + k] : 0.f;
      bl[u] = in ? Bl[(long)(q0 + lr) * n_ov + k] : 0.f;
    }
  };
  load(kbeg);
  for (long k0 = kbeg; k0 < kend; k0 += TK) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float h, l;
      df_split(av[u], h, l);
      Ah_s[lk + u][lr] = h;
      Al_s[lk + u][lr] = l;
      Bh_s[lk + u][lr] = bh[u];
      Bl_s[lk + u][lr] = bl[u];
    }
    if (k0 + TK < kend) load(k0 + TK);
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < TK; ++kk) {
      float a_h[4], a_l[4], b_h[4], b_l[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = 2 * ty + (i & 1) + 32 * (i >> 1);
        a_h[i] = Ah_s[kk][c];
        a_l[i] = Al_s[kk][c];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        b_h[j] = Bh_s[kk][tx + 16 * j];
        b_l[j] = Bl_s[kk][tx + 16 * j];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) df_mac(a_h[i], a_l[i], b_h[j], b_l[j], ah_[i][j], al_[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = m0 + 2 * ty + (i & 1) + 32 * (i >> 1);
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int P = q0 + tx + 16 * j;
      if (P >= n_aux) continue;
      const double v = (double)ah_[i][j] + (double)al_[i][j];
      if (gridDim.z > 1) {
        part[((long)blockIdx.z * M + r) * n_aux + P] = v;
        continue;
      }
      const double vin = V[(long)r * n_aux + P];
      out[(long)r * n_aux + P] = ((r & 1) ? -vin : vin) - v;
    }
  }
}

// out[r][P] = (r odd ? -V : V)[r][P] - sum of the ranges' parts, in order.
__global__ void df_part_kernel(const double* __restrict__ part, int ks, int M, int n_aux, const double* __restrict__ V,
                               double* __restrict__ out) {
  const long n = (long)M * n_aux;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int z = 0; z < ks; ++z) v += part[z * n + i];
    out[i] = ((i / n_aux) & 1 ? -V[i] : V[i]) - v;
  }
}

__global__ void df_split_kernel(const double* __restrict__ x, long n, float* __restrict__ h, float* __restrict__ l) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
    float hh, ll;
    df_split(x[i], hh, ll);
    if (h) h[i] = hh;
    l[i] = ll;
  }
}

}  // namespace

void launch_df_split(const double* x, long n, float* h, float* l, cudaStream_t s) {
  if (n > 0) df_split_kernel<<<1216, 256, 0, s>>>(x, n, h, l);
}

void launch_op_gemm1_df(const double* V, const float* Bh, const float* Bl, long ldh, const double* Dk, long n_ov,
                        int n_aux, const double* x, double eta, int nr, double* U, cudaStream_t s) {
  const dim3 grid((unsigned)((n_ov + TN - 1) / TN), (2 * nr + TM - 1) / TM);
  if (nr > 0) op_gemm1_df_kernel<<<grid, NT, 0, s>>>(V, Bh, Bl, ldh, Dk, n_ov, n_aux, x, eta, nr, U);
}

// Few right-hand sides leave most SMs without a tile, and a batch's tiles fill their last round badly: K ranges of at
// least 512 columns, the fewest that fill nine tenths of the rounds (two CTAs an SM), or those that fill them best.
int op_gemm2_df_ranges(int n_aux, long n_ov, int nr) {
  const long tiles = (long)((n_aux + TN - 1) / TN) * ((2 * nr + TM - 1) / TM), slots = 304;
  int best = 1;
  double best_fill = 0.0;
  for (int ks = 1; ks <= 16; ++ks) {
    if (ks > 1 && (ks * tiles > kDfPartTiles || n_ov / ks < 512)) break;
    const long rounds = (ks * tiles + slots - 1) / slots;
    const double fill = (double)(ks * tiles) / (double)(rounds * slots);
    if (fill > best_fill) {
      best_fill = fill;
      best = ks;
    }
    if (fill >= 0.9) break;
  }
  return best;
}

void launch_op_gemm2_df(const double* U, const float* Bh, const float* Bl, long ldh, int n_aux, int n_ov, int nr,
                        const double* V, double* out, double* part, cudaStream_t s) {
  if (nr <= 0) return;
  const int ks = op_gemm2_df_ranges(n_aux, n_ov, nr), range = ((n_ov + ks - 1) / ks + TK - 1) / TK * TK;
  const dim3 grid((n_aux + TN - 1) / TN, (2 * nr + TM - 1) / TM, ks);
  op_gemm2_df_kernel<<<grid, NT, 0, s>>>(U, Bh, Bl, ldh, n_aux, (long)n_ov, nr, V, out, range, part);
  if (ks > 1) df_part_kernel<<<608, 256, 0, s>>>(part, ks, 2 * nr, n_aux, V, out);
}

void launch_deriv_resonant(const double* V64, const double* B, long n_ov, int n_aux, const double* Dsort,
                           const int* kidx, const double* xs, int nr, double eta, double cut, double* dw,
                           cudaStream_t s) {
  if (nr > 0) deriv_resonant_kernel<<<nr, 256, 0, s>>>(V64, B, n_ov, n_aux, Dsort, kidx, xs, eta, cut, dw);
}

// ------------------------------------------------------------------ launchers
template <typename T>
void launch_cholesky(T* base, int n, long stride, int batch, int* info, cudaStream_t s) {
  cholesky_kernel<T><<<batch, CH_THREADS, 0, s>>>(base, n, stride, info);
}

void launch_pi_syrk(const double* B, const double* Dk, long n_ov, int n_aux, const double* xi, int n_xi, double* out,
                    int mode, cudaStream_t s, const int* flags) {
  const int nb = (n_aux + TM - 1) / TM;
  pi_syrk_kernel<<<dim3(nb * (nb + 1) / 2, n_xi), NT, 0, s>>>(B, Dk, n_ov, n_aux, xi, out, mode, flags);
}

cudaError_t launch_tri_inv(const double* L, long stride, int n, int batch, double* X, long xstride, cudaStream_t s) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidValue;
  const int smem = (int)sizeof(double) * 2 * 64 * 65;
  const cudaError_t e = cudaFuncSetAttribute(tri_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  tri_inv_kernel<<<dim3((n + 63) / 64, batch), NT, smem, s>>>(L, stride, n, X, xstride);
  return cudaGetLastError();
}

cudaError_t launch_w_minus_norm(const double* Bn, int n, long R, int n_cols, double* W, cudaStream_t s) {
  if (R > 0) w_minus_norm_kernel<<<(unsigned)(R < 4 * 4096 ? (R + 3) / 4 : 4096), 128, 0, s>>>(Bn, n, R, n_cols, W);
  return cudaGetLastError();
}

int trsm_w_default_ctas() {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  return 2 * (nsm > 0 ? nsm : 148);
}

template <typename T>
size_t trsm_w_scratch_elems(int n, int n_cta) {
  return (size_t)n_cta * (size_t)(((n + 63) / 64) * 64) * 64;
}

template <typename T>
cudaError_t launch_trsm_w(const T* Lbase, long Lstride, int n, int n_g, const int* g_out, const T* Bn, int R,
                          double* W, int w_ld, T* scratch, int n_cta, cudaStream_t s) {
  size_t smem = sizeof(T) * (2 * TK * (TM + 4) + 2 * 64 * 65) + sizeof(double) * 2 * 16 * 64;
  cudaError_t e = cudaFuncSetAttribute(trsm_w_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  long items = (long)n_g * ((R + 63) / 64);
  int grid = (int)(items < n_cta ? items : n_cta);
  if (grid <= 0) return cudaSuccess;
  // cudaLaunchKernel returns this launch's own status (an earlier error pending on the thread is left alone)
  void* args[] = {(void*)&Lbase, (void*)&Lstride, (void*)&n, (void*)&n_g, (void*)&g_out, (void*)&Bn,
                  (void*)&R, (void*)&W, (void*)&w_ld, (void*)&scratch};
  return cudaLaunchKernel((const void*)trsm_w_kernel<T>, dim3(grid), dim3(NT), args, smem, s);
}

void launch_op_gemm1(const double* V, const double* B, const double* Dk, long n_ov, int n_aux, const double* x,
                     double eta, int nr, double* U, cudaStream_t s, const int* run_if) {
  const dim3 grid((unsigned)((n_ov + 31) / 32), (2 * nr + CR - 1) / CR);
  if (nr > 0) op_chain1_kernel<<<grid, 256, 0, s>>>(V, B, Dk, n_ov, n_aux, x, eta, 2 * nr, U, run_if);
}

void launch_op_gemm2(const double* U, const double* B, int n_aux, long n_ov, int nr, const double* V, double* out,
                     int mode, cudaStream_t s, const int* run_if) {
  const dim3 grid((n_aux + 31) / 32, (2 * nr + CR - 1) / CR);
  if (nr > 0) op_chain2_kernel<<<grid, 256, 0, s>>>(U, B, n_aux, n_ov, 2 * nr, V, out, mode, run_if);
}

void launch_op_skinny(const float* V, const float* B, long ldb, const double* Dk, int n_ov, int n_aux, const double* x,
                      float eta, int nr, float* U, float* S, int mode, cudaStream_t s, const int* run_if) {
  const unsigned g1 = (unsigned)((ldb + SKC - 1) / SKC), g2 = (n_aux + 3) / 4;
  if (nr == 1) {
    op_skinny1_kernel<2><<<g1, 256, 0, s>>>(V, B, ldb, Dk, n_ov, n_aux, x, eta, 2, U, run_if);
    op_skinny2_kernel<2><<<g2, 256, 0, s>>>(U, B, ldb, n_aux, 2, V, S, mode, run_if);
  } else if (nr == 2) {
    op_skinny1_kernel<4><<<g1, 256, 0, s>>>(V, B, ldb, Dk, n_ov, n_aux, x, eta, 4, U, run_if);
    op_skinny2_kernel<4><<<g2, 256, 0, s>>>(U, B, ldb, n_aux, 4, V, S, mode, run_if);
  } else if (nr <= kSkinnyRhs) {
    op_skinny1_kernel<8><<<g1, 256, 0, s>>>(V, B, ldb, Dk, n_ov, n_aux, x, eta, 2 * nr, U, run_if);
    op_skinny2_kernel<8><<<g2, 256, 0, s>>>(U, B, ldb, n_aux, 2 * nr, V, S, mode, run_if);
  }
}

template <typename T>
void launch_deriv(const T* V, const T* B, const double* Dk, long n_ov, int n_aux, const double* x, double eta, int nr,
                  double* dw, double cut, long ldb, cudaStream_t s) {
  const dim3 grid((unsigned)((n_ov + TN - 1) / TN), (2 * nr + TM - 1) / TM);
  if (nr > 0) deriv_kernel<T><<<grid, NT, 0, s>>>(V, B, Dk, n_ov, n_aux, x, eta, nr, dw, cut, ldb);
}

template void launch_deriv<double>(const double*, const double*, const double*, long, int, const double*, double, int,
                                   double*, double, long, cudaStream_t);
template void launch_deriv<float>(const float*, const float*, const double*, long, int, const double*, double, int,
                                  double*, double, long, cudaStream_t);
template void launch_cholesky<double>(double*, int, long, int, int*, cudaStream_t);
template size_t trsm_w_scratch_elems<double>(int, int);
template cudaError_t launch_trsm_w<double>(const double*, long, int, int, const int*, const double*, int, double*, int,
                                           double*, int, cudaStream_t);

}  // namespace gw

// =====================================================================================================
// W table from caller-supplied Cholesky factors without any device allocation.
//
// Some callers cannot allocate device memory when they call into this library: a serving process that
// reserves all GPU memory for its own pool at start-up, a host application whose allocator forbids
// cudaMalloc after initialisation, or code on a latency-critical path where an allocation (which may
// synchronise the device) is not acceptable.  gw_w_table_noalloc gives them the W-table triangular solves
// with the per-CTA work space taken from the fixed array below instead of cudaMalloc.
// =====================================================================================================
#define GW_NOALLOC_SCRATCH_BYTES (32u << 20)   // 32 MiB, held by every GPU that loads the library
#define GW_NOALLOC_MAX_MATS 4096

static __device__ __align__(256) unsigned char g_noalloc_scratch[GW_NOALLOC_SCRATCH_BYTES];
static __device__ __align__(256) int g_noalloc_index[GW_NOALLOC_MAX_MATS];

namespace {
struct NoallocDevice {
  void* scratch = nullptr;
  int* index = nullptr;
  bool ready = false;
};
std::mutex g_noalloc_mu;
NoallocDevice g_noalloc_dev[128];
int g_noalloc_host_index[GW_NOALLOC_MAX_MATS];
}  // namespace

extern "C" gw_status gw_w_table_noalloc(const double* L, int n_aux, int n_mats, const double* Bn, int n_rows,
                                        double* W, int w_ld, void* stream) {
  if (!L || !Bn || !W || n_aux <= 0 || n_mats <= 0 || n_rows <= 0 || w_ld < n_mats) return GW_ERR_ARG;
  if (n_mats > GW_NOALLOC_MAX_MATS) return GW_ERR_ARG;
  const size_t slice = (size_t)((n_aux + 63) / 64) * 64 * 64 * sizeof(double);
  if (slice > GW_NOALLOC_SCRATCH_BYTES) return GW_ERR_ARG;   // n_aux beyond 65536
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return GW_ERR_CUDA;
  NoallocDevice& d = g_noalloc_dev[dev];
  {
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!d.ready) {
      // once per device, with that device current: device addresses of the fixed arrays and the
      // frequency index table 0, 1, 2, ... (a synchronous copy, before any stream capture)
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) return GW_ERR_CUDA;
      d.scratch = p;
      if (cudaGetSymbolAddress(&p, g_noalloc_index) != cudaSuccess) return GW_ERR_CUDA;
      d.index = static_cast<int*>(p);
      for (int i = 0; i < GW_NOALLOC_MAX_MATS; ++i) g_noalloc_host_index[i] = i;
      if (cudaMemcpyToSymbol(g_noalloc_index, g_noalloc_host_index, sizeof(g_noalloc_host_index)) != cudaSuccess)
        return GW_ERR_CUDA;
      d.ready = true;
    }
  }
  int n_cta = (int)(GW_NOALLOC_SCRATCH_BYTES / slice);
  const int full = gw::trsm_w_default_ctas();
  n_cta = n_cta < full ? n_cta : full;
  // the status is this launch's own (cudaFuncSetAttribute, then cudaLaunchKernel): an error that other work left
  // pending on the thread is neither reported here nor cleared
  const cudaError_t e = gw::launch_trsm_w<double>(L, (long)n_aux * n_aux, n_aux, n_mats, d.index, Bn, n_rows, W,
                                                  w_ld, static_cast<double*>(d.scratch), n_cta,
                                                  static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? GW_OK : GW_ERR_CUDA;
}
