// Spectral-decomposition route (Sec. 2.2 and 3.2): the Casida problem in its Hermitian form
//   M T = T Omega^2,   M = D^1/2 (D + 4K) D^1/2,   K = B_ia^T B_ia   (N_ov x N_ov, symmetric positive definite),
// diagonalised by a parallel cyclic Jacobi method in FP64, then the pole weights
//   w2[t][m][s] = (b_tm . V_s)^2 / (2 Omega_s),   V = 2 B_ia D^1/2 T,
// so that Sigma^c_nn(omega) = sum_m sum_s w2 / (omega - e_m + Omega_s - i eta)  (m occupied)
//                           + sum_m sum_s w2 / (omega - e_m - Omega_s + i eta)  (m virtual).
// Jacobi rounds use the round-robin pairing of the indices: every round rotates N/2 disjoint pairs (p, q), each
// by the angle that zeroes M_pq, applied to rows (M <- J^T M), columns (M <- M J) and the eigenvectors (T <- T J).
//
// N <= 8192 first tries a direct route: Householder tridiagonalisation in one cooperative kernel, eigenvalues by
// bisection, eigenvectors by twisted factorisations and back-transformation, then the refinement of Ogita and Aishima
// ("Iterative refinement for symmetric eigenvalue decomposition", 2018) on exact digit products until the same
// off-diagonal criterion holds that ends the Jacobi sweeps.  Where it does not (clusters too tight for the twisted
// vectors), the sweeps take over.  At N 760 the sweeps take 240 ms (24 thousand launches, each a pass over the matrix),
// the direct route 11 ms: tridiagonalisation 5.3, back-transformation 2.1, bisection 1.5, twisted vectors 0.7, the
// products of two refinement passes 0.9.  N >= 8, where a warp has a row to share; 8192 is what the vectors of one CTA
// allow in shared memory.
#include "gw_internal.cuh"
#include "tc_ptx.cuh"

#include <cmath>

namespace gw {
namespace {

constexpr int ST = 16;     // SIMT tile edge of the small GEMMs

// Round-robin pairing of 2h players (index 2h - 1 is fixed): pair k of round r.
__device__ __forceinline__ void rr_pair(int r, int k, int h, int& p, int& q) {
  const int m = 2 * h - 1;
  if (k == 0) {
    p = m;
    q = r % m;
  } else {
    p = (r + k) % m;
    q = (r - k + m) % m;
  }
  if (p > q) { const int t = p; p = q; q = t; }
}

// M = D^1/2 (D + 4 B^T B) D^1/2, padded to Np (extra indices: identity, never coupled).
__global__ void casida_matrix_kernel(const double* __restrict__ B, const double* __restrict__ Dk, int n_aux, int N,
                                     int Np, double* __restrict__ M) {
  __shared__ double As[ST][ST + 1], Bs[ST][ST + 1];
  const int i = blockIdx.y * ST + threadIdx.y, j = blockIdx.x * ST + threadIdx.x;
  double acc = 0.0;
  for (int p0 = 0; p0 < n_aux; p0 += ST) {
    const int pa = p0 + threadIdx.x, pb = p0 + threadIdx.y;
    As[threadIdx.y][threadIdx.x] = (i < N && pa < n_aux) ? B[(long)pa * N + i] : 0.0;
    Bs[threadIdx.y][threadIdx.x] = (j < N && pb < n_aux) ? B[(long)pb * N + j] : 0.0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < ST; ++u) acc += As[threadIdx.y][u] * Bs[u][threadIdx.x];
    __syncthreads();
  }
  if (i < Np && j < Np) {
    double v;
    if (i < N && j < N) v = sqrt(Dk[i]) * (4.0 * acc + (i == j ? Dk[i] : 0.0)) * sqrt(Dk[j]);
    else v = (i == j) ? 1.0 : 0.0;
    M[(long)i * Np + j] = v;
  }
}

__global__ void identity_kernel(double* __restrict__ T, int Np) {
  const long n = (long)Np * Np;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x)
    T[e] = (e / Np == e % Np) ? 1.0 : 0.0;
}

// Rotation of every pair of round r: (c, s) zeroing M_pq, stored per pair.
__global__ void jacobi_angles_kernel(const double* __restrict__ M, int Np, int r, double* __restrict__ cs) {
  const int h = Np / 2;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= h) return;
  int p, q;
  rr_pair(r, k, h, p, q);
  const double apq = M[(long)p * Np + q], app = M[(long)p * Np + p], aqq = M[(long)q * Np + q];
  double c = 1.0, s = 0.0;
  if (apq != 0.0 && fabs(apq) > 1e-300) {
    const double tau = (aqq - app) / (2.0 * apq);
    const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
    c = 1.0 / sqrt(1.0 + t * t);
    s = t * c;
  }
  cs[2 * k] = c;
  cs[2 * k + 1] = s;
}

// Rows p, q of M for every pair: (M_p, M_q) <- (c M_p - s M_q, s M_p + c M_q).
__global__ void jacobi_rows_kernel(double* __restrict__ M, int Np, int r, const double* __restrict__ cs) {
  const int h = Np / 2, k = blockIdx.y;
  int p, q;
  rr_pair(r, k, h, p, q);
  const double c = cs[2 * k], s = cs[2 * k + 1];
  if (s == 0.0) return;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < Np; j += gridDim.x * blockDim.x) {
    const double a = M[(long)p * Np + j], b = M[(long)q * Np + j];
    M[(long)p * Np + j] = c * a - s * b;
    M[(long)q * Np + j] = s * a + c * b;
  }
}

// Columns p, q of X (M, or the eigenvectors T): (X_.p, X_.q) <- (c X_.p - s X_.q, s X_.p + c X_.q).
__global__ void jacobi_cols_kernel(double* __restrict__ X, int Np, int r, const double* __restrict__ cs) {
  const int h = Np / 2, k = blockIdx.y;
  int p, q;
  rr_pair(r, k, h, p, q);
  const double c = cs[2 * k], s = cs[2 * k + 1];
  if (s == 0.0) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < Np; i += gridDim.x * blockDim.x) {
    const double a = X[(long)i * Np + p], b = X[(long)i * Np + q];
    X[(long)i * Np + p] = c * a - s * b;
    X[(long)i * Np + q] = s * a + c * b;
  }
}

// off[0] += sum of squares of the off-diagonal elements, off[1] += of the diagonal ones.
__global__ void offdiag_kernel(const double* __restrict__ M, int Np, double* __restrict__ off) {
  __shared__ double red[2][32];
  double o = 0.0, d = 0.0;
  const long n = (long)Np * Np;
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < n; e += (long)gridDim.x * blockDim.x) {
    const double v = M[e];
    if (e / Np == e % Np) d += v * v; else o += v * v;
  }
  for (int w = 16; w > 0; w >>= 1) {
    o += __shfl_xor_sync(0xffffffffu, o, w);
    d += __shfl_xor_sync(0xffffffffu, d, w);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = o;
    red[1][threadIdx.x >> 5] = d;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double so = 0.0, sd = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { so += red[0][w]; sd += red[1][w]; }
    atomicAdd(off, so);
    atomicAdd(off + 1, sd);
  }
}

// V[P][s] = 2 sum_k B[P][k] sqrt(D_k) T[k][s]  (the eigenvectors in the auxiliary basis), s < N.
__global__ void casida_v_kernel(const double* __restrict__ B, const double* __restrict__ Dk,
                                const double* __restrict__ T, int n_aux, int N, int Np, double* __restrict__ V) {
  __shared__ double As[ST][ST + 1], Bs[ST][ST + 1];
  const int P = blockIdx.y * ST + threadIdx.y, sc = blockIdx.x * ST + threadIdx.x;
  double acc = 0.0;
  for (int k0 = 0; k0 < N; k0 += ST) {
    const int ka = k0 + threadIdx.x, kb = k0 + threadIdx.y;
    As[threadIdx.y][threadIdx.x] = (P < n_aux && ka < N) ? B[(long)P * N + ka] * sqrt(Dk[ka]) : 0.0;
    Bs[threadIdx.y][threadIdx.x] = (sc < N && kb < N) ? T[(long)kb * Np + sc] : 0.0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < ST; ++u) acc += As[threadIdx.y][u] * Bs[u][threadIdx.x];
    __syncthreads();
  }
  if (P < n_aux && sc < N) V[(long)P * N + sc] = 2.0 * acc;
}

// w2[r][s] = (b_r . V_s)^2 / (2 Omega_s) for the rows r of Bn [R][n_aux].
__global__ void casida_w2_kernel(const double* __restrict__ Bn, const double* __restrict__ V,
                                 const double* __restrict__ Om, int n_aux, int R, int N, double* __restrict__ w2) {
  __shared__ double As[ST][ST + 1], Bs[ST][ST + 1];
  const int r = blockIdx.y * ST + threadIdx.y, sc = blockIdx.x * ST + threadIdx.x;
  double acc = 0.0;
  for (int p0 = 0; p0 < n_aux; p0 += ST) {
    const int pa = p0 + threadIdx.x, pb = p0 + threadIdx.y;
    As[threadIdx.y][threadIdx.x] = (r < R && pa < n_aux) ? Bn[(long)r * n_aux + pa] : 0.0;
    Bs[threadIdx.y][threadIdx.x] = (sc < N && pb < n_aux) ? V[(long)pb * N + sc] : 0.0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < ST; ++u) acc += As[threadIdx.y][u] * Bs[u][threadIdx.x];
    __syncthreads();
  }
  if (r < R && sc < N) w2[(long)r * N + sc] = acc * acc / (2.0 * Om[sc]);
}

__global__ void casida_omega_kernel(const double* __restrict__ M, int Np, int N, double* __restrict__ Om) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < N) Om[s] = sqrt(fmax(M[(long)s * Np + s], 0.0));
}

// ------------------------------------------------------------------ tridiagonalisation
// A (symmetric, full storage, row length ld, overwritten) = Q T Q^T by N - 2 Householder steps, all CTAs together, CTA c
// holding rows c, c + grid, ... (in shared memory when they fit, SM).  Step k: column k is brought up to date; one pass
// over the rows applies the previous reflector's rank-2 update and forms t = A x and a = A e_{k+1} with the raw column x
// (A v = t - alpha a for the reflector v = x - alpha e_{k+1}, so its scalars are formed while the barrier fills); after
// the one grid barrier of the step every CTA forms v and w for itself.  H[k][.] = v_k (zero up to k), beta[k]; d, e the
// diagonals of T.  Bound by a step's chain of latencies (two L2 round trips, barrier, block sums) and the FP64 vector
// work every CTA repeats; the pass, three FMAs an element over all SMs, is the smaller part.
// bar: zeroed counter; every wait gives up after ptx::kWaitNs and sets *err.
__device__ void grid_arrive(unsigned* bar) {      // after a __syncthreads, one thread
  __threadfence();
  atomicAdd(bar, 1u);
}

__device__ bool grid_wait(unsigned* bar, unsigned target, int* err) {
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    int ok = 1;
    unsigned long long t0 = 0;
    for (unsigned it = 1; *(volatile unsigned*)bar < target; ++it) {
      if ((it & 63) != 0) continue;
      const unsigned long long t = ptx::globaltimer_ns();
      if (t0 == 0) t0 = t;
      if (*(volatile int*)err != 0 || t - t0 > ptx::kWaitNs) {
        atomicCAS(err, 0, 81);
        ok = 0;
        break;
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

constexpr int TRI_T = 256;

// Block sum, the same order in every CTA.  Lanes of warp 0 add the eight warps' values, so that the FP64 pipe (16 clocks
// a warp instruction) sees 13 instructions and not 13 a warp.  Barriers on both sides of red and res.
__device__ double tri_sum(double v, double* red, double* res) {
  red[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = red[threadIdx.x];
#pragma unroll
    for (int i = 1; i < TRI_T / 32; ++i) t += red[threadIdx.x + 32 * i];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) *res = t;
  }
  __syncthreads();
  return *res;
}

template <bool SM>
__global__ void __launch_bounds__(TRI_T, 1) tridiag_kernel(double* A, int N, long ld, double* __restrict__ H,
                                                           double* __restrict__ beta, double* __restrict__ d,
                                                           double* __restrict__ e, double* p_buf, unsigned* bar,
                                                           int* err) {
  extern __shared__ double tsm[];
  double* v = tsm;             // previous reflector and its w
  double* w = v + N;
  double* x = w + N;           // the column
  double* rows = x + N;        // SM: row r of this CTA (matrix row r grid + blockIdx) at r N
  __shared__ double red[TRI_T], res[2], scal[2];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, G = gridDim.x;
  const int nr = (N - (int)blockIdx.x + G - 1) / G;
  for (int i = tid; i < N; i += TRI_T) {
    v[i] = w[i] = 0.0;
    x[i] = A[i];
  }
  if (SM)
    for (int r = wid; r < nr; r += TRI_T / 32)
      for (int j = lane; j < N; j += 32) rows[(long)r * N + j] = A[((long)r * G + blockIdx.x) * ld + j];
  __syncthreads();
  for (int k = 0; k < N; ++k) {
    const double vk = v[k], wk = w[k];
    double s = 0.0;
    for (int i = k + tid; i < N; i += TRI_T) {
      const double a = x[i] - v[i] * wk - w[i] * vk;
      x[i] = a;
      if (i >= k + 2) s = fma(a, a, s);
    }
    __syncthreads();
    double* p = p_buf + (long)(k & 1) * 2 * N;
    if (k + 2 < N) {
      for (int r = wid; r < nr; r += TRI_T / 32) {
        const int i = r * G + blockIdx.x;
        if (i <= k) continue;
        double* Ag = A + (long)i * ld;
        double* Ai = SM ? rows + (long)r * N : Ag;
        const double vi = v[i], wi = w[i];
        const bool next = SM && i == k + 1;          // the next column, for all CTAs
        double t = 0.0, a1 = 0.0;
        for (int j0 = k + 1 + lane; j0 < N; j0 += 128) {
          double a[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = j0 + 32 * u;
            a[u] = j < N ? (SM ? Ai[j] : __ldcg(Ai + j)) : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = j0 + 32 * u;
            if (j < N) {
              a[u] = fma(-vi, w[j], a[u]);
              a[u] = fma(-wi, v[j], a[u]);
              t = fma(a[u], x[j], t);
              if (SM) Ai[j] = a[u];
              if (!SM || next) __stcg(Ag + j, a[u]);
            }
          }
          if (j0 == k + 1) a1 = a[0];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) {
          __stcg(p + i, t);
          __stcg(p + N + i, a1);
        }
      }
      __syncthreads();
      if (tid == 0) grid_arrive(bar);
    }
    const double rest = tri_sum(s, red, res);
    if (tid < 32) {                                  // the reflector's scalars, one warp
      const double x1 = k + 1 < N ? x[k + 1] : 0.0;
      double b = 0.0, alpha = x1;
      if (rest > 0.0) {
        const double sig = fma(x1, x1, rest);
        alpha = x1 > 0.0 ? -sqrt(sig) : sqrt(sig);
        b = 1.0 / (sig - alpha * x1);
      }
      if (tid == 0) {
        scal[0] = b;
        scal[1] = alpha;
        if (blockIdx.x == 0) {
          d[k] = x[k];
          if (k + 1 < N) e[k] = alpha;
          beta[k] = b;
        }
      }
    }
    if (k + 2 >= N) {
      if (k + 1 < N && blockIdx.x == (N - 1) % G && tid == 0) {      // only the last diagonal element is left
        const double a = SM ? rows[(long)((N - 1) / G) * N + N - 1] : __ldcg(A + (long)(N - 1) * ld + N - 1);
        d[N - 1] = a - 2.0 * v[N - 1] * w[N - 1];
        beta[N - 1] = 0.0;
      }
      return;
    }
    if (!grid_wait(bar, (unsigned)(k + 1) * G, err)) return;         // its __syncthreads also publishes scal
    const double b = scal[0], alpha = scal[1];
    const bool mine = (int)blockIdx.x == k % G;
    s = 0.0;
    for (int i = k + 1 + tid; i < N; i += TRI_T) {
      const double q = b * (__ldcg(p + i) - alpha * __ldcg(p + N + i));
      const double nx = __ldcg(A + (long)(k + 1) * ld + i);
      const double vi = i > k + 1 ? x[i] : (b != 0.0 ? x[i] - alpha : 0.0);
      w[i] = q;
      v[i] = vi;
      x[i] = nx;
      if (mine) H[(long)k * ld + i] = vi;
      s = fma(q, vi, s);
    }
    if (mine)
      for (int i = tid; i <= k; i += TRI_T) H[(long)k * ld + i] = 0.0;
    const double K = 0.5 * b * tri_sum(s, red, res + 1);
    for (int i = k + 1 + tid; i < N; i += TRI_T) w[i] = fma(-K, v[i], w[i]);
    __syncthreads();
  }
}

// Eigenvalue s of T by (L + 1)-section on the count of negative pivots, as sign changes of the scaled characteristic
// recurrence p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1} (three FP64 operations a step, no division), to a width of two
// ulp of the spectral bound; L lanes an eigenvalue.  A step's latency is about that of five warps' issue on the FP64
// pipe, so lanes are free up to there: L = 16 (13 passes instead of 53) up to 2800 eigenvalues, 4 (23) above.  One lane
// an eigenvalue took 7.1 ms at N 760.
template <int L>
__global__ void __launch_bounds__(128) tri_bisect_kernel(const double* __restrict__ d, const double* __restrict__ e,
                                                         int N, double* __restrict__ lam) {
  extern __shared__ double bsm[];
  double* ds = bsm;
  double* e2 = bsm + N;
  __shared__ double lim[2][4];
  const int tid = threadIdx.x, lane = tid & 31;
  double lo = INFINITY, hi = -INFINITY;
  for (int i = tid; i < N; i += 128) {
    const double l = i > 0 ? fabs(e[i - 1]) : 0.0, r = i + 1 < N ? fabs(e[i]) : 0.0;
    ds[i] = d[i];
    e2[i] = i > 0 ? e[i - 1] * e[i - 1] : 0.0;
    lo = fmin(lo, d[i] - l - r);
    hi = fmax(hi, d[i] + l + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) {
    lim[0][tid >> 5] = lo;
    lim[1][tid >> 5] = hi;
  }
  __syncthreads();
  for (int i = 0; i < 4; ++i) {
    lo = fmin(lo, lim[0][i]);
    hi = fmax(hi, lim[1][i]);
  }
  const double width = 4.5e-16 * fmax(fabs(lo), fabs(hi));
  const int s = (blockIdx.x * 128 + tid) / L, q = lane % L;
  lo -= width;
  hi += width;
  for (int it = 0; it < 80 && __any_sync(0xffffffffu, hi - lo > width); ++it) {
    const double h = (hi - lo) * (1.0 / (L + 1));
    const double x = fma(h, (double)(q + 1), lo);
    double p0 = 1.0, p1 = ds[0] - x;
    int cnt = __double2hiint(p1) < 0;
    for (int i = 1; i < N; ++i) {
      double p2 = fma(ds[i] - x, p1, -e2[i] * p0);
      const int s1 = __double2hiint(p1) >> 31;
      // a zero (of either sign) counts as the sign opposite to its predecessor's
      if (((__double2hiint(p2) & 0x7fffffff) | __double2loint(p2)) == 0) p2 = s1 ? 1e-300 : -1e-300;
      cnt += (s1 ^ (__double2hiint(p2) >> 31)) & 1;
      p0 = p1;
      p1 = p2;
      if ((i & 3) == 0) {                    // keep the pair near 1: scale by a power of two
        const int ex = max((__double2hiint(p0) >> 20) & 0x7ff, (__double2hiint(p1) >> 20) & 0x7ff);
        if (ex > 1023 + 200 || ex < 1023 - 200) {
          const double f = __hiloint2double(min(2045, max(1, 2046 - ex)) << 20, 0);
          p0 *= f;
          p1 *= f;
        }
      }
    }
    // counts grow with x: the eigenvalue lies above the last point whose count is <= s
    const unsigned m = __ballot_sync(0xffffffffu, cnt <= s) >> (lane - q);
    const int below = __popc(m & (L == 32 ? 0xffffffffu : (1u << L) - 1u));
    if (below < L) hi = fma(h, (double)(below + 1), lo);
    if (below > 0) lo = fma(h, (double)below, lo);
  }
  if (q == 0 && s < N) lam[s] = 0.5 * (lo + hi);
}

// Eigenvector of T to lam[s] by the twisted factorisation of T - lam: forward pivots q+_i = (d_i - lam) - e_{i-1} l+_{i-1}
// and backward ones q-_i = (d_i - lam) - e_i l-_{i+1}, l = e / q, the twist at the smallest |(d_i - lam) - e_{i-1} l+_{i-1}
// - e_i l-_{i+1}|, and the products of -l outward from it.  Warp 0 runs the forward recurrence, warp 1 the backward one
// (each bound by the latency of a division a step).  Z[s][.] (row length ld), its squared norm in nrm[s]; Lp, Lm [N][ldw]
// work space (vector s in column s; Lp[i] = e_i / q+_i, Lm[i] = e_{i-1} / q-_i).
__global__ void __launch_bounds__(64) tri_vector_kernel(const double* __restrict__ d, const double* __restrict__ e, int N,
                                                        const double* __restrict__ lam, double* __restrict__ Lp,
                                                        double* __restrict__ Lm, long ldw, double* __restrict__ Z,
                                                        long ld, double* __restrict__ nrm) {
  __shared__ double s_min[2][32], s_n2[2][32];
  __shared__ int s_k[2][32];
  const int lane = threadIdx.x & 31, half = threadIdx.x >> 5, s = min(blockIdx.x * 32 + lane, N - 1);
  const bool mine = blockIdx.x * 32 + lane < N;
  const double x = lam[s], tiny = 1e-290;
  double l = 0.0;
  for (int c = 0; c < N; ++c) {
    const int i = half ? N - 1 - c : c;
    const double eb = half ? (i + 1 < N ? e[i] : 0.0) : (i > 0 ? e[i - 1] : 0.0);    // towards where it comes from
    const double ea = half ? (i > 0 ? e[i - 1] : 0.0) : (i + 1 < N ? e[i] : 0.0);
    double q = (d[i] - x) - eb * l;
    if (!(fabs(q) >= tiny)) q = -tiny;
    l = ea / q;
    if (mine) (half ? Lm : Lp)[i * ldw + s] = l;
  }
  __syncthreads();
  double best = INFINITY;
  int k = 0;
#pragma unroll 4
  for (int i = half; i < N; i += 2) {
    double g = d[i] - x;
    if (i > 0) g -= e[i - 1] * Lp[(i - 1) * ldw + s];
    if (i + 1 < N) g -= e[i] * Lm[(i + 1) * ldw + s];
    if (fabs(g) < best) { best = fabs(g); k = i; }
  }
  s_min[half][lane] = best;
  s_k[half][lane] = k;
  __syncthreads();
  k = s_min[1][lane] < s_min[0][lane] ? s_k[1][lane] : s_k[0][lane];
  double z = 1.0, n2 = 0.0;
  double* Zs = Z + (long)s * ld;
  if (half == 0) {
    if (mine) Zs[k] = 1.0;
    n2 = 1.0;
#pragma unroll 4
    for (int i = k - 1; i >= 0; --i) {
      z *= -Lp[i * ldw + s];
      if (mine) Zs[i] = z;
      n2 = fma(z, z, n2);
    }
  } else {
#pragma unroll 4
    for (int i = k + 1; i < N; ++i) {
      z *= -Lm[i * ldw + s];
      if (mine) Zs[i] = z;
      n2 = fma(z, z, n2);
    }
  }
  s_n2[half][lane] = n2;
  __syncthreads();
  if (half == 0 && mine) nrm[s] = s_n2[0][lane] + s_n2[1][lane];
}

// Rows Z[s] <- Q z_s / |z_s|: the reflectors from last to first, one warp a vector (held in shared memory).  Bound by a
// reflector's chain (dot product, shuffles, update); a prefetch of the next reflector's row made it slower (2.1 ms to
// 2.4 ms at N 760).
__global__ void tri_back_kernel(const double* __restrict__ H, const double* __restrict__ beta, int N, long ld,
                                const double* __restrict__ nrm, double* __restrict__ Z) {
  extern __shared__ double zsm[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, s = blockIdx.x * (blockDim.x >> 5) + w;
  if (s >= N) return;
  double* z = zsm + (long)w * N;
  double* Zs = Z + (long)s * ld;
  const double f = 1.0 / sqrt(nrm[s]);
  for (int i = lane; i < N; i += 32) z[i] = Zs[i] * f;
  __syncwarp();
  for (int k = N - 3; k >= 0; --k) {
    const double b = beta[k];
    if (b == 0.0) continue;
    const double* h = H + (long)k * ld;
    double t = 0.0;
    // lanes keep their own elements (i = lane mod 32), so no exchange through z is needed
    const int i0 = k + 1 + ((lane - (k + 1)) & 31);
#pragma unroll 4
    for (int i = i0; i < N; i += 32) t = fma(h[i], z[i], t);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    t *= b;
#pragma unroll 4
    for (int i = i0; i < N; i += 32) z[i] = fma(-t, h[i], z[i]);
  }
  for (int i = lane; i < N; i += 32) Zs[i] = z[i];
}

// Refinement (Ogita and Aishima) of rows V (V M V^T = S, V V^T = G): E_st = (S_st + lam_t R_st) / (lam_t - lam_s) off the diagonal (R_st / 2
// where the two are closer than `close`), E_ss = R_ss / 2, R = I - G, lam_s = S_ss / (1 - R_ss); rows V_t <- V_t + sum_s
// E_st V_s, so G is overwritten by I + E^T.  norms: [0] off-diagonal and [1] diagonal squares of S, [2] squares of R.
__global__ void __launch_bounds__(256) eig_norms_kernel(const double* __restrict__ S, const double* __restrict__ G, int N,
                                                        double* __restrict__ norms) {
  __shared__ double red[3][8];
  double v[3] = {0.0, 0.0, 0.0};
  for (long i = blockIdx.x * 256L + threadIdx.x; i < (long)N * N; i += gridDim.x * 256L) {
    const bool diag = i / N == i % N;
    const double a = S[i], r = (diag ? 1.0 : 0.0) - G[i];
    v[diag ? 1 : 0] += a * a;
    v[2] += r * r;
  }
  for (int c = 0; c < 3; ++c) {
    for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
    if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = v[c];
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int i = 0; i < 8; ++i) t += red[threadIdx.x][i];
    atomicAdd(norms + threadIdx.x, t);
  }
}

__global__ void __launch_bounds__(256) eig_update_kernel(const double* __restrict__ S, double* __restrict__ G, int N,
                                                         double* __restrict__ C, const double* __restrict__ norms) {
  // close: below the rounding level of S's off-diagonal elements against the gap
  const double close = 2.0 * (sqrt(norms[0]) + sqrt(norms[1]) * sqrt(norms[2]));
  for (long i = blockIdx.x * 256L + threadIdx.x; i < (long)N * N; i += gridDim.x * 256L) {
    const int t = (int)(i / N), q = (int)(i % N);     // C[t][q] = delta + E_qt
    const double r = (t == q ? 1.0 : 0.0) - G[i];
    double v;
    if (t == q) {
      v = 1.0 + 0.5 * r;
    } else {
      const double lt = S[(long)t * N + t] / G[(long)t * N + t], lq = S[(long)q * N + q] / G[(long)q * N + q];
      const double gap = lt - lq;
      v = fabs(gap) > close ? (S[i] + lt * r) / gap : 0.5 * r;
    }
    C[i] = v;
  }
}

__global__ void eig_omega_kernel(const double* __restrict__ S, const double* __restrict__ G, int N,
                                 double* __restrict__ Om) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < N) Om[s] = sqrt(fmax(S[(long)s * N + s] / G[(long)s * N + s], 0.0));
}

// rows x N with row length ld to row length N.
__global__ void pack_rows_kernel(const double* __restrict__ X, int rows, int N, long ld, double* __restrict__ Y) {
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < (long)rows * N; i += (long)gridDim.x * blockDim.x)
    Y[i] = X[i / N * ld + i % N];
}

__global__ void twice_sqrt_kernel(const double* __restrict__ Dk, int N, double* __restrict__ w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) w[i] = 2.0 * sqrt(Dk[i]);
}

// Sigma at evaluation points p: target tmap[p] (its G energies eps + spin offset, occupations occ) at omega[p]; grid.y
// CTAs share a point's n_bas N terms (one CTA a point took 0.48 ms at 65 thousand terms), their sums added in order.
__global__ void sigma_sd_kernel(const double* __restrict__ w2, const double* __restrict__ Om, int N, int n_bas,
                                const double* __restrict__ eps, const int* __restrict__ tmap,
                                const int* __restrict__ spin, const int* __restrict__ occ_t, int n_occ,
                                const double* __restrict__ omega, double eta, double* __restrict__ part) {
  __shared__ double red[2][8];
  const int p = blockIdx.x;
  const int t = tmap ? tmap[p] : p;
  const double* e = eps + (spin ? (long)spin[t] * n_bas : 0);
  const int occ = occ_t ? occ_t[t] : n_occ;
  const double w = omega[p];
  double s = 0.0, d = 0.0;
  const long n = (long)n_bas * N;
  for (long idx = blockIdx.y * 256L + threadIdx.x; idx < n; idx += gridDim.y * 256L) {
    const int m = (int)(idx / N), k = (int)(idx - (long)m * N);
    const double wt = w2[((long)t * n_bas + m) * N + k];
    // occupied m: 1/(w - e_m + Omega - i eta); virtual m: 1/(w - e_m - Omega + i eta)
    const double a = m < occ ? w - e[m] + Om[k] : w - e[m] - Om[k];
    const double den = a * a + eta * eta;
    s += wt * a / den;
    d -= wt * (a * a - eta * eta) / (den * den);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    d += __shfl_xor_sync(0xffffffffu, d, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = s;
    red[1][threadIdx.x >> 5] = d;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double ts = 0.0, td = 0.0;
    for (int i = 0; i < 8; ++i) { ts += red[0][i]; td += red[1][i]; }
    part[2 * ((long)p * gridDim.y + blockIdx.y)] = ts;
    part[2 * ((long)p * gridDim.y + blockIdx.y) + 1] = td;
  }
}

__global__ void sigma_sd_sum_kernel(const double* __restrict__ part, int n, int npts, double* __restrict__ S,
                                    double* __restrict__ dS) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npts) return;
  double s = 0.0, d = 0.0;
  for (int i = 0; i < n; ++i) {
    s += part[2 * ((long)p * n + i)];
    d += part[2 * ((long)p * n + i) + 1];
  }
  S[p] = s;
  dS[p] = d;
}

}  // namespace

cudaError_t sd_casida_matrix(const double* B, const double* Dk, int n_aux, int N, int Np, double* M, double* T,
                             cudaStream_t s) {
  dim3 g((Np + ST - 1) / ST, (Np + ST - 1) / ST);
  casida_matrix_kernel<<<g, dim3(ST, ST), 0, s>>>(B, Dk, n_aux, N, Np, M);
  identity_kernel<<<1024, 256, 0, s>>>(T, Np);
  return cudaGetLastError();
}

cudaError_t sd_jacobi_sweep(double* M, double* T, int Np, double* cs, cudaStream_t s) {
  const int h = Np / 2;
  const dim3 gr((Np + 255) / 256 < 8 ? (Np + 255) / 256 : 8, h);
  for (int r = 0; r < Np - 1; ++r) {
    jacobi_angles_kernel<<<(h + 127) / 128, 128, 0, s>>>(M, Np, r, cs);
    jacobi_rows_kernel<<<gr, 256, 0, s>>>(M, Np, r, cs);
    jacobi_cols_kernel<<<gr, 256, 0, s>>>(M, Np, r, cs);
    jacobi_cols_kernel<<<gr, 256, 0, s>>>(T, Np, r, cs);
  }
  return cudaGetLastError();
}

cudaError_t sd_offdiag(const double* M, int Np, double* off, cudaStream_t s) {
  cudaMemsetAsync(off, 0, 2 * sizeof(double), s);
  offdiag_kernel<<<256, 256, 0, s>>>(M, Np, off);
  return cudaGetLastError();
}

int sd_direct_max() { return 8192; }       // three vectors of the tridiagonalisation in one SM's shared memory

cudaError_t sd_tridiagonal(double* A, int N, long ld, double* H, double* beta, double* d, double* e, double* p_buf,
                           unsigned* bar, int* err, cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaError_t c = cudaGetDevice(&dev);
  if (c == cudaSuccess) c = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (c != cudaSuccess) return c;
  const int grid = N < nsm ? N : nsm;        // one CTA an SM, at most one a row
  const long with_rows = (3L + (N + grid - 1) / grid) * N * (long)sizeof(double);
  const bool sm = with_rows <= 220 * 1024;   // N up to about 1800
  const int smem = sm ? (int)with_rows : 3 * N * (int)sizeof(double);
  const void* f = sm ? (const void*)tridiag_kernel<true> : (const void*)tridiag_kernel<false>;
  c = sm ? allow_smem<tridiag_kernel<true>>() : allow_smem<tridiag_kernel<false>>();
  if (c == cudaSuccess) c = cudaMemsetAsync(bar, 0, sizeof(unsigned), s);
  if (c != cudaSuccess) return c;
  void* args[] = {(void*)&A, (void*)&N, (void*)&ld, (void*)&H, (void*)&beta, (void*)&d, (void*)&e, (void*)&p_buf,
                  (void*)&bar, (void*)&err};
  return cudaLaunchCooperativeKernel(f, dim3(grid), dim3(TRI_T), args, smem, s);
}

cudaError_t sd_tridiagonal_vectors(const double* d, const double* e, int N, double* lam, double* W1, double* W2, long ldw,
                                   const double* H, const double* beta, long ld, double* nrm, double* Z,
                                   cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaError_t c = cudaGetDevice(&dev);
  if (c == cudaSuccess) c = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int bs = 2 * N * (int)sizeof(double);
  if (c == cudaSuccess) c = allow_smem<tri_bisect_kernel<16>>();
  if (c == cudaSuccess) c = allow_smem<tri_bisect_kernel<4>>();
  if (c == cudaSuccess) c = allow_smem<tri_back_kernel>();
  if (c != cudaSuccess) return c;
  if (N <= 2800) tri_bisect_kernel<16><<<(N + 7) / 8, 128, bs, s>>>(d, e, N, lam);
  else tri_bisect_kernel<4><<<(N + 31) / 32, 128, bs, s>>>(d, e, N, lam);
  tri_vector_kernel<<<(N + 31) / 32, 64, 0, s>>>(d, e, N, lam, W1, W2, ldw, Z, ld, nrm);
  // a vector a warp, as many as fit, but no more than an even share of the SMs
  int warps = (200 * 1024) / (N * (int)sizeof(double));
  const int even = (N + nsm - 1) / nsm;
  warps = warps < even ? warps : even;
  warps = warps < 1 ? 1 : (warps > 8 ? 8 : warps);
  const int zs = warps * N * (int)sizeof(double);
  tri_back_kernel<<<(N + warps - 1) / warps, 32 * warps, zs, s>>>(H, beta, N, ld, nrm, Z);
  return cudaGetLastError();
}

cudaError_t sd_eig_norms(const double* S, const double* G, int N, double* norms, cudaStream_t s) {
  const cudaError_t c = cudaMemsetAsync(norms, 0, 3 * sizeof(double), s);
  if (c != cudaSuccess) return c;
  eig_norms_kernel<<<304, 256, 0, s>>>(S, G, N, norms);
  return cudaGetLastError();
}

cudaError_t sd_eig_update(const double* S, double* G, int N, double* C, const double* norms, cudaStream_t s) {
  eig_update_kernel<<<608, 256, 0, s>>>(S, G, N, C, norms);
  return cudaGetLastError();
}

cudaError_t sd_pack_rows(const double* X, int rows, int N, long ld, double* Y, cudaStream_t s) {
  pack_rows_kernel<<<608, 256, 0, s>>>(X, rows, N, ld, Y);
  return cudaGetLastError();
}

cudaError_t sd_twice_sqrt(const double* Dk, int N, double* w, cudaStream_t s) {
  twice_sqrt_kernel<<<(N + 255) / 256, 256, 0, s>>>(Dk, N, w);
  return cudaGetLastError();
}

cudaError_t sd_rows_weights(const double* S, const double* G, const double* V, const double* Bn, int n_aux, int N, int R,
                            double* Om, double* w2, cudaStream_t s) {
  eig_omega_kernel<<<(N + 255) / 256, 256, 0, s>>>(S, G, N, Om);
  casida_w2_kernel<<<dim3((N + ST - 1) / ST, (R + ST - 1) / ST), dim3(ST, ST), 0, s>>>(Bn, V, Om, n_aux, R, N, w2);
  return cudaGetLastError();
}

cudaError_t sd_weights(const double* B, const double* Dk, const double* M, const double* T, const double* Bn,
                       int n_aux, int N, int Np, int R, double* Om, double* V, double* w2, cudaStream_t s) {
  casida_omega_kernel<<<(N + 255) / 256, 256, 0, s>>>(M, Np, N, Om);
  casida_v_kernel<<<dim3((N + ST - 1) / ST, (n_aux + ST - 1) / ST), dim3(ST, ST), 0, s>>>(B, Dk, T, n_aux, N, Np, V);
  casida_w2_kernel<<<dim3((N + ST - 1) / ST, (R + ST - 1) / ST), dim3(ST, ST), 0, s>>>(Bn, V, Om, n_aux, R, N, w2);
  return cudaGetLastError();
}

int sd_sigma_parts(int n_bas, int N) {
  const long t = ((long)n_bas * N + 255) / 256;
  return (int)(t < 1 ? 1 : (t > 64 ? 64 : t));
}

cudaError_t sd_sigma(const double* w2, const double* Om, int N, int n_bas, const double* eps, const int* tmap,
                     const int* spin, const int* occ_t, int n_occ, const double* omega, int npts, double eta,
                     double* part, double* S, double* dS, cudaStream_t s) {
  if (npts <= 0) return cudaSuccess;
  const int parts = sd_sigma_parts(n_bas, N);
  sigma_sd_kernel<<<dim3(npts, parts), 256, 0, s>>>(w2, Om, N, n_bas, eps, tmap, spin, occ_t, n_occ, omega, eta, part);
  sigma_sd_sum_kernel<<<(npts + 127) / 128, 128, 0, s>>>(part, parts, npts, S, dS);
  return cudaGetLastError();
}

}  // namespace gw
