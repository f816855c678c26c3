// Batched dense solves of the residue systems (1 - Pi(x)) y = b for right-hand sides whose MINRES run
// stayed above the fallback threshold (Sec. 3.3: "the dielectric matrix is actually built" and factorised;
// the paper uses Bunch-Kaufman, this library a complex LU with partial pivoting, which gives the same solution).
// One CTA per matrix; the complex matrix is stored as two real planes (Ar, Ai), row-major n x n.
#include "gw_internal.cuh"
#include "oz_digits.cuh"
#include "oz_gemm.cuh"
#include "pi_tc.cuh"

#include <algorithm>

namespace gw {
namespace {

constexpr int LU_T = 512;        // threads per CTA

template <typename T>
struct cplx {
  T r, i;
};

template <typename T>
__device__ __forceinline__ cplx<T> cdiv(cplx<T> a, cplx<T> b) {
  const T d = b.r * b.r + b.i * b.i;
  return {(a.r * b.r + a.i * b.i) / d, (a.i * b.r - a.r * b.i) / d};
}

// Block-wide argmax of |a|^2 over rows [r0, n) of column c; ties to the lower row.
template <typename T>
__device__ int pivot_row(const T* Ar, const T* Ai, int n, int c, int r0, double* sv, int* si) {
  double best = -1.0;
  int bidx = r0;
  for (int i = r0 + threadIdx.x; i < n; i += blockDim.x) {
    const double m = (double)Ar[(long)i * n + c] * Ar[(long)i * n + c] + (double)Ai[(long)i * n + c] * Ai[(long)i * n + c];
    if (m > best) { best = m; bidx = i; }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bidx, o);
    if (ob > best || (ob == best && oi < bidx)) { best = ob; bidx = oi; }
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = best; si[threadIdx.x >> 5] = bidx; }
  __syncthreads();
  double bb = -1.0;
  int ii = r0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
    if (sv[w] > bb || (sv[w] == bb && si[w] < ii)) { bb = sv[w]; ii = si[w]; }
  return bb > 0.0 ? ii : -1;
}

// Solve A y = rhs with the LU factors and the row permutation; rhs/y complex in two planes of length n (yr, yi),
// overwritten in place.  Forward and back substitution in blocks of SB rows: one warp per row sums the contribution of
// the finished unknowns (held in shared memory) with eight loads in flight, the SB x SB triangle, fetched to shared
// memory meanwhile, is solved by one warp.  Bound by the factors' one read per solve at what a single SM can fetch
// (226 matrices of n 1800: 5.3 ms a solve with 32-row blocks, dependent loads and the swaps replayed one by one).
// SWAPS: for n beyond lu_panel_kernel, perm holds the swaps (lu_panel_global_kernel), the unknowns stay in global memory.
constexpr int SB = 64;
template <typename T, bool SWAPS>
__global__ void __launch_bounds__(LU_T) zlu_solve_kernel(const T* Ar_base, const T* Ai_base, long stride, int n,
                                                         const int* perm_base, T* yr_base, T* yi_base, long ystride) {
  extern __shared__ __align__(16) unsigned char sm[];
  T* tr = reinterpret_cast<T*>(sm);                // [SB][SB + 1] the block's triangle
  T* ti = tr + SB * (SB + 1);
  T* br = ti + SB * (SB + 1);                      // [SB]
  T* bi = br + SB;
  const T* Ar = Ar_base + (long)blockIdx.x * stride;
  const T* Ai = Ai_base + (long)blockIdx.x * stride;
  const int* perm = perm_base + (long)blockIdx.x * n;
  T* yr = yr_base + (long)blockIdx.x * ystride;
  T* yi = yi_base + (long)blockIdx.x * ystride;
  T* vr = SWAPS ? yr : bi + SB;                    // [n] the unknowns
  T* vi = SWAPS ? yi : vr + n;
  if (SWAPS) {
    if (threadIdx.x == 0)
      for (int c = 0; c < n; ++c) {
        const int p = perm[c];
        if (p != c) {
          T t = yr[c]; yr[c] = yr[p]; yr[p] = t;
          t = yi[c]; yi[c] = yi[p]; yi[p] = t;
        }
      }
  } else {
    for (int i = threadIdx.x; i < n; i += LU_T) {
      const int p = perm[i];
      vr[i] = yr[p];
      vi[i] = yi[p];
    }
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nblk = (n + SB - 1) / SB;
  for (int pass = 0; pass < 2; ++pass)             // 0: L (unit lower), ascending; 1: U, descending
    for (int kb = 0; kb < nblk; ++kb) {
      const int blk = pass == 0 ? kb : nblk - 1 - kb;
      const int k0 = blk * SB, nb = min(SB, n - k0);
      const int q0 = pass == 0 ? 0 : k0 + nb, q1 = pass == 0 ? k0 : n;
      for (int idx = threadIdx.x; idx < nb * nb; idx += LU_T) {
        const int r = idx / nb, c = idx - r * nb;
        tr[r * (SB + 1) + c] = Ar[(long)(k0 + r) * n + k0 + c];
        ti[r * (SB + 1) + c] = Ai[(long)(k0 + r) * n + k0 + c];
      }
      for (int r = wid; r < nb; r += LU_T / 32) {
        const T* ar = Ar + (long)(k0 + r) * n;
        const T* ai = Ai + (long)(k0 + r) * n;
        T sr = T(0), si = T(0);
#pragma unroll 4
        for (int q = q0 + lane; q < q1; q += 32) {
          const T lr = ar[q], li = ai[q], ur = vr[q], ui = vi[q];
          sr += lr * ur - li * ui;
          si += lr * ui + li * ur;
        }
        for (int o = 16; o > 0; o >>= 1) {
          sr += __shfl_xor_sync(0xffffffffu, sr, o);
          si += __shfl_xor_sync(0xffffffffu, si, o);
        }
        if (lane == 0) {
          br[r] = vr[k0 + r] - sr;
          bi[r] = vi[k0 + r] - si;
        }
      }
      __syncthreads();
      if (wid == 0) {                              // lanes hold rows lane and lane + 32
        T x0r = lane < nb ? br[lane] : T(0), x0i = lane < nb ? bi[lane] : T(0);
        T x1r = lane + 32 < nb ? br[lane + 32] : T(0), x1i = lane + 32 < nb ? bi[lane + 32] : T(0);
        if (pass == 1) {                           // divide by the diagonal first: rows scaled to a unit triangle
          for (int h = 0; h < 2; ++h) {
            const int r = lane + 32 * h;
            if (r >= nb) continue;
            const cplx<T> dd = {tr[r * (SB + 1) + r], ti[r * (SB + 1) + r]};
            const bool z = dd.r == T(0) && dd.i == T(0);
            const cplx<T> inv = z ? cplx<T>{T(0), T(0)} : cdiv(cplx<T>{T(1), T(0)}, dd);
            // the row is scaled where it is used: keep the reciprocal in the diagonal's place
            tr[r * (SB + 1) + r] = inv.r;
            ti[r * (SB + 1) + r] = inv.i;
          }
          __syncwarp();
        }
        for (int t = 0; t < nb; ++t) {
          const int q = pass == 0 ? t : nb - 1 - t;
          T uq_r = __shfl_sync(0xffffffffu, q < 32 ? x0r : x1r, q & 31);
          T uq_i = __shfl_sync(0xffffffffu, q < 32 ? x0i : x1i, q & 31);
          if (pass == 1) {
            const T ir = tr[q * (SB + 1) + q], ii = ti[q * (SB + 1) + q];
            const T a = uq_r * ir - uq_i * ii;
            uq_i = uq_r * ii + uq_i * ir;
            uq_r = a;
            if (lane == (q & 31)) {
              if (q < 32) { x0r = uq_r; x0i = uq_i; } else { x1r = uq_r; x1i = uq_i; }
            }
          }
          const bool on0 = pass == 0 ? lane > q : lane < q;
          const bool on1 = (pass == 0 ? lane + 32 > q : lane + 32 < q) && lane + 32 < nb;
          if (on0 && lane < nb) {
            const T lr = tr[lane * (SB + 1) + q], li = ti[lane * (SB + 1) + q];
            x0r -= lr * uq_r - li * uq_i;
            x0i -= lr * uq_i + li * uq_r;
          }
          if (on1) {
            const T lr = tr[(lane + 32) * (SB + 1) + q], li = ti[(lane + 32) * (SB + 1) + q];
            x1r -= lr * uq_r - li * uq_i;
            x1i -= lr * uq_i + li * uq_r;
          }
        }
        if (lane < nb) { vr[k0 + lane] = x0r; vi[k0 + lane] = x0i; }
        if (lane + 32 < nb) { vr[k0 + lane + 32] = x1r; vi[k0 + lane + 32] = x1i; }
      }
      __syncthreads();
    }
  if (!SWAPS)
    for (int i = threadIdx.x; i < n; i += LU_T) {
      yr[i] = vr[i];
      yi[i] = vi[i];
    }
}

// ---------------------------------------------------------------------------------------------------------------
// Blocked LU with the trailing update on the tensor cores.  Per panel of TC_PW columns [k0, kend):
//   1. lu_panel_kernel factors the panel (rows k0..n-1, partial pivoting) and leaves the panel's row permutation and
//      the inverse of its unit lower triangle L11;
//   2. lu_cols_kernel permutes the rows of all other columns and, right of the panel, forms U12 = L11^-1 A12 and its
//      operand for the update;
//   3. the complex update A22 -= L21 U12 as one real product with K = 2 TC_PW:
//        [Re; Im] A22 -= [[Re L, -Im L]; [Im L, Re L]] [Re U12; Im U12],
//      in FP32 factors as three BF16 parts (six products, about FP32-accurate; tc_gemm_ex), in FP64 factors as exact
//      digits (oz_gemm), whose epilogues subtract the stacked result from the two planes.
constexpr int TC_PW = 64;
constexpr int TC_LDK = 2 * TC_PW;           // row length of the operands (a multiple of 8)
constexpr int SW_LD = 4 * TC_PW + 2;        // ints per matrix of the panel's permutation: count, then (row, source)

// One CTA per matrix; its threads hold NB columns of the panel in registers (RPT rows each: row k0 + t + 512 r), so a
// column costs two barriers and no global traffic: pivot search by shuffles, the two swapped rows through shared
// memory, the rank-1 update in registers.  Each NB columns are first brought up to date with the panel's earlier ones
// (U by one warp per column from L11 in shared memory, then one pass over the rows' earlier multipliers), and the
// panel's other columns follow the swaps.  Bound by the latency of its loads (the rows' earlier multipliers, 8 bytes a
// thread; 152 matrices share L2) and of the columns' barriers: the first panel at n 1800 takes 0.71 ms in FP32 (0.38 on
// average over the matrix; 0.85 and 0.43 for 152 matrices at once) and 5.1 ms in FP64 (16 clocks a warp instruction),
// where factoring column by column in global memory took 1.4 ms in FP32.  NB shrinks as rows a thread grow, to stay in
// 64 registers.
// Magnitudes as integer keys (the bits of |a|^2; NaN counts as 0), so that the pivot search stays off the FP64 pipe.
__device__ __forceinline__ unsigned pivot_key(float v) {
  const unsigned b = __float_as_uint(v);
  return b > 0x7f800000u ? 0u : b;
}
__device__ __forceinline__ unsigned long long pivot_key(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return b > 0x7ff0000000000000ull ? 0ull : b;
}
// Largest key of the warp, the lowest row among equals.
__device__ __forceinline__ void warp_pivot(unsigned& key, int& row) {
  const unsigned mx = __reduce_max_sync(0xffffffffu, key);
  row = (int)__reduce_min_sync(0xffffffffu, key == mx ? (unsigned)row : 0x7fffffffu);
  key = mx;
}
__device__ __forceinline__ void warp_pivot(unsigned long long& key, int& row) {
  const unsigned hi = (unsigned)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = hi == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
  const unsigned long long mx = ((unsigned long long)mh << 32) | ml;
  row = (int)__reduce_min_sync(0xffffffffu, key == mx ? (unsigned)row : 0x7fffffffu);
  key = mx;
}

// L11^-1 (unit lower) of a full panel from its multipliers Lr, Li [TC_PW][TC_PW + 1] to linv; X: 2 TC_PW^2 elements of
// shared memory.  Thread (row tid / 8, columns tid % 8 + 8 t); step q adds row q to the rows below it.  All LU_T threads.
template <typename T>
__device__ __forceinline__ void invert_l11(const T* Lr, const T* Li, T* Xr, T* linv) {
  constexpr int LD = TC_PW + 1;
  const int tid = threadIdx.x;
  T* Xi = Xr + TC_PW * TC_PW;
  const int r = tid >> 3, j0 = tid & 7;
  T xr[8], xi[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    xr[t] = r == j0 + 8 * t ? T(1) : T(0);
    xi[t] = T(0);
    Xr[r * TC_PW + j0 + 8 * t] = xr[t];
    Xi[r * TC_PW + j0 + 8 * t] = xi[t];
  }
  __syncthreads();
  for (int q = 0; q + 1 < TC_PW; ++q) {
    if (r > q) {
      const T lr = Lr[r * LD + q], li = Li[r * LD + q];
#pragma unroll
      for (int t = 0; t < 8; ++t)
        if (8 * t <= q) {
          const T ur = Xr[q * TC_PW + j0 + 8 * t], ui = Xi[q * TC_PW + j0 + 8 * t];
          xr[t] = fma(-lr, ur, xr[t]);
          xr[t] = fma(li, ui, xr[t]);
          xi[t] = fma(-lr, ui, xi[t]);
          xi[t] = fma(-li, ur, xi[t]);
        }
      if (r == q + 1)
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          Xr[r * TC_PW + j0 + 8 * t] = xr[t];
          Xi[r * TC_PW + j0 + 8 * t] = xi[t];
        }
    }
    __syncthreads();
  }
  // [q][row]: column q of L11^-1 contiguous in the row, as lu_cols_kernel reads it
  T* vi = linv + TC_PW * TC_PW;
  for (int i = tid; i < TC_PW * TC_PW; i += LU_T) {
    const int q = i / TC_PW, row = i % TC_PW;
    linv[i] = Xr[row * TC_PW + q];
    vi[i] = Xi[row * TC_PW + q];
  }
}

template <typename T, int RPT, int NB>
__global__ void __launch_bounds__(LU_T, 1) lu_panel_kernel(T* Ar_base, T* Ai_base, long stride, int n, int k0, int kend,
                                                           int* perm_base, int* info, int* sw_base, T* linv_base) {
  extern __shared__ __align__(16) unsigned char sm[];
  constexpr int LD = TC_PW + 1;
  T* Lr = reinterpret_cast<T*>(sm);                // [TC_PW][LD] multipliers of the panel's finished rows
  T* Li = Lr + TC_PW * LD;
  T* Ur = Li + TC_PW * LD;                         // [TC_PW][NB]
  T* Ui = Ur + TC_PW * NB;
  T* stage = Ui + TC_PW * NB;                      // [2 NB][2 TC_PW]
  int* map = reinterpret_cast<int*>(stage + 2 * NB * 2 * TC_PW);   // [n - k0]
  typedef decltype(pivot_key(T(0))) Key;
  __shared__ T prow[2 * NB + 2], crow[2 * NB];     // prow: the pivot row and the pivot's reciprocal
  __shared__ Key rv[LU_T / 32];
  __shared__ int ri[LU_T / 32], pv[TC_PW], lst[2 * NB], src[2 * NB];
  __shared__ int cnt, s_bad;
  T* Ar = Ar_base + (long)blockIdx.x * stride + (long)k0 * n + k0;    // the panel's corner
  T* Ai = Ai_base + (long)blockIdx.x * stride + (long)k0 * n + k0;
  int* perm = perm_base + (long)blockIdx.x * n;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int m = n - k0, pw = kend - k0;
  if (k0 == 0)
    for (int i = tid; i < n; i += LU_T) perm[i] = i;
  for (int i = tid; i < m; i += LU_T) map[i] = i;
  if (tid == 0) s_bad = 0;
  T ar[RPT][NB], ai[RPT][NB];
  for (int c0 = 0; c0 < pw; c0 += NB) {
    const int nb = min(NB, pw - c0);
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const int i = tid + LU_T * r;
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const bool in = i < m && j < nb;
        ar[r][j] = in ? Ar[(long)i * n + c0 + j] : T(0);
        ai[r][j] = in ? Ai[(long)i * n + c0 + j] : T(0);
      }
    }
    if (c0 > 0) {
      if (tid < c0)
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          Ur[tid * NB + j] = ar[0][j];
          Ui[tid * NB + j] = ai[0][j];
        }
      __syncthreads();
      // U = L11^-1 (top rows), one element a thread (row tid / 8): only warps with rows below q work in step q
      {
        const int r = tid >> 3, j = tid & 7;
        const bool on = j < NB && r < c0;
        T xr = on ? Ur[r * NB + j] : T(0), xi = on ? Ui[r * NB + j] : T(0);
        for (int q = 0; q + 1 < c0; ++q) {
          if (on && r > q) {
            const T lr = Lr[r * LD + q], li = Li[r * LD + q], ur = Ur[q * NB + j], ui = Ui[q * NB + j];
            xr = fma(-lr, ur, xr);
            xr = fma(li, ui, xr);
            xi = fma(-lr, ui, xi);
            xi = fma(-li, ur, xi);
            if (r == q + 1) {
              Ur[r * NB + j] = xr;
              Ui[r * NB + j] = xi;
            }
          }
          __syncthreads();
        }
      }
      if (tid < c0)
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          ar[0][j] = Ur[tid * NB + j];
          ai[0][j] = Ui[tid * NB + j];
        }
      // rows c0..m-1: minus (their multipliers of the panel's earlier columns) x U
#pragma unroll (RPT <= 2 && sizeof(T) == 4 ? 4 : 2)
      for (int q = 0; q < c0; ++q) {
        T lr[RPT], li[RPT];
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
          const int i = tid + LU_T * r;
          const bool in = i >= c0 && i < m;
          lr[r] = in ? Ar[(long)i * n + q] : T(0);
          li[r] = in ? Ai[(long)i * n + q] : T(0);
        }
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const T ur = Ur[q * NB + j], ui = Ui[q * NB + j];
#pragma unroll
          for (int r = 0; r < RPT; ++r)
            if (32 * wid + LU_T * r < m) {         // warps without rows stay off the FMA pipe
              ar[r][j] = fma(-lr[r], ur, ar[r][j]);
              ar[r][j] = fma(li[r], ui, ar[r][j]);
              ai[r][j] = fma(-lr[r], ui, ai[r][j]);
              ai[r][j] = fma(-li[r], ur, ai[r][j]);
            }
        }
      }
    }
    // ---- factor the NB columns
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      if (j >= nb) break;
      const int c = c0 + j;
      Key best = 0;
      int row = c;
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const int i = tid + LU_T * r;
        if (i >= c && i < m) {
          const Key v = pivot_key(ar[r][j] * ar[r][j] + ai[r][j] * ai[r][j]);
          if (v > best) { best = v; row = i; }
        }
      }
      if (best == 0) row = 0x7fffffff;
      warp_pivot(best, row);
      if (lane == 0) { rv[wid] = best; ri[wid] = row; }
      __syncthreads();
      best = lane < LU_T / 32 ? rv[lane] : 0;
      row = lane < LU_T / 32 ? ri[lane] : 0x7fffffff;
      warp_pivot(best, row);
      const bool none = best == 0;
      const int p = none ? c : row;
      if (tid == 0) {
        pv[c] = p;
        if (none) s_bad = k0 + c + 1;
      }
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const int i = tid + LU_T * r;
        if (i == p) {
#pragma unroll
          for (int jj = 0; jj < NB; ++jj) { prow[jj] = ar[r][jj]; prow[NB + jj] = ai[r][jj]; }
          const cplx<T> d = {ar[r][j], ai[r][j]};
          const bool dz = d.r == T(0) && d.i == T(0);
          const cplx<T> inv = dz ? cplx<T>{T(0), T(0)} : cdiv(cplx<T>{T(1), T(0)}, d);
          prow[2 * NB] = inv.r;
          prow[2 * NB + 1] = inv.i;
        }
        if (i == c)
#pragma unroll
          for (int jj = 0; jj < NB; ++jj) { crow[jj] = ar[r][jj]; crow[NB + jj] = ai[r][jj]; }
      }
      __syncthreads();
      const cplx<T> inv = {prow[2 * NB], prow[2 * NB + 1]};
#pragma unroll
      for (int r = 0; r < RPT; ++r) {
        const int i = tid + LU_T * r;
        if (i == p)
#pragma unroll
          for (int jj = 0; jj < NB; ++jj) { ar[r][jj] = crow[jj]; ai[r][jj] = crow[NB + jj]; }
        if (i == c)
#pragma unroll
          for (int jj = 0; jj < NB; ++jj) { ar[r][jj] = prow[jj]; ai[r][jj] = prow[NB + jj]; }
        if (i > c && i < m) {
          const T lr = ar[r][j] * inv.r - ai[r][j] * inv.i, li = ar[r][j] * inv.i + ai[r][j] * inv.r;
          ar[r][j] = lr;
          ai[r][j] = li;
#pragma unroll
          for (int jj = 0; jj < NB; ++jj)
            if (jj > j) {
              const T ur = prow[jj], ui = prow[NB + jj];
              ar[r][jj] = fma(-lr, ur, ar[r][jj]);
              ar[r][jj] = fma(li, ui, ar[r][jj]);
              ai[r][jj] = fma(-lr, ui, ai[r][jj]);
              ai[r][jj] = fma(-li, ur, ai[r][jj]);
            }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RPT; ++r) {
      const int i = tid + LU_T * r;
#pragma unroll
      for (int j = 0; j < NB; ++j)
        if (i < m && j < nb) {
          Ar[(long)i * n + c0 + j] = ar[r][j];
          Ai[(long)i * n + c0 + j] = ai[r][j];
        }
    }
    // ---- the panel's other columns follow these swaps: final source of every row touched, then one gather and store
    if (wid == 0) {
      // lane t holds row lst[t] of the list and the list index its content comes from
      int k = nb, row = lane < nb ? c0 + lane : -1, from = lane;
      for (int j = 0; j < nb; ++j) {
        const int p = pv[c0 + j];
        const unsigned hit = __ballot_sync(0xffffffffu, row == p);
        const int at = hit ? __ffs(hit) - 1 : k;
        if (!hit) {
          if (lane == k) row = p;
          ++k;
        }
        const int fj = __shfl_sync(0xffffffffu, from, j), fa = __shfl_sync(0xffffffffu, from, at);
        if (lane == j) from = fa;
        if (lane == at) from = fj;
      }
      // the panel's permutation so far: map[row] = the row its content came from
      const int old = lane < k ? map[row] : 0;
      const int now = __shfl_sync(0xffffffffu, old, from);
      if (lane < k) {
        lst[lane] = row;
        src[lane] = from;
        map[row] = now;
      }
      if (lane == 0) cnt = k;
    }
    __syncthreads();
    if (tid < 2 * pw) {
      const int col = tid < pw ? tid : tid - pw;
      if (col < c0 || col >= c0 + nb) {
        T* A = tid < pw ? Ar : Ai;
        const int k = cnt;
#pragma unroll
        for (int t = 0; t < 2 * NB; ++t)
          if (t < k) stage[t * 2 * TC_PW + tid] = A[(long)lst[t] * n + col];
        for (int t = 0; t < k; ++t)
          if (src[t] != t) A[(long)lst[t] * n + col] = stage[src[t] * 2 * TC_PW + tid];
      }
    }
    __syncthreads();
    for (int idx = tid; idx < nb * TC_PW; idx += LU_T) {     // the finished rows' multipliers
      const int r = c0 + idx / TC_PW, q = idx % TC_PW;
      if (q < r) {
        Lr[r * LD + q] = Ar[(long)r * n + q];
        Li[r * LD + q] = Ai[(long)r * n + q];
      }
    }
    __syncthreads();
  }
  // ---- the panel's permutation as (row, source row) pairs of the rows that move, and the running permutation
  if (tid == 0) cnt = 0;
  __syncthreads();
  int* sw = sw_base + (long)blockIdx.x * SW_LD;
  int old0 = 0, old1 = 0, dst1 = -1;
  if (tid < pw) {
    sw[1 + 2 * tid] = k0 + tid;                    // the panel's own rows, in order
    sw[2 + 2 * tid] = k0 + map[tid];
    old0 = perm[k0 + map[tid]];
    const int p = pv[tid];
    bool mine = p >= pw;                           // rows below it, once each
    for (int j = 0; j < tid && mine; ++j) mine = pv[j] != p;
    if (mine) {
      const int at = pw + atomicAdd(&cnt, 1);
      sw[1 + 2 * at] = k0 + p;
      sw[2 + 2 * at] = k0 + map[p];
      dst1 = p;
      old1 = perm[k0 + map[p]];
    }
  }
  __syncthreads();
  if (tid < pw) {
    perm[k0 + tid] = old0;
    if (dst1 >= 0) perm[k0 + dst1] = old1;
  }
  if (tid == 0) {
    sw[0] = pw + cnt;
    if (k0 == 0) info[blockIdx.x] = s_bad;
    else if (s_bad && info[blockIdx.x] == 0) info[blockIdx.x] = s_bad;
  }
  if (kend >= n) return;
  invert_l11(Lr, Li, Ur, linv_base + (long)blockIdx.x * 2 * TC_PW * TC_PW);   // over Ur, Ui, stage (and map, read above)
}

// A panel of more rows than lu_panel_kernel holds, in global memory: columns brought up to date one by one (the rows'
// multipliers times the column's U part, thread per row), pivot, swap within the panel, scale.  perm[c] receives the row
// swapped with row c, sw and linv as in lu_panel_kernel.  Bound by the rows' multipliers, read once a column from L2 by
// one SM: a mixed residue at n 16397 takes 3.8 s (15 ms a panel), an FP64 one at 8203 1.4 s.  The whole matrix in one CTA,
// which this replaces, would run the trailing updates' (8/3) n^3 at the rate of one SM: minutes.
template <typename T>
__global__ void __launch_bounds__(LU_T) lu_panel_global_kernel(T* Ar_base, T* Ai_base, long stride, int n, int k0,
                                                               int kend, int* perm_base, int* info, int* sw_base,
                                                               T* linv_base) {
  extern __shared__ __align__(16) unsigned char sm[];
  constexpr int LD = TC_PW + 1;
  T* Lr = reinterpret_cast<T*>(sm);                // [TC_PW][LD] multipliers of the panel's finished rows
  T* Li = Lr + TC_PW * LD;
  T* X = Li + TC_PW * LD;                          // [2][TC_PW][TC_PW]
  __shared__ double sv[32];
  __shared__ int si[32], pv[TC_PW], row[2 * TC_PW], from[2 * TC_PW];
  __shared__ T ur[TC_PW], ui[TC_PW];
  T* Ar = Ar_base + (long)blockIdx.x * stride;
  T* Ai = Ai_base + (long)blockIdx.x * stride;
  const int tid = threadIdx.x, pw = kend - k0;
  int bad = 0;
  for (int cc = 0; cc < pw; ++cc) {
    const int c = k0 + cc;
    // U part of the column: u = L11^-1 (rows k0 .. c - 1)
    T xr = tid < cc ? Ar[(long)(k0 + tid) * n + c] : T(0), xi = tid < cc ? Ai[(long)(k0 + tid) * n + c] : T(0);
    if (tid < cc) { ur[tid] = xr; ui[tid] = xi; }
    __syncthreads();
    for (int q = 0; q + 1 < cc; ++q) {
      if (tid > q && tid < cc) {
        const T lr = Lr[tid * LD + q], li = Li[tid * LD + q];
        xr -= lr * ur[q] - li * ui[q];
        xi -= lr * ui[q] + li * ur[q];
        if (tid == q + 1) { ur[tid] = xr; ui[tid] = xi; }
      }
      __syncthreads();
    }
    if (tid < cc) {
      Ar[(long)(k0 + tid) * n + c] = xr;
      Ai[(long)(k0 + tid) * n + c] = xi;
    }
    if (cc > 0)
      for (int i = c + tid; i < n; i += LU_T) {    // rows c .. n - 1
        const T* lr = Ar + (long)i * n + k0;
        const T* li = Ai + (long)i * n + k0;
        T sr = T(0), s2 = T(0);
        for (int q = 0; q < cc; ++q) {
          sr += lr[q] * ur[q] - li[q] * ui[q];
          s2 += lr[q] * ui[q] + li[q] * ur[q];
        }
        Ar[(long)i * n + c] -= sr;
        Ai[(long)i * n + c] -= s2;
      }
    __syncthreads();
    int p = pivot_row(Ar, Ai, n, c, c, sv, si);
    if (p < 0) { bad = c + 1; p = c; }
    if (tid == 0) pv[cc] = p;
    if (p != c && tid < 2 * pw) {
      T* A = (tid < pw ? Ar : Ai) + k0 + (tid < pw ? tid : tid - pw);
      const T t = A[(long)c * n];
      A[(long)c * n] = A[(long)p * n];
      A[(long)p * n] = t;
    }
    __syncthreads();
    if (tid < cc) {
      Lr[cc * LD + tid] = Ar[(long)c * n + k0 + tid];
      Li[cc * LD + tid] = Ai[(long)c * n + k0 + tid];
    }
    const cplx<T> d = {Ar[(long)c * n + c], Ai[(long)c * n + c]};
    const bool dz = d.r == T(0) && d.i == T(0);
    for (int i = c + 1 + tid; i < n; i += LU_T) {
      cplx<T> l = {Ar[(long)i * n + c], Ai[(long)i * n + c]};
      l = dz ? cplx<T>{T(0), T(0)} : cdiv(l, d);
      Ar[(long)i * n + c] = l.r;
      Ai[(long)i * n + c] = l.i;
    }
    __syncthreads();
  }
  int* sw = sw_base + (long)blockIdx.x * SW_LD;
  if (tid == 0) {
    // the rows that move and the rows their content comes from: the panel's own rows, in order, then others as met
    int cnt = pw;
    for (int j = 0; j < pw; ++j) row[j] = from[j] = k0 + j;
    for (int j = 0; j < pw; ++j) {
      int at = pv[j] < kend ? pv[j] - k0 : pw;
      while (at < cnt && row[at] != pv[j]) ++at;
      if (at == cnt) { row[at] = from[at] = pv[j]; ++cnt; }
      const int t = from[j];
      from[j] = from[at];
      from[at] = t;
    }
    sw[0] = cnt;
    for (int t = 0; t < cnt; ++t) { sw[1 + 2 * t] = row[t]; sw[2 + 2 * t] = from[t]; }
    if (k0 == 0) info[blockIdx.x] = bad;
    else if (bad && info[blockIdx.x] == 0) info[blockIdx.x] = bad;
  }
  if (tid < pw) perm_base[(long)blockIdx.x * n + k0 + tid] = pv[tid];
  if (kend < n) invert_l11(Lr, Li, X, linv_base + (long)blockIdx.x * 2 * TC_PW * TC_PW);
}

__device__ __forceinline__ void split3(float v, __nv_bfloat16* p0, __nv_bfloat16* p1, __nv_bfloat16* p2, long o) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  const float r = v - __bfloat162float(h);
  const __nv_bfloat16 l = __float2bfloat16_rn(r);
  p0[o] = h;
  p1[o] = l;
  p2[o] = __float2bfloat16_rn(r - __bfloat162float(l));
}

// Rows of the stacked left operand for the m = n - kend rows below the panel: row r = [Re L_r, -Im L_r],
// row m + r = [Im L_r, Re L_r] (L_r = row kend + r, panel columns k0..k0+TC_PW-1); out [batch][2m][TC_LDK].
// lim: elements addressable from Ar_base (the Ai plane and every matrix of the batch lie inside it); wlim: elements of
// each operand part.  An index beyond is recorded in *err (codes 62, 63) and skipped.
__global__ void lu_split_l_kernel(const float* Ar_base, const float* Ai_base, long stride, int n, int k0, int kend,
                                  __nv_bfloat16* p0, __nv_bfloat16* p1, __nv_bfloat16* p2, long lim, long wlim,
                                  int* err) {
  const int m = n - kend;
  const int r = 2 * blockIdx.x + (threadIdx.x >> 7), q = threadIdx.x & 127;
  if (r >= m) return;
  const float* Ar = Ar_base + (long)blockIdx.y * stride;
  const float* Ai = Ai_base + (long)blockIdx.y * stride;
  const long src = (long)(kend + r) * n + k0 + (q & (TC_PW - 1));
  if ((long)blockIdx.y * stride + (Ai_base - Ar_base) + src >= lim) { atomicCAS(err, 0, 62); return; }
  const float lr = Ar[src], li = Ai[src];
  const long ob = (long)blockIdx.y * 2 * m * TC_LDK;
  if (ob + (long)(m + r) * TC_LDK + q >= wlim) { atomicCAS(err, 0, 63); return; }
  split3(q < TC_PW ? lr : -li, p0, p1, p2, ob + (long)r * TC_LDK + q);
  split3(q < TC_PW ? li : lr, p0, p1, p2, ob + (long)(m + r) * TC_LDK + q);
}

// Eight elements split into three BF16 parts, 16 bytes each.
__device__ __forceinline__ void split3x8(const float (&v)[8], __nv_bfloat16* p0, __nv_bfloat16* p1,
                                         __nv_bfloat16* p2) {
  __nv_bfloat162 h[4], l[4], t[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    const float r0 = v[2 * i] - __low2float(h[i]), r1 = v[2 * i + 1] - __high2float(h[i]);
    l[i] = __floats2bfloat162_rn(r0, r1);
    t[i] = __floats2bfloat162_rn(r0 - __low2float(l[i]), r1 - __high2float(l[i]));
  }
  *reinterpret_cast<uint4*>(p0) = *reinterpret_cast<uint4*>(h);
  *reinterpret_cast<uint4*>(p1) = *reinterpret_cast<uint4*>(l);
  *reinterpret_cast<uint4*>(p2) = *reinterpret_cast<uint4*>(t);
}

// 64 columns a CTA, outside the panel (first those left of it, then those right of it): rows permuted as the panel's;
// right of it U12 = L11^-1 A12 (4 x 4 outputs a thread) and the operand of the update, row c = [Re U12[:, c],
// Im U12[:, c]]: FP32 split into three BF16 parts p0, p1, p2 of [batch][m][TC_LDK], FP64 as digits dig
// [batch][OZ_S][m][TC_LDK] with the row scales usc [batch][m].  b0: the batch's first matrix within the operand's
// sub-batch.  olim: elements of the operand (an index beyond is recorded in *err, code 65, and skipped).
// Bound by the latency of its loads: two CTAs an SM fit, the loads of one have only the other's FMAs (a tenth of the
// time) to hide behind, and DRAM runs at 11 % (0.47 ms for 160 matrices of n 1800).  The triangular solve it replaces ran
// column by column.
template <typename T>
__global__ void __launch_bounds__(256) lu_cols_kernel(T* Ar_base, T* Ai_base, long stride, int n, int k0, int kend,
                                                      const int* __restrict__ sw_base, const T* __restrict__ linv_base,
                                                      __nv_bfloat16* p0, __nv_bfloat16* p1, __nv_bfloat16* p2,
                                                      double* usc, long olim, int* err) {
  extern __shared__ __align__(16) unsigned char sm[];
  constexpr int W = TC_PW;                         // panel rows = columns a CTA
  T* O = reinterpret_cast<T*>(sm);                 // [2][W][W] the rows as they were; later [W][TC_LDK + 1]
  T* N = O + 2 * W * W;                            // [2][W][W] permuted
  T* V = N + 2 * W * W;                            // [2][W][W] L11^-1, [q][row]
  const int b = blockIdx.y;
  T* A[2] = {Ar_base + (long)b * stride, Ai_base + (long)b * stride};
  const int* sw = sw_base + (long)b * SW_LD;
  const int n_left = (k0 + W - 1) / W;
  const bool left = (int)blockIdx.x < n_left;
  const int j0 = left ? blockIdx.x * W : kend + (blockIdx.x - n_left) * W;
  const int nc = min(W, (left ? k0 : n) - j0);
  const int cnt = sw[0], pw = kend - k0;
  const int tid = threadIdx.x, cx = tid & (W - 1), ry = tid / W;       // 4 rows at a time
  for (int pl = 0; pl < 2; ++pl)
    for (int i = ry; i < pw; i += 4) {
      const int s = sw[2 + 2 * i];
      O[(pl * W + i) * W + cx] = cx < nc ? A[pl][(long)(k0 + i) * n + j0 + cx] : T(0);
      if (s >= kend) N[(pl * W + i) * W + cx] = cx < nc ? A[pl][(long)s * n + j0 + cx] : T(0);
    }
  if (!left)
    for (int i = tid; i < 2 * W * W; i += 256) V[i] = linv_base[(long)b * 2 * W * W + i];
  __syncthreads();
  for (int pl = 0; pl < 2; ++pl) {
    for (int i = ry; i < pw; i += 4) {
      const int s = sw[2 + 2 * i];
      if (s < kend) N[(pl * W + i) * W + cx] = O[(pl * W + s - k0) * W + cx];
    }
    for (int i = pw + ry; i < cnt; i += 4)         // rows below the panel receive rows of the panel only
      if (cx < nc) A[pl][(long)sw[1 + 2 * i] * n + j0 + cx] = O[(pl * W + sw[2 + 2 * i] - k0) * W + cx];
  }
  __syncthreads();
  if (left) {
    for (int pl = 0; pl < 2; ++pl)
      for (int i = ry; i < pw; i += 4)
        if (cx < nc) A[pl][(long)(k0 + i) * n + j0 + cx] = N[(pl * W + i) * W + cx];
    return;
  }
  // U12 tile: rows 4 ty + i, columns 4 tx + j (right columns exist only for full panels: pw = W)
  const int tx = tid & 15, ty = tid >> 4;
  T ur[4][4], ui[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) ur[i][j] = ui[i][j] = T(0);
  for (int q = 0; q < 4 * ty + 4; ++q) {           // L11^-1 is lower triangular
    T lr[4], li[4], br[4], bi[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      lr[i] = V[q * W + 4 * ty + i];
      li[i] = V[W * W + q * W + 4 * ty + i];
      br[i] = N[q * W + 4 * tx + i];
      bi[i] = N[W * W + q * W + 4 * tx + i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        ur[i][j] = fma(lr[i], br[j], ur[i][j]);
        ur[i][j] = fma(-li[i], bi[j], ur[i][j]);
        ui[i][j] = fma(lr[i], bi[j], ui[i][j]);
        ui[i][j] = fma(li[i], br[j], ui[i][j]);
      }
  }
  constexpr int OLD = TC_LDK + 1;
  T* R = O;                                        // [W][OLD] over O and N's start: N is read above
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int q = 4 * ty + i, c = 4 * tx + j;
      if (c < nc) {
        A[0][(long)(k0 + q) * n + j0 + c] = ur[i][j];
        A[1][(long)(k0 + q) * n + j0 + c] = ui[i][j];
      }
      R[c * OLD + q] = ur[i][j];
      R[c * OLD + W + q] = ui[i][j];
    }
  __syncthreads();
  const int m = n - kend;
  for (int it = tid; it < W * 16; it += 256) {     // 16 threads a column, eight elements each
    const int c = it >> 4, g = it & 15, cg = j0 - kend + c;
    T v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = R[c * OLD + 8 * g + t];
    if constexpr (sizeof(T) == 4) {
      const long o = ((long)b * m + cg) * TC_LDK + 8 * g;
      if (cg >= m) continue;
      if (o + 8 > olim) { atomicCAS(err, 0, 65); continue; }
      split3x8(v, p0 + o, p1 + o, p2 + o);
    } else {
      unsigned long long mx = 0;
#pragma unroll
      for (int t = 0; t < 8; ++t) mx = max(mx, oz::mag(v[t]));
#pragma unroll
      for (int s = 8; s > 0; s >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, s));
      const double sc = oz::scale_of(mx);
      if (cg >= m) continue;
      if (((long)(b + 1) * oz::S * m) * TC_LDK > olim) { atomicCAS(err, 0, 65); continue; }
      if (g == 0) usc[(long)b * m + cg] = sc;
      oz::store8(v, sc, p0 + (((long)b * oz::S) * m + cg) * TC_LDK + 8 * g, (long)m * TC_LDK);
    }
  }
}

// FP64 left operand of the update: rows r = [Re L_r, -Im L_r] and m + r = [Im L_r, Re L_r] as digits
// [batch][OZ_S][2 m][TC_LDK] with scales lsc [batch][2 m]; 16 threads a row.
__global__ void __launch_bounds__(128) lu_digits_l_kernel(const double* Ar_base, const double* Ai_base, long stride,
                                                          int n, int k0, int kend, __nv_bfloat16* dig, double* lsc,
                                                          long olim, int* err) {
  const int m = n - kend, b = blockIdx.y;
  const int r = blockIdx.x * 8 + (threadIdx.x >> 4), g = threadIdx.x & 15;
  const bool on = r < m;
  const double* A = (g < 8 ? Ar_base : Ai_base) + (long)b * stride + (long)(kend + (on ? r : 0)) * n + k0 + 8 * (g & 7);
  double v[8];
  unsigned long long mx = 0;
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    v[t] = on ? A[t] : 0.0;
    mx = max(mx, oz::mag(v[t]));
  }
#pragma unroll
  for (int s = 8; s > 0; s >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, s));
  const double sc = oz::scale_of(mx);
  if (!on) return;
  if (((long)(b + 1) * oz::S * 2 * m) * TC_LDK > olim) { atomicCAS(err, 0, 63); return; }
  if (g == 0) lsc[(long)b * 2 * m + r] = lsc[(long)b * 2 * m + m + r] = sc;
  __nv_bfloat16* base = dig + (long)b * oz::S * 2 * m * TC_LDK;
  const long dstr = 2L * m * TC_LDK;
  // Re: row r at its place, row m + r in the second half; Im: row m + r first half, negated in row r's second half
  oz::store8(v, sc, base + (long)(g < 8 ? r : m + r) * TC_LDK + 8 * (g & 7), dstr);
  if (g >= 8)
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = -v[t];
  oz::store8(v, sc, base + (long)(g < 8 ? m + r : r) * TC_LDK + TC_PW + 8 * (g & 7), dstr);
}

}  // namespace

namespace {
// Largest n that lu_panel_kernel holds in registers; beyond it lu_panel_global_kernel factors the panels.
template <typename T>
constexpr int panel_rows() { return (sizeof(T) == 4 ? 32 : 16) * LU_T; }

template <typename T, int RPT, int NB>
cudaError_t panel(T* A, long plane, long stride, int n, int batch, int k0, int kend, int* perm, int* info, int* sw,
                  T* linv, cudaStream_t s) {
  const size_t work = sizeof(T) * (2 * TC_PW * NB + 2 * NB * 2 * TC_PW) + sizeof(int) * (size_t)(n - k0);
  const size_t smem = sizeof(T) * 2 * TC_PW * (TC_PW + 1) + std::max(work, sizeof(T) * 2 * TC_PW * TC_PW);
  const cudaError_t e = allow_smem<lu_panel_kernel<T, RPT, NB>>();
  if (e != cudaSuccess) return e;
  lu_panel_kernel<T, RPT, NB><<<batch, LU_T, smem, s>>>(A, A + plane, stride, n, k0, kend, perm, info, sw, linv);
  return cudaGetLastError();
}

cudaError_t launch_panel(float* A, long plane, long stride, int n, int batch, int k0, int kend, int* perm, int* info,
                         int* sw, float* linv, cudaStream_t s) {
  const int rpt = (n - k0 + LU_T - 1) / LU_T;
  if (rpt <= 1) return panel<float, 1, 8>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  if (rpt <= 2) return panel<float, 2, 8>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  if (rpt <= 4) return panel<float, 4, 8>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  if (rpt <= 8) return panel<float, 8, 4>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  if (rpt <= 16) return panel<float, 16, 2>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  return panel<float, 32, 1>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
}

cudaError_t launch_panel(double* A, long plane, long stride, int n, int batch, int k0, int kend, int* perm, int* info,
                         int* sw, double* linv, cudaStream_t s) {
  const int rpt = (n - k0 + LU_T - 1) / LU_T;
  if (rpt <= 1) return panel<double, 1, 8>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  if (rpt <= 2) return panel<double, 2, 8>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  if (rpt <= 4) return panel<double, 4, 4>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  if (rpt <= 8) return panel<double, 8, 2>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
  return panel<double, 16, 1>(A, plane, stride, n, batch, k0, kend, perm, info, sw, linv, s);
}

template <typename T>
cudaError_t launch_cols(T* A, long plane, long stride, int n, int batch, int k0, int kend, const int* sw, const T* linv,
                        __nv_bfloat16* p0, __nv_bfloat16* p1, __nv_bfloat16* p2, double* usc, long olim, int* err,
                        cudaStream_t s) {
  const int smem = (int)sizeof(T) * (6 * TC_PW * TC_PW + TC_PW);
  const cudaError_t e = allow_smem<lu_cols_kernel<T>>();
  if (e != cudaSuccess) return e;
  const int gx = (k0 + TC_PW - 1) / TC_PW + (n - kend + TC_PW - 1) / TC_PW;
  if (gx > 0)
    lu_cols_kernel<T><<<dim3(gx, batch), 256, smem, s>>>(A, A + plane, stride, n, k0, kend, sw, linv, p0, p1, p2, usc,
                                                         olim, err);
  return cudaGetLastError();
}

template <typename T>
cudaError_t global_panel(T* A, long plane, long stride, int n, int batch, int k0, int kend, int* perm, int* info, int* sw,
                         T* linv, cudaStream_t s) {
  const int smem = (int)sizeof(T) * 2 * (TC_PW * (TC_PW + 1) + TC_PW * TC_PW);
  const cudaError_t e = allow_smem<lu_panel_global_kernel<T>>();
  if (e != cudaSuccess) return e;
  lu_panel_global_kernel<T><<<batch, LU_T, smem, s>>>(A, A + plane, stride, n, k0, kend, perm, info, sw, linv);
  return cudaGetLastError();
}
}  // namespace

// Per matrix and part: the left operand's 2 m rows and the right one's m rows of TC_LDK elements.
size_t zlu_operand_elems(int n, int batch, bool fp64) {
  const long m = n > TC_PW ? n - TC_PW : 0;
  return (size_t)(fp64 ? OZ_S : 3) * batch * 3 * m * TC_LDK;
}
size_t zlu_index_ints(int batch) { return (size_t)batch * SW_LD; }
size_t zlu_linv_elems(int batch) { return (size_t)batch * 2 * TC_PW * TC_PW; }
size_t zlu_scale_elems(int n, int batch) { return (size_t)batch * 3 * (n > TC_PW ? n - TC_PW : 0); }

template <typename T>
cudaError_t launch_zlu(T* A, long stride, long plane, int n, int batch, int* perm, int* info, __nv_bfloat16* work,
                       size_t work_elems, int* idx, T* linv, double* scales, int* err, cudaStream_t s) {
  constexpr bool D = sizeof(T) == 8;
  if (batch <= 0) return cudaSuccess;
  if (plane + (long)n * n > stride || batch > 65535) return cudaErrorInvalidValue;
  const bool global = n > panel_rows<T>();
  // the operands of one panel update are held for sub-batches of bs matrices
  const size_t per = zlu_operand_elems(n, 1, D);
  if (n > TC_PW && work_elems < per) return cudaErrorInvalidValue;
  const int bs = n > TC_PW ? (int)std::min<size_t>((size_t)batch, work_elems / per) : batch;
  for (int b0 = 0; b0 < batch; b0 += bs) {         // a sub-batch runs through all of its panels
    const int nb = std::min(bs, batch - b0);
    T* Ab = A + (long)b0 * stride;
    int* sw = idx;
    for (int k0 = 0; k0 < n; k0 += TC_PW) {
      const int kend = std::min(k0 + TC_PW, n);
      cudaError_t e =
          global ? global_panel(Ab, plane, stride, n, nb, k0, kend, perm + (long)b0 * n, info + b0, sw, linv, s)
                 : launch_panel(Ab, plane, stride, n, nb, k0, kend, perm + (long)b0 * n, info + b0, sw, linv, s);
      if (e != cudaSuccess) return e;
      const int m = n - kend;
      const long lsz = (long)nb * 2 * m * TC_LDK, usz = (long)nb * m * TC_LDK;     // elements of one part or digit
      if constexpr (D) {
        __nv_bfloat16* dl = work;
        __nv_bfloat16* du = work + OZ_S * lsz;
        double* sl = scales;
        double* su = scales + (long)nb * 2 * m;
        e = launch_cols<double>(Ab, plane, stride, n, nb, k0, kend, sw, linv, du, nullptr, nullptr, su, OZ_S * usz, err,
                                s);
        if (e != cudaSuccess || m == 0) { if (e != cudaSuccess) return e; break; }
        lu_digits_l_kernel<<<dim3((m + 7) / 8, nb), 128, 0, s>>>(Ab, Ab + plane, stride, n, k0, kend, dl, sl,
                                                                 OZ_S * lsz, err);
        OzEpi ep{};
        ep.kind = OZ_EPI_SUB2;
        ep.out = Ab + (long)kend * n + kend;
        ep.out_bstride = stride;
        ep.ldo = n;
        ep.plane = plane;
        ep.half = m;
        e = oz_gemm(OzOperand{dl, sl, 1}, OzOperand{du, su, 1}, nb, 2 * m, m, TC_LDK, ep, err, s);
        if (e != cudaSuccess) return e;
      } else {
        __nv_bfloat16* lp[3] = {work, work + lsz, work + 2 * lsz};
        __nv_bfloat16* ub[3] = {work + 3 * lsz, work + 3 * lsz + usz, work + 3 * lsz + 2 * usz};
        e = launch_cols<float>(Ab, plane, stride, n, nb, k0, kend, sw, linv, ub[0], ub[1], ub[2], nullptr, usz, err, s);
        if (e != cudaSuccess || m == 0) { if (e != cudaSuccess) return e; break; }
        const long limb = (long)(batch - b0) * stride;
        lu_split_l_kernel<<<dim3((m + 1) / 2, nb), 256, 0, s>>>(Ab, Ab + plane, stride, n, k0, kend, lp[0], lp[1],
                                                                 lp[2], limb, lsz, err);
        TcEpi ep{};
        ep.kind = TC_EPI_SUB2;
        ep.out = Ab + (long)kend * n + kend;
        ep.out_bstride = stride;
        ep.ldo = n;
        ep.plane = plane;
        ep.half = m;
        ep.limit = limb - ((long)kend * n + kend);
        const TcOperand ao{{lp[0], lp[1], lp[2]}}, bo{{ub[0], ub[1], ub[2]}};
        e = tc_gemm_ex(ao, nb, bo, 1, 3, 2 * m, m, TC_LDK, ep, err, s);
        if (e != cudaSuccess) return e;
      }
    }
  }
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_zlu_solve(const T* Ar, const T* Ai, long stride, int n, int batch, const int* perm, T* yr, T* yi,
                             long ystride, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  const size_t tri = sizeof(T) * (2 * SB * (SB + 1) + 2 * SB);
  if (n > panel_rows<T>()) {
    const cudaError_t e = allow_smem<zlu_solve_kernel<T, true>>();
    if (e != cudaSuccess) return e;
    zlu_solve_kernel<T, true><<<batch, LU_T, tri, s>>>(Ar, Ai, stride, n, perm, yr, yi, ystride);
    return cudaGetLastError();
  }
  const size_t smem = tri + sizeof(T) * 2 * (size_t)n;
  const cudaError_t e = allow_smem<zlu_solve_kernel<T, false>>();
  if (e != cudaSuccess) return e;
  zlu_solve_kernel<T, false><<<batch, LU_T, smem, s>>>(Ar, Ai, stride, n, perm, yr, yi, ystride);
  return cudaGetLastError();
}

template cudaError_t launch_zlu<float>(float*, long, long, int, int, int*, int*, __nv_bfloat16*, size_t, int*, float*,
                                       double*, int*, cudaStream_t);
template cudaError_t launch_zlu<double>(double*, long, long, int, int, int*, int*, __nv_bfloat16*, size_t, int*,
                                        double*, double*, int*, cudaStream_t);
template cudaError_t launch_zlu_solve<float>(const float*, const float*, long, int, int, const int*, float*, float*,
                                             long, cudaStream_t);
template cudaError_t launch_zlu_solve<double>(const double*, const double*, long, int, int, const int*, double*,
                                              double*, long, cudaStream_t);

}  // namespace gw
