// FP64 products on the BF16 tensor cores (after Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix
// multiplication", 2012): every operand row is scaled by a power of two to 63-bit integers and cut into eight balanced
// base-256 digits, which BF16 holds exactly;
//   A[m][k] B[n][k] = 2^(ea + eb - 124) sum_{i,j} a_i b_j 256^(14 - i - j),  a_i, b_j in [-128, 127],
// and the products with i + j = d (d <= 7; the rest is below 2^-64 of the rows' scales) are summed per d in the
// tensor core's FP32 accumulators over K = 128 at a time.  |a_i b_j| <= 2^14, so such a sum of at most 8 x 128 terms
// stays within 2^24 and every partial sum is an integer that FP32 holds: the tensor core adds without error.  The
// drain warps add the integers into two 64-bit fixed-point sums per element (d < 4 and d >= 4), again exactly, and one
// rounding to FP64 ends the element.
//
// Error: besides that rounding, an element is within K 2^-59 sa sb of the exact sum, sa and sb the powers of two of its
// two rows (the seven dropped products with i + j = 8 are up to 7 x 2^-62 of sa sb a term, the digits' own rounding
// 2^-62; typical is sqrt(K) 2^-62).  That is relative to the rows' largest elements, not to the sum of |terms| as an FP64
// chain's K 2^-53: it is the smaller of the two unless the sum of |terms| is below 2^-6 sa sb, which takes rows whose
// largest elements meet small ones.  Where that matters:
//   * weighted products sum_k x_mk w_k x_nk share the weight between the rows (x w 2^-h, rounded to FP64 once as a chain
//     rounds x w, and x 2^h, 4^h ~ |w|): whatever
//     the spread of the weights (a pair in resonance has 2/eta), sa sb is at most 8 times the geometric mean of the two
//     diagonal sums of |terms|, t_m and t_n.  The error is then below K 2^-56 sqrt(t_m t_n), an eighth of an FP64 chain's
//     bound in the same terms, which are those of the Cholesky factorisation that follows;
//   * polarizabilities handed to the caller are checked element by element (oz_cover) and tiles with a sum of |terms|
//     below sa sb / 8 are computed again on the FP64 pipe;
//   * in the other uses (inverse factors against rows of B, LU updates, y^T Pi' y, eigenvector refinement) the results are
//     no better than the rows' 2-norms allow, and K 2^-59 sa sb is below K 2^-57 |a| |b|, a sixteenth of an FP64 chain's.
//
// Why: FP64 runs at two multiply-adds a clock and SM on this chip (0.58 T/s in all), the digits' 36 BF16 products at
// about 50 times that in the tensor cores.  What bounds it: shared-memory reads of the M128 N64 K16 products (6 KiB
// each at 128 B a clock: 48 clocks, where the tensor core alone would take 32), then the drains, which the single
// TMEM buffer (8 sums x 64 columns = all 512) does not overlap with the next 128 of K.
#include "gw_internal.cuh"
#include "oz_gemm.cuh"
#include "oz_digits.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cstdint>

namespace gw {
namespace {
using namespace ptx;
using namespace oz;

constexpr int BM = 128, BN = 64, BK = 32;
constexpr int KCHUNK = 4;                        // k-blocks per exact sum (K = 128)
constexpr int STAGES = 2;
constexpr int A_BYTES = S * BM * BK * 2;         // 64 KiB
constexpr int B_BYTES = S * BN * BK * 2;         // 32 KiB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int BAR_OFF = STAGES * STAGE_BYTES;
constexpr int SMEM_BYTES = BAR_OFF + 1024 + 128;
constexpr int DRAIN_WARPS = 8;
constexpr int THREADS = 32 * (DRAIN_WARPS + 2);
constexpr uint32_t TMEM_COLS = 512;
static_assert(S * BN <= (int)TMEM_COLS, "one accumulator of BN columns per digit sum");
static_assert(SMEM_BYTES + 1024 <= 232448, "shared memory per block");
// kind::f16 instruction descriptor: D = F32, A = B = BF16, both K-major, N = 64, M = 128
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(BM >> 4) << 24);
constexpr uint32_t SBO64 = 8 * 64, SWZ64 = 4;    // 64-byte rows, 64-byte swizzle

struct OzMaps {
  CUtensorMap a, b;
};

// grid.x: tile, grid.y: entry.  Warps 0-7 drain (TMEM lane quarter = warp & 3, column half = warp >> 2),
// warp 8 TMA, warp 9 MMA.
__global__ void __launch_bounds__(THREADS, 1)
    oz_gemm_kernel(const __grid_constant__ OzMaps maps, int M, int N, int K, int a_batched, int b_batched,
                   const double* __restrict__ sca, const double* __restrict__ scb, const OzEpi ep,
                   int* __restrict__ err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  const uint32_t bar0 = base + BAR_OFF;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + BAR_OFF + 64);
  auto full = [bar0](int s) { return bar0 + 8u * (uint32_t)s; };
  auto empty = [bar0](int s) { return bar0 + 8u * (uint32_t)(STAGES + s); };
  const uint32_t acc_full = bar0 + 8u * (2 * STAGES), acc_empty = acc_full + 8u, fin = acc_full + 16u;
  __shared__ int s_abort;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.x, b = blockIdx.y;
  int bm, bn;
  if (ep.kind == OZ_EPI_STORE && ep.lower) {     // row block bm holds the column blocks 0 .. 2 bm + 1
    bm = (int)((sqrt(4.0 * tile + 1.0) - 1.0) * 0.5);
    while ((bm + 1) * (bm + 2) <= tile) ++bm;
    while (bm * (bm + 1) > tile) --bm;
    bn = tile - bm * (bm + 1);
  } else {
    const int nbn = (N + BN - 1) / BN;
    bm = tile / nbn;
    bn = tile % nbn;
  }
  const int m0 = bm * BM, n0 = bn * BN;
  if (m0 >= M || n0 >= N) return;                // the lower enumeration's last column block may lie past N
  const int nk = ((ep.kind == OZ_EPI_SUMSQ ? min(K, n0 + BN) : K) + BK - 1) / BK;

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, DRAIN_WARPS);
    mbar_init(fin, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == DRAIN_WARPS) {
    if (lane == 0) {
      // ---------------- TMA producer: one box of all eight digits per operand and k-block
      int issued = 0;
      bool ok = true;
      for (int kb = 0; kb < nk && ok; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES;
        if (u > 0 && !mbar_wait(empty(s), (u - 1) & 1, err, 71)) { ok = false; break; }
        if (*(volatile int*)&s_abort) { ok = false; break; }
        const uint32_t st = base + s * STAGE_BYTES;
        mbar_expect_tx(full(s), STAGE_BYTES);
        tma_load_3d(st, &maps.a, kb * BK, m0, a_batched ? b * S : 0, full(s));
        tma_load_3d(st + A_BYTES, &maps.b, kb * BK, n0, b_batched ? b * S : 0, full(s));
        issued = kb + 1;
      }
      if (!ok) {
        s_abort = 1;
        for (int kb = issued > STAGES ? issued - STAGES : 0; kb < issued; ++kb)
          mbar_wait(full(kb % STAGES), (kb / STAGES) & 1, err, 72);
      }
    }
  } else if (warp == DRAIN_WARPS + 1) {
    if (lane == 0) {
      // ---------------- MMA issuer
      const uint64_t dA = sdesc(base, SBO64, SWZ64), dB = sdesc(base + A_BYTES, SBO64, SWZ64);
      bool ok = true;
      for (int kb = 0; kb < nk && ok; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES, c = kb / KCHUNK;
        const bool first = kb % KCHUNK == 0;
        if (first && c > 0 && !mbar_wait(acc_empty, (c - 1) & 1, err, 73)) { ok = false; break; }
        if (!mbar_wait(full(s), u & 1, err, 74)) { ok = false; break; }
        if (*(volatile int*)&s_abort) { ok = false; break; }
        tc_fence_after();
        const uint64_t a0 = dA + (uint64_t)((s * STAGE_BYTES) >> 4), b0 = dB + (uint64_t)((s * STAGE_BYTES) >> 4);
#pragma unroll 1
        for (int k = 0; k < BK / 16; ++k) {
#pragma unroll 1
          for (int i = 0; i < S; ++i) {
            const uint64_t ad = a0 + (uint64_t)(i * ((BM * BK * 2) >> 4) + 2 * k);
            for (int j = 0; i + j < S; ++j)
              mma_bf16(tmem + (uint32_t)((i + j) * BN), ad, b0 + (uint64_t)(j * ((BN * BK * 2) >> 4) + 2 * k), IDESC,
                       (first && k == 0 && i == 0) ? 0u : 1u);
          }
        }
        mma_commit(empty(s));
        if (kb % KCHUNK == KCHUNK - 1 || kb == nk - 1) mma_commit(acc_full);
      }
      if (!ok) s_abort = 1;
      mma_commit(fin);             // every product issued above has completed once this flips
      mbar_wait(fin, 0, err, 76);
    }
  }
  bool ok = true;
  const int q = warp & 3, h = (warp >> 2) & 1;
  long long hi[32], lo[32];
  if (warp < DRAIN_WARPS) {
    // ---------------- drain: integers of the digit sums into the fixed-point sums
#pragma unroll
    for (int j = 0; j < 32; ++j) hi[j] = lo[j] = 0;
    const int nchunks = (nk + KCHUNK - 1) / KCHUNK;
    const uint32_t addr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * 32);
    for (int c = 0; c < nchunks; ++c) {
      ok = !*(volatile int*)&s_abort && mbar_wait(acc_full, c & 1, err, 75);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int d = 0; d < S; ++d) {
        uint32_t v[32];
        tmem_ld32(addr + (uint32_t)(d * BN), v);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int x = __float2int_rn(__uint_as_float(v[j]));
          if (d < 4) hi[j] += (long long)x * (1ll << (8 * (3 - d)));
          else lo[j] += (long long)x * (1ll << (8 * (7 - d)));
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    }
    if (!ok) s_abort = 1;
  }
  __syncwarp();
  const bool all_ok = __syncthreads_and(ok && !*(volatile int*)&s_abort) != 0;
  if (all_ok && warp < DRAIN_WARPS) {
    const int m = m0 + q * 32 + lane, c = n0 + h * 32;
    const double sm = m < M ? sca[(a_batched ? (long)b * M : 0) + m] * 1.4551915228366852e-11 : 0.0;   // 2^-36
    const double* sn = scb + (b_batched ? (long)b * N : 0);
    if (ep.kind == OZ_EPI_SUMSQ) {
      // this row's sum over the tile's columns; hi 2^12 + lo 2^-20 is within 2^-60 of the scales' product and needs
      // one conversion an element on the FP64 pipe instead of two
      double t = 0.0;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (c + j < N) {
          const double v = (double)((hi[j] << 12) + (lo[j] >> 20)) * sn[c + j];
          t = fma(v, v, t);
        }
      if (m < M)                                                                                    // 2^-24
        ep.part[((long)b * 2 * ((N + BN - 1) / BN) + 2 * bn + h) * M + m] = t * (sm * sm) * 5.9604644775390625e-08;
    } else if (ep.kind == OZ_EPI_SUB2) {
      if (m < M) {
        double* o = ep.out + (long)b * ep.out_bstride + (m < ep.half ? (long)m * ep.ldo
                                                                     : ep.plane + (long)(m - ep.half) * ep.ldo);
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (c + j < N) o[c + j] -= fma((double)lo[j], 2.3283064365386963e-10, (double)hi[j]) * sm * sn[c + j];
      }
    } else {
      const int mode = (b & 1) ? ep.mode_odd : ep.mode_even;
      double* o = ep.out + (long)b * ep.out_bstride;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const int n = c + j;
        if (m >= M || n >= N || (ep.lower && n > m)) continue;
        double v = fma((double)lo[j], 2.3283064365386963e-10, (double)hi[j]) * sm * sn[n];
        const long at = (long)m * ep.ldo + n;
        if (mode != 0) v = -v;
        if (ep.accumulate) v += o[at];
        else if (mode == 1 && m == n) v += 1.0;
        o[at] = v;
        if (ep.lower && n < m) o[(long)n * ep.ldo + m] = v;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// The tiles' sums of OZ_EPI_SUMSQ in ascending order, so that a table repeats itself bit for bit (roots of the QP search
// move by 1e-8 with the order near poles of Sigma).  One pass over part, 1/64 of the bytes of the rows' digits an entry.
__global__ void __launch_bounds__(256) oz_sumsq_add_kernel(const double* __restrict__ part, int tiles, int M,
                                                           double* __restrict__ W, int ldw,
                                                           const int* __restrict__ gidx) {
  const int m = blockIdx.x * 256 + threadIdx.x, b = blockIdx.y;
  if (m >= M) return;
  double s = 0.0;
  for (int t = 0; t < tiles; ++t) s += part[((long)b * tiles + t) * M + m];
  W[(long)m * ldw + gidx[b]] += s;
}

typedef CUresult (*PFN_encodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

PFN_encodeTiled encoder() {
  static PFN_encodeTiled fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_encodeTiled>(p);
  }
  return fn;
}

// [batch * S][rows][ld] digits, boxes of BK columns x box_rows rows x S digits.
bool map_digits(CUtensorMap* map, const void* ptr, int rows, int K, long planes, int box_rows) {
  PFN_encodeTiled enc = encoder();
  if (!enc || (reinterpret_cast<uintptr_t>(ptr) & 15)) return false;
  const cuuint64_t ld = (cuuint64_t)oz_ld(K);
  cuuint64_t dims[3] = {ld, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {ld * 2, ld * 2 * (cuuint64_t)rows};
  cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, (cuuint32_t)S};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ------------------------------------------------------------------ digits
// One thread: eight columns of one row of matrix blockIdx.z (stride xbs).
__global__ void __launch_bounds__(128) oz_split_kernel(const double* __restrict__ x, long xbs, int rows, int k0,
                                                       int cols, long ld, const double* __restrict__ sc,
                                                       __nv_bfloat16* __restrict__ dig, int ldd) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.z;
  const int c = 8 * g;
  if (c >= ldd) return;
  for (int r = blockIdx.y; r < rows; r += gridDim.y) {
    const int e = scale_exp(sc[(long)b * rows + r]);
    const double* xr = x + (long)b * xbs + (long)r * ld + k0;
    long long f[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) f[t] = to_fixed(c + t < cols ? xr[c + t] : 0.0, e);
    uint4 d[S];
    digits8(f, d);
#pragma unroll
    for (int i = 0; i < S; ++i)
      *reinterpret_cast<uint4*>(dig + (((long)b * S + i) * rows + r) * ldd + c) = d[i];
  }
}

// Biased exponent of a non-zero finite value (subnormals as 1), 0 for zero, 4096 for NaN and infinities.
__device__ __forceinline__ int exp_of(double v) {
  const unsigned long long m = mag(v);
  const int e = (int)(m >> 52);
  return e == 0x7ff ? 4096 : (e == 0 && m != 0 ? 1 : e);
}

// Scale of a row from the largest biased exponent of its non-zero elements (kNoExp: none, 4096 or more: NaN).
constexpr int kNoExp = -8192, kZeroWeight = -(1 << 20);
__device__ __forceinline__ double scale_from_exp(int mx) {
  if (mx == kNoExp) return 1.0;
  const int e = max(mx - 1022, -900);
  return e > 900 ? __longlong_as_double(0x7ff8000000000000ll) : __longlong_as_double((long long)(1023 + e) << 52);
}

// One CTA a row: digits and scale of x f (operand A) and, with PAIR, of x 2^h (operand B) for entry blockIdx.y, each row
// scaled to its own largest element.  A first pass over the row (cached) finds the two exponents.  One FP64 product an
// element and pass; the shift by h is integer arithmetic.
template <bool PAIR>
__global__ void __launch_bounds__(128) oz_split_weighted_kernel(const double* __restrict__ x, int rows, int k0, int cols,
                                                                long ld, const double* __restrict__ f,
                                                                const int* __restrict__ h, long ldw,
                                                                __nv_bfloat16* __restrict__ digA,
                                                                double* __restrict__ scA,
                                                                __nv_bfloat16* __restrict__ digB,
                                                                double* __restrict__ scB, int ldd) {
  __shared__ int red[2][4];
  const int r = blockIdx.x, b = blockIdx.y;
  const double* xr = x + (long)r * ld + k0;
  const double* fr = f + (long)b * ldw + k0;
  const int* hr = PAIR ? h + (long)b * ldw + k0 : nullptr;
  int ma = kNoExp, mb = kNoExp;
  for (int c = threadIdx.x; c < cols; c += 128) {
    const double v = xr[c];
    const int ea = exp_of(v * fr[c]);
    if (ea) ma = max(ma, ea);
    if (PAIR && hr[c] != kZeroWeight) {
      const int eb = exp_of(v);
      if (eb) mb = max(mb, eb >= 4096 ? eb : eb + hr[c]);
    }
  }
  ma = __reduce_max_sync(0xffffffffu, ma);
  mb = __reduce_max_sync(0xffffffffu, mb);
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = ma;
    red[1][threadIdx.x >> 5] = mb;
  }
  __syncthreads();
  for (int i = 0; i < 4; ++i) {
    ma = max(ma, red[0][i]);
    mb = max(mb, red[1][i]);
  }
  const double sa = scale_from_exp(ma), sb = scale_from_exp(mb);
  const int ea = scale_exp(sa), eb = scale_exp(sb);
  const long at = (long)b * rows + r;
  if (threadIdx.x == 0) {
    scA[at] = sa;
    if (PAIR) scB[at] = sb;
  }
  for (int c = 8 * (int)threadIdx.x; c < ldd; c += 8 * 128) {
    long long fa[8], fb[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const bool in = c + t < cols;
      const double v = in ? xr[c + t] : 0.0;
      fa[t] = to_fixed(in ? v * fr[c + t] : 0.0, ea);
      if (PAIR) {
        const int hk = in ? hr[c + t] : kZeroWeight;
        fb[t] = hk == kZeroWeight ? 0ll : to_fixed(v, eb - hk);
      }
    }
    uint4 d[S];
    digits8(fa, d);
#pragma unroll
    for (int i = 0; i < S; ++i) *reinterpret_cast<uint4*>(digA + (((long)b * S + i) * rows + r) * ldd + c) = d[i];
    if (PAIR) {
      digits8(fb, d);
#pragma unroll
      for (int i = 0; i < S; ++i) *reinterpret_cast<uint4*>(digB + (((long)b * S + i) * rows + r) * ldd + c) = d[i];
    }
  }
}

// Sums of |terms| of the lower 64 x 64 tiles of a digit product, from the two leading digits of each element in FP32: a
// tile where one is below sa sb / 8 (and neither row is zero), or where a row holds a NaN or an infinity (its scale is
// NaN), gets its flag.  flags [batch][tiles], tiles in the order of pi_syrk_kernel.  1/36 of the product's multiply-adds on the FP32 pipes: 2.3 ms for 129 entries of n 504, K 3040 at
// their peak, for products handed to the caller only.
constexpr int CT = 64, CKK = 16;
__global__ void __launch_bounds__(256) oz_cover_kernel(const __nv_bfloat16* __restrict__ digA,
                                                       const __nv_bfloat16* __restrict__ digB,
                                                       const double* __restrict__ scA, const double* __restrict__ scB,
                                                       int n, int ldd, int* __restrict__ flags) {
  __shared__ float As[CKK][CT + 4], Bs[CKK][CT + 4];
  const int t = blockIdx.x, b = blockIdx.y;
  int bi = (int)((sqrt(8.0 * t + 1.0) - 1.0) * 0.5);
  while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
  while (bi * (bi + 1) / 2 > t) --bi;
  const int bj = t - bi * (bi + 1) / 2, p0 = bi * CT, q0 = bj * CT;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lr = tid >> 2, lk = (tid & 3) * 4;
  const long plane = (long)n * ldd;
  const __nv_bfloat16* A = digA + (long)b * S * plane + (long)(p0 + lr) * ldd;
  const __nv_bfloat16* B = digB + (long)b * S * plane + (long)(q0 + lr) * ldd;
  auto load = [plane](const __nv_bfloat16* p, float (&v)[4]) {       // |x| / 2^e of four elements to 2^-14
    const __nv_bfloat162* d0 = reinterpret_cast<const __nv_bfloat162*>(p);
    const __nv_bfloat162* d1 = reinterpret_cast<const __nv_bfloat162*>(p + plane);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float2 a = __bfloat1622float2(d0[u]), c = __bfloat1622float2(d1[u]);
      v[2 * u] = fabsf(fmaf(a.x, 256.f, c.x)) * 0.00006103515625f;
      v[2 * u + 1] = fabsf(fmaf(a.y, 256.f, c.y)) * 0.00006103515625f;
    }
  };
  float acc[4][4], sa[4], sb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    sa[i] = sb[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  }
  for (int k0 = 0; k0 < ldd; k0 += CKK) {
    const int k = k0 + lk;
    float va[4] = {0.f, 0.f, 0.f, 0.f}, vb[4] = {0.f, 0.f, 0.f, 0.f};
    if (k < ldd && p0 + lr < n) load(A + k, va);             // ldd is a multiple of 8
    if (k < ldd && q0 + lr < n) load(B + k, vb);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      As[lk + u][lr] = va[u];
      Bs[lk + u][lr] = vb[u];
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < CKK; ++kk) {
      float a[4], c[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = As[kk][ty + 16 * i];
        c[i] = Bs[kk][tx + 16 * i];
        sa[i] += a[i];
        sb[i] += c[i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], c[j], acc[i][j]);
    }
    __syncthreads();
  }
  bool low = false;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int p = p0 + ty + 16 * i, q = q0 + tx + 16 * j;
      if (p >= n || q > p) continue;
      if (sa[i] > 0.f && sb[j] > 0.f && !(acc[i][j] >= 0.125f)) low = true;
      if (isnan(scA[(long)b * n + p]) || isnan(scB[(long)b * n + q])) low = true;
    }
  if (__syncthreads_or(low) && tid == 0) flags[(long)b * gridDim.x + t] = 1;
}

// Transposed operand: block of 32 source columns (operand rows) x 64 source rows through shared memory.
__global__ void __launch_bounds__(256) oz_split_t_kernel(const double* __restrict__ x, int rows, int cols, long ld,
                                                         const double* __restrict__ sc,
                                                         __nv_bfloat16* __restrict__ dig, int ldd) {
  __shared__ double t[64][33];
  const int c0 = blockIdx.x * 32, p0 = blockIdx.y * 64;
  for (int i = threadIdx.x; i < 64 * 32; i += 256) {
    const int p = p0 + (i >> 5), c = c0 + (i & 31);
    t[i >> 5][i & 31] = (p < rows && c < cols) ? x[(long)p * ld + c] : 0.0;
  }
  __syncthreads();
  const int cc = threadIdx.x >> 3, g = threadIdx.x & 7;     // 32 operand rows x 8 groups of eight
  const int c = c0 + cc, p = p0 + 8 * g;
  if (c >= cols || p >= ldd) return;
  const int e = scale_exp(sc[c]);
  long long f[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) f[u] = to_fixed(t[8 * g + u][cc], e);
  uint4 d[S];
  digits8(f, d);
#pragma unroll
  for (int i = 0; i < S; ++i) *reinterpret_cast<uint4*>(dig + ((long)i * cols + c) * ldd + p) = d[i];
}

__global__ void __launch_bounds__(256) oz_row_scale_kernel(const double* __restrict__ x, long cols, long ld,
                                                           double* __restrict__ sc) {
  __shared__ unsigned long long red[8];
  const long r = blockIdx.x;
  unsigned long long mx = 0;
  for (long k = threadIdx.x; k < cols; k += 256) {
    const unsigned long long v = (unsigned long long)__double_as_longlong(x[r * ld + k]) & 0x7fffffffffffffffull;
    mx = v > mx ? v : mx;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) mx = red[i] > mx ? red[i] : mx;
    sc[r] = scale_of(mx);
  }
}

__global__ void __launch_bounds__(256) oz_col_scale_kernel(const double* __restrict__ x, int rows, int cols, long ld,
                                                           double* __restrict__ sc) {
  __shared__ unsigned long long red[8][33];
  const int c = blockIdx.x * 32 + (threadIdx.x & 31), w = threadIdx.x >> 5;
  unsigned long long mx = 0;
  if (c < cols)
    for (int p = w; p < rows; p += 8) {
      const unsigned long long v = (unsigned long long)__double_as_longlong(x[(long)p * ld + c]) & 0x7fffffffffffffffull;
      mx = v > mx ? v : mx;
    }
  red[w][threadIdx.x & 31] = mx;
  __syncthreads();
  if (w == 0 && c < cols) {
    for (int i = 1; i < 8; ++i) mx = red[i][threadIdx.x] > mx ? red[i][threadIdx.x] : mx;
    sc[c] = scale_of(mx);
  }
}

// w = f 2^h with 4^h within a factor of two of |w|: the two rows of a weighted product get w 2^-h and 2^h.
__global__ void oz_weight_kernel(const double* __restrict__ Dk, int K, const int* __restrict__ kinds,
                                 const double* __restrict__ params, double eta, double* __restrict__ f,
                                 int* __restrict__ h) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
  if (k >= K) return;
  const int kind = kinds[b];
  const double D = Dk[k], p = params[b];
  double v;
  if (kind == 0) {
    v = -4.0 * D / (D * D + p * p);
  } else {
    const double a1 = p - D, a2 = -p - D, e2 = eta * eta;
    const double d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
    v = kind == 1 ? 2.0 * (a1 / d1 + a2 / d2) : 2.0 * (-eta / d1 - eta / d2);
  }
  const long at = (long)b * K + k;
  const int e = max(min((int)(mag(v) >> 52) - 1023, 1023), -1022), hh = (e + 1) >> 1;
  h[at] = v == 0.0 ? kZeroWeight : hh;
  f[at] = v * __longlong_as_double((long long)(1023 - hh) << 52);
}

// ------------------------------------------------------------------ derivative pass
__device__ __forceinline__ unsigned long long block_max(unsigned long long mx, unsigned long long* red) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = v > mx ? v : mx;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) mx = red[i] > mx ? red[i] : mx;
  return mx;
}

// Digits of one row by the whole block, eight columns a thread.
__device__ __forceinline__ void row_to_digits(const double* xr, int cols, int ldd, double sc, int rows, int r,
                                              __nv_bfloat16* dig) {
  const int e = scale_exp(sc);
  for (int c = 8 * (int)threadIdx.x; c < ldd; c += 8 * blockDim.x) {
    long long f[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) f[t] = to_fixed(c + t < cols ? xr[c + t] : 0.0, e);
    uint4 d[S];
    digits8(f, d);
#pragma unroll
    for (int i = 0; i < S; ++i) *reinterpret_cast<uint4*>(dig + ((long)i * rows + r) * ldd + c) = d[i];
  }
}

__global__ void __launch_bounds__(128) oz_row_digits_kernel(const double* __restrict__ x, int rows, int cols, long ld,
                                                            double* __restrict__ sc, __nv_bfloat16* __restrict__ dig,
                                                            int ldd) {
  __shared__ unsigned long long red[4];
  const int r = blockIdx.x;
  const double* xr = x + (long)r * ld;
  unsigned long long mx = 0;
  for (int c = threadIdx.x; c < cols; c += blockDim.x) mx = max(mx, mag(xr[c]));
  const double s = scale_of(block_max(mx, red));
  if (threadIdx.x == 0) sc[r] = s;
  row_to_digits(xr, cols, ldd, s, rows, r, dig);
}

__global__ void __launch_bounds__(256) oz_pole_derivative_kernel(const double* __restrict__ T, int K,
                                                                 const double* __restrict__ Dk,
                                                                 const double* __restrict__ xs, double eta,
                                                                 double* __restrict__ dw) {
  __shared__ double red[8];
  const int j = blockIdx.x;
  const double* t0 = T + (long)(2 * j) * K;
  const double* t1 = t0 + K;
  const double x = xs[j], e2 = eta * eta;
  double sum = 0.0;
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    const double tr = t0[k], ti = -t1[k], D = Dk[k];
    const double a1 = x - D, a2 = -x - D;
    const double d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
    const double q1r = (a1 * a1 - e2) / (d1 * d1), q1i = -2.0 * a1 * eta / (d1 * d1);
    const double q2r = (a2 * a2 - e2) / (d2 * d2), q2i = -2.0 * a2 * eta / (d2 * d2);
    const double cr = 2.0 * (-q1r + q2r), ci = 2.0 * (-q1i + q2i);
    sum += cr * (tr * tr - ti * ti) - ci * (2.0 * tr * ti);
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < 8; ++i) sum += red[i];
    dw[j] = sum;
  }
}

}  // namespace

int oz_sumsq_tiles(int N) { return 2 * ((N + BN - 1) / BN); }     // a warp's 32 columns each

cudaError_t oz_sumsq_add(const double* part, int batch, int tiles, int M, double* W, int ldw, const int* gidx,
                         cudaStream_t s) {
  if (batch > 65535) return cudaErrorInvalidValue;
  if (batch > 0 && M > 0)
    oz_sumsq_add_kernel<<<dim3((M + 255) / 256, batch), 256, 0, s>>>(part, tiles, M, W, ldw, gidx);
  return cudaGetLastError();
}

int oz_ld(int K) { return (K + 7) / 8 * 8; }
size_t oz_elems(int rows, int K) { return (size_t)S * rows * oz_ld(K); }

cudaError_t oz_gemm(const OzOperand& A, const OzOperand& B, int batch, int M, int N, int K, const OzEpi& ep, int* err,
                    cudaStream_t s) {
  if (batch <= 0 || M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidValue;
  OzMaps maps;
  if (!map_digits(&maps.a, A.dig, M, K, (long)S * (A.batched ? batch : 1), BM) ||
      !map_digits(&maps.b, B.dig, N, K, (long)S * (B.batched ? batch : 1), BN))
    return cudaErrorInvalidValue;
  static PerDevice attr;
  const cudaError_t ae = attr.run(
      [] { return cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES); });
  if (ae != cudaSuccess) return ae;
  const long nbm = (M + BM - 1) / BM, nbn = (N + BN - 1) / BN;
  const long tiles = ep.kind == OZ_EPI_STORE && ep.lower ? nbm * (nbm + 1) : nbm * nbn;
  oz_gemm_kernel<<<dim3((unsigned)tiles, batch), THREADS, SMEM_BYTES, s>>>(maps, M, N, K, A.batched, B.batched, A.sc, B.sc,
                                                                       ep, err);
  return cudaGetLastError();
}

cudaError_t oz_row_scale(const double* x, int rows, long cols, long ld, double* sc, cudaStream_t s) {
  if (rows > 0) oz_row_scale_kernel<<<rows, 256, 0, s>>>(x, cols, ld, sc);
  return cudaGetLastError();
}

cudaError_t oz_col_scale(const double* x, int rows, int cols, long ld, double* sc, cudaStream_t s) {
  if (cols > 0) oz_col_scale_kernel<<<(cols + 31) / 32, 256, 0, s>>>(x, rows, cols, ld, sc);
  return cudaGetLastError();
}

cudaError_t oz_split(const double* x, long xbs, int rows, int k0, int cols, long ld, const double* sc, int nb,
                     __nv_bfloat16* dig, cudaStream_t s) {
  const int ldd = oz_ld(cols);
  if (nb > 65535) return cudaErrorInvalidValue;
  if (rows > 0 && cols > 0 && nb > 0)
    oz_split_kernel<<<dim3((ldd / 8 + 127) / 128, std::min(rows, 65535), nb), 128, 0, s>>>(x, xbs, rows, k0, cols, ld, sc,
                                                                                          dig, ldd);
  return cudaGetLastError();
}

cudaError_t oz_split_weighted(const double* x, int rows, int k0, int cols, long ld, const double* f, const int* h,
                              long ldw, int nb, __nv_bfloat16* digA, double* scA, __nv_bfloat16* digB, double* scB,
                              cudaStream_t s) {
  const int ldd = oz_ld(cols);
  if (nb > 65535) return cudaErrorInvalidValue;
  if (rows <= 0 || cols <= 0 || nb <= 0) return cudaGetLastError();
  if (h)
    oz_split_weighted_kernel<true><<<dim3(rows, nb), 128, 0, s>>>(x, rows, k0, cols, ld, f, h, ldw, digA, scA, digB, scB,
                                                                  ldd);
  else
    oz_split_weighted_kernel<false><<<dim3(rows, nb), 128, 0, s>>>(x, rows, k0, cols, ld, f, h, ldw, digA, scA, digB, scB,
                                                                   ldd);
  return cudaGetLastError();
}

int oz_cover_tiles(int n) { return (n + CT - 1) / CT * ((n + CT - 1) / CT + 1) / 2; }

cudaError_t oz_cover(const OzOperand& A, const OzOperand& B, int n, int cols, int nb, int* flags, cudaStream_t s) {
  if (nb > 65535 || !A.batched || !B.batched) return cudaErrorInvalidValue;
  if (n > 0 && cols > 0 && nb > 0)
    oz_cover_kernel<<<dim3(oz_cover_tiles(n), nb), 256, 0, s>>>(A.dig, B.dig, A.sc, B.sc, n, oz_ld(cols), flags);
  return cudaGetLastError();
}

cudaError_t oz_split_transpose(const double* x, int rows, int cols, long ld, const double* sc, __nv_bfloat16* dig,
                               cudaStream_t s) {
  const int ldd = oz_ld(rows);
  if (rows > 0 && cols > 0)
    oz_split_t_kernel<<<dim3((cols + 31) / 32, (ldd + 63) / 64), 256, 0, s>>>(x, rows, cols, ld, sc, dig, ldd);
  return cudaGetLastError();
}

cudaError_t oz_pair_weights(const double* Dk, int K, const int* kinds, const double* params, double eta, int nb,
                            double* f, int* h, cudaStream_t s) {
  if (K > 0 && nb > 0) oz_weight_kernel<<<dim3((K + 255) / 256, nb), 256, 0, s>>>(Dk, K, kinds, params, eta, f, h);
  return cudaGetLastError();
}

cudaError_t oz_row_digits(const double* x, int rows, int cols, long ld, double* sc, __nv_bfloat16* dig,
                          cudaStream_t s) {
  if (rows > 0 && cols > 0) oz_row_digits_kernel<<<rows, 128, 0, s>>>(x, rows, cols, ld, sc, dig, oz_ld(cols));
  return cudaGetLastError();
}

cudaError_t oz_pole_derivative(const double* T, int K, const double* Dk, const double* xs, double eta, int nr,
                               double* dw, cudaStream_t s) {
  if (nr > 0) oz_pole_derivative_kernel<<<nr, 256, 0, s>>>(T, K, Dk, xs, eta, dw);
  return cudaGetLastError();
}

}  // namespace gw
