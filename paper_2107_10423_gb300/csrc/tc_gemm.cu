// tcgen05 (5th-generation tensor core) batched GEMM with BF16 split operands, used for the dense contractions of the
// mixed-precision path other than Pi (pi_fused.cu): Newton-Schulz products and the W reduction, the MINRES and
// refinement operators, the LU's trailing updates:
//   out_b[m][n] = f( sum_k A_b[m][k] * B_b[n][k] ),   A = Ahi + Alo (+ Alo2),  B = Bhi + Blo (+ Blo2)  (BF16)
// as Ahi*Bhi + Ahi*Blo + Alo*Bhi, or the six products of three parts, with FP32 accumulation in tensor memory (TMEM).
// Operands are staged by TMA (cp.async.bulk.tensor, 128-byte swizzle) into a 3-stage shared-memory
// ring; one elected thread issues tcgen05.mma; the accumulator is read back with tcgen05.ld.
// Every mbarrier wait is bounded: on timeout the kernel records an error code and unwinds.
#include "pi_tc.cuh"
#include "gw_internal.cuh"
#include "tc_ptx.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <algorithm>
#include <cstdint>
#include <cstdio>

namespace gw {
namespace {

constexpr int BM = 128, BN = 128, BK = 64, THREADS = 192;
constexpr int EPI_U = 8;         // epilogue elements per thread whose global reads are in flight together
constexpr int TILE_BYTES = BM * BK * 2;               // one 128 x 64 BF16 tile = 16 KiB

// NSP split parts per operand: 2 (hi, lo: products hh, hl, lh) or 3 (hi, mid, lo: the six products with
// part indices i + j <= 2, about FP32-accurate).  A stage holds NSP A tiles and NSP B tiles.
template <int NSP>
struct TcCfg {
  static constexpr int CHUNK = NSP == 2 ? 4 : 1;     // k-blocks per TMEM chunk before the drain
  static constexpr int STAGES = NSP == 2 ? 3 : 2;
  static constexpr int STAGE_BYTES = 2 * NSP * TILE_BYTES;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
  static_assert(BM * (BN + 1) * 4 + 3 * (BN + BM / 2) * 4 <= STAGES * STAGE_BYTES, "the staged tile reuses the ring");
};
// Two chunk buffers x two accumulators (hi*hi alone; every cross product together) x 128 columns.  Keeping the
// dominant hi*hi product apart leaves its accumulator one accumulate per k-step; the cross terms are 2^8
// smaller, so their accumulator's rounding is negligible.
constexpr uint32_t TMEM_COLS = 512;
constexpr long long WAIT_LIMIT = 1ll << 26;           // bounded spin on every mbarrier

// tcgen05 instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major, N = BN, M = BM.
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait; returns false (and records `code`) if the phase did not complete in time.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err, int code) {
  for (long long i = 0; i < WAIT_LIMIT; ++i)
    if (mbar_try(bar, parity)) return true;
  atomicCAS(err, 0, code);
  return false;
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor: K-major tile with 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused with 128-byte swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset
  d |= (uint64_t)1 << 46;                  // descriptor version
  d |= (uint64_t)2 << 61;                  // SWIZZLE_128B
  return d;
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(IDESC), "r"(accum)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Epilogues.  The tile is staged in shared memory as stg[BM][BN + 1] (row = output row), so any thread can combine
// elements of different rows (the complex pairs of the residue operator are adjacent rows).
__device__ __forceinline__ void split_store(float v, __nv_bfloat16* hi, __nv_bfloat16* lo, long o,
                                            __nv_bfloat16* lo2 = nullptr) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  hi[o] = h;
  const float r = v - __bfloat162float(h);
  const __nv_bfloat16 m = __float2bfloat16_rn(r);
  lo[o] = m;
  if (lo2) lo2[o] = __float2bfloat16_rn(r - __bfloat162float(m));
}

// a + b = s + (returned) without error (Knuth's TwoSum).
__device__ __forceinline__ float two_sum(float a, float b, float& s) {
  s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  return __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
}

// s += a b in three FP32 words (the exact product by an FMA error term, then TwoSums down to the third word): more bits
// than an FP64 sum, which would take three operations an element on the FP64 pipe (16 clocks a warp each) where this
// takes 22 on the FP32 pipes.
__device__ __forceinline__ void sum3_fma(float a, float b, float& s0, float& s1, float& s2) {
  const float p = __fmul_rn(a, b), pe = __fmaf_rn(a, b, -p);
  const float e0 = two_sum(s0, p, s0);
  const float e1 = two_sum(s1, pe, s1);
  const float e2 = two_sum(s1, e0, s1);
  s2 = __fadd_rn(s2, __fadd_rn(e1, e2));
}

// a + b as one FP32 value from the three words of each (a = a0 + a1 + a2 exactly), within an ulp whatever cancels.
__device__ __forceinline__ float sum3(float a0, float a1, float a2, float b0, float b1, float b2) {
  float s, t, u;
  const float e0 = two_sum(a0, b0, s), e1 = two_sum(a1, b1, t);
  const float e2 = two_sum(s, t, u);                   // the first words may cancel to the size of the second ones
  return __fadd_rn(u, __fadd_rn(e2, __fadd_rn(e0, __fadd_rn(e1, __fadd_rn(a2, b2)))));
}

// stg: [BM][TN + 1] staged tile; aux: 3 (TN + BM / 2) floats of shared memory.
template <int TN, int NTH>
__device__ void epilogue(const TcEpi& ep, const float* stg, float* aux, int m0, int n0, int M, int N, int b, int* err) {
  constexpr int LDS_ = TN + 1;
  if (ep.kind == TC_EPI_STORE) {
    float* o = ep.out + (long)b * ep.out_bstride;
    for (int idx = threadIdx.x; idx < BM * TN; idx += NTH) {
      const int rr = idx / TN, cc = idx % TN;
      const int m = m0 + rr, n = n0 + cc;
      if (m < M && n < N) o[(long)m * ep.ldo + n] = stg[rr * LDS_ + cc];
    }
  } else if (ep.kind == TC_EPI_CPAIR) {
    // rows (2j, 2j+1) hold B^T u and B^T v of z_j = u - i v; column k is the pair ia.
    // w = c_k(x_j) (t_r + i t_i) with t = B^T z, c_k(x) = 2[1/(x - D_k + i eta) + 1/(-x - D_k + i eta)];
    // Re w and Im w go to rows 2j, 2j+1 of the split operand of the second GEMM.  x and D enter as three FP32 words
    // (all 53 bits), split once a row and column: x - D in FP64 for every element was four operations on the FP64 pipe,
    // 8 us a tile.
    constexpr int XD = TN + BM / 2;                    // columns' D, then rows' x, per word
    for (int i = threadIdx.x; i < XD; i += NTH) {
      const bool col = i < TN;
      const int at = col ? n0 + i : (m0 >> 1) + i - TN;
      const double v = col ? (at < N ? ep.Dk[at] : 0.0) : (at < (M >> 1) ? ep.x[at] : 0.0);
      const float h = (float)v;
      const double r = v - (double)h;
      const float l = (float)r;
      aux[i] = h;
      aux[XD + i] = l;
      aux[2 * XD + i] = (float)(r - (double)l);
    }
    __syncthreads();
    const float e2 = ep.eta * ep.eta;
    for (int idx = threadIdx.x; idx < (BM / 2) * TN; idx += NTH) {
      const int pr = idx / TN, cc = idx % TN;
      const int m = m0 + 2 * pr, n = n0 + cc;
      if (m >= M || n >= N) continue;
      const float x0 = aux[TN + pr], x1 = aux[XD + TN + pr], x2 = aux[2 * XD + TN + pr];
      const float D0 = aux[cc], D1 = aux[XD + cc], D2 = aux[2 * XD + cc];
      const float a1 = sum3(x0, x1, x2, -D0, -D1, -D2), a2 = -sum3(x0, x1, x2, D0, D1, D2);
      const float d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
      const float cr = 2.f * (a1 / d1 + a2 / d2);
      const float ci = -2.f * ep.eta * (1.f / d1 + 1.f / d2);
      const float tr = stg[(2 * pr) * LDS_ + cc], ti = -stg[(2 * pr + 1) * LDS_ + cc];
      split_store(cr * tr - ci * ti, ep.ohi, ep.olo, (long)m * ep.ldh + n, ep.olo2);
      split_store(cr * ti + ci * tr, ep.ohi, ep.olo, (long)(m + 1) * ep.ldh + n, ep.olo2);
    }
  } else if (ep.kind == TC_EPI_AXPBY) {
    // two columns a thread (the split rows are 16-byte multiples, so pairs stay aligned); EPI_U pairs a pass, whose
    // global reads are issued together before any store
    for (int base = threadIdx.x; base < BM * TN / 2; base += NTH * EPI_U) {
      float2 xv[EPI_U];
#pragma unroll
      for (int u = 0; u < EPI_U; ++u) {
        const int idx = base + u * NTH, rr = idx / (TN / 2), cc = 2 * (idx % (TN / 2)), m = m0 + rr, n = n0 + cc;
        xv[u] = make_float2(0.f, 0.f);
        if (ep.xin && idx < BM * TN / 2 && m < M && n < N) {
          const float* x = ep.xin + (long)b * ep.x_bstride + (long)m * ep.ldo + n;
          xv[u].x = x[0];
          if (n + 1 < N) xv[u].y = x[1];
        }
      }
#pragma unroll
      for (int u = 0; u < EPI_U; ++u) {
        const int idx = base + u * NTH, rr = idx / (TN / 2), cc = 2 * (idx % (TN / 2)), m = m0 + rr, n = n0 + cc;
        if (idx >= BM * TN / 2 || m >= M || n >= N) continue;
        const float y0 = ep.gamma * stg[rr * LDS_ + cc] + (m == n ? ep.beta : 0.f) + ep.alpha * xv[u].x;
        const float y1 = n + 1 < N ? ep.gamma * stg[rr * LDS_ + cc + 1] + (m == n + 1 ? ep.beta : 0.f) +
                                         ep.alpha * xv[u].y
                                   : 0.f;              // the row's padding
        if (ep.out) {
          float* o = ep.out + (long)b * ep.out_bstride + (long)m * ep.ldo + n;
          o[0] = y0;
          if (n + 1 < N) o[1] = y1;
        }
        if (ep.ohi) {
          const long o = (long)b * ep.oh_bstride + (long)m * ep.ldh + n;
          const __nv_bfloat162 h = __floats2bfloat162_rn(y0, y1);
          const float r0 = y0 - __low2float(h), r1 = y1 - __high2float(h);
          const __nv_bfloat162 l = __floats2bfloat162_rn(r0, r1);
          *reinterpret_cast<__nv_bfloat162*>(ep.ohi + o) = h;
          *reinterpret_cast<__nv_bfloat162*>(ep.olo + o) = l;
          if (ep.olo2)
            *reinterpret_cast<__nv_bfloat162*>(ep.olo2 + o) = __floats2bfloat162_rn(r0 - __low2float(l),
                                                                                    r1 - __high2float(l));
        }
      }
    }
  } else if (ep.kind == TC_EPI_WRED) {
    // column n of the tile: sum over the tile's rows m of bvec[n][m] * v[m][n], added into W
    if (threadIdx.x < TN) {
      const int cc = threadIdx.x, n = n0 + cc;
      if (n < N) {
        const float* bv = ep.bvec + (long)n * ep.ldb + m0;
        float s0 = 0.f, s1 = 0.f, s2 = 0.f;
        const int rows = min(BM, M - m0);
#pragma unroll 8
        for (int rr = 0; rr < rows; ++rr) sum3_fma(bv[rr], stg[rr * LDS_ + cc], s0, s1, s2);
        atomicAdd(ep.W + (long)n * ep.wld + ep.gidx[b], (double)s0 + ((double)s1 + (double)s2));
      }
    }
  } else if (ep.kind == TC_EPI_PART) {
    float* o = ep.out + (long)blockIdx.z * M * N;
    for (int idx = threadIdx.x; idx < BM * TN; idx += NTH) {
      const int rr = idx / TN, cc = idx % TN, m = m0 + rr, n = n0 + cc;
      if (m < M && n < N) o[(long)m * N + n] = stg[rr * LDS_ + cc];
    }
  } else if (ep.kind == TC_EPI_SUB2) {
    float* o = ep.out + (long)b * ep.out_bstride;
    for (int base = threadIdx.x; base < BM * TN; base += NTH * EPI_U) {
      long off[EPI_U];
      float cv[EPI_U];
#pragma unroll
      for (int u = 0; u < EPI_U; ++u) {
        const int idx = base + u * NTH, rr = idx / TN, cc = idx % TN, m = m0 + rr, n = n0 + cc;
        off[u] = -1;
        if (idx < BM * TN && m < M && n < N) {
          const long o1 = m < ep.half ? (long)m * ep.ldo + n : ep.plane + (long)(m - ep.half) * ep.ldo + n;
          if ((long)b * ep.out_bstride + o1 >= ep.limit || o1 < 0) atomicCAS(err, 0, 66);
          else off[u] = o1;
        }
        cv[u] = off[u] >= 0 ? o[off[u]] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < EPI_U; ++u) {
        const int idx = base + u * NTH, rr = idx / TN, cc = idx % TN;
        if (off[u] >= 0) o[off[u]] = cv[u] - stg[rr * LDS_ + cc];
      }
    }
  } else if (ep.kind == TC_EPI_EMBED) {
    // real 2n embedding of (1 - Pi) z: rows 2j: u - (B w)_r, rows 2j+1: -v - (B w)_i
    for (int base = threadIdx.x; base < BM * TN; base += NTH * EPI_U) {
      float vv[EPI_U];
#pragma unroll
      for (int u = 0; u < EPI_U; ++u) {
        const int idx = base + u * NTH, rr = idx / TN, cc = idx % TN, m = m0 + rr, n = n0 + cc;
        vv[u] = (idx < BM * TN && m < M && n < N) ? ep.vin[(long)m * ep.ldv + n] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < EPI_U; ++u) {
        const int idx = base + u * NTH, rr = idx / TN, cc = idx % TN, m = m0 + rr, n = n0 + cc;
        if (idx >= BM * TN || m >= M || n >= N) continue;
        ep.out[(long)m * ep.ldo + n] = ((m & 1) ? -vv[u] : vv[u]) - stg[rr * LDS_ + cc];
      }
    }
  }
}

// grid.x: output tile, grid.y: batch entry, grid.z: K range.
// Warp roles: warps 0-3 drain the accumulator (TMEM lane quarter = warp), warp 4 issues TMA, warp 5 issues MMA.
// The contraction is cut into chunks of CHUNK k-blocks; each chunk accumulates in one of two TMEM buffers and
// is then added into FP32 registers by the drain warps (round to nearest), so no partial sum runs through more
// than 4 * CHUNK tensor-core accumulates of the dominant hi*hi product (the tensor-core accumulator loses about
// one ulp per accumulate, which over long K leaves a systematic relative error).
struct TcMaps {
  CUtensorMap a[3], b[3];
};

template <int NSP>
__global__ void __launch_bounds__(THREADS, 1)
    tc_gemm_kernel(const __grid_constant__ TcMaps maps, int M, int N, int K, int b_batched, const TcEpi ep, int* __restrict__ err) {
  constexpr int STAGES = TcCfg<NSP>::STAGES;
  constexpr int STAGE_BYTES = TcCfg<NSP>::STAGE_BYTES;
  constexpr int CHUNK = TcCfg<NSP>::CHUNK;
  if (ep.run_if && *ep.run_if == 0) return;     // uniform over the grid: nothing is allocated yet
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  // barriers: full[S], empty[S], acc_full[2], acc_empty[2]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 4);
  __shared__ int s_abort;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nbn = (N + BN - 1) / BN;
  const int bm = blockIdx.x / nbn, bn = blockIdx.x % nbn;
  const int m0 = bm * BM, n0 = bn * BN, b = blockIdx.y;
  // this CTA's range of k-blocks (grid.z > 1: TC_EPI_PART)
  const int nk_all = (K + BK - 1) / BK, kb0 = (int)((long)nk_all * blockIdx.z / gridDim.z);
  const int nk = (int)((long)nk_all * (blockIdx.z + 1) / gridDim.z) - kb0;
  const int nchunks = (nk + CHUNK - 1) / CHUNK;

  uint32_t full[STAGES], empty[STAGES];
  for (int s = 0; s < STAGES; ++s) {
    full[s] = smem_u32(&bars[s]);
    empty[s] = smem_u32(&bars[STAGES + s]);
  }
  const uint32_t acc_full[2] = {smem_u32(&bars[2 * STAGES]), smem_u32(&bars[2 * STAGES + 1])};
  const uint32_t acc_empty[2] = {smem_u32(&bars[2 * STAGES + 2]), smem_u32(&bars[2 * STAGES + 3])};

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full[s], 1);
      mbar_init(empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(acc_full[i], 1);
      mbar_init(acc_empty[i], 4);      // one arrival per drain warp
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  float acc[BN];                    // drain warps: FP32 sum of the chunk partials for row (warp*32 + lane)
  bool ok = true;
  int issued = 0;
  if (warp == 4) {
    if (lane == 0) {
      // ---------------- TMA producer
      for (int kb = 0; kb < nk; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES;
        if (u > 0 && !mbar_wait(empty[s], (u - 1) & 1, err, 1)) { s_abort = 1; break; }
        if (*(volatile int*)&s_abort) break;
        const uint32_t st = base + s * STAGE_BYTES;
        mbar_expect_tx(full[s], STAGE_BYTES);
#pragma unroll
        for (int i = 0; i < NSP; ++i) tma_load_3d(st + i * TILE_BYTES, &maps.a[i], (kb0 + kb) * BK, m0, b, full[s]);
#pragma unroll
        for (int j = 0; j < NSP; ++j)
          tma_load_3d(st + (NSP + j) * TILE_BYTES, &maps.b[j], (kb0 + kb) * BK, n0, b_batched ? b : 0, full[s]);
        issued = kb + 1;
      }
    }
  } else if (warp == 5) {
    if (lane == 0) {
      // ---------------- MMA issuer
      for (int kb = 0; kb < nk && !*(volatile int*)&s_abort; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES;
        const int c = kb / CHUNK, buf = c & 1, first = (kb % CHUNK) == 0;
        if (first && c >= 2 && !mbar_wait(acc_empty[buf], ((c >> 1) - 1) & 1, err, 5)) { s_abort = 1; break; }
        if (!mbar_wait(full[s], u & 1, err, 2)) { s_abort = 1; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t st = base + s * STAGE_BYTES;
        const uint32_t dbig = tmem + (uint32_t)(buf * 2 * BN), dsmall = dbig + BN;
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) {
          const uint32_t off = k * 32;
#pragma unroll
          for (int i = 0; i < NSP; ++i)
#pragma unroll
            for (int j = 0; j + i < NSP; ++j) {
              const uint64_t ad = sdesc(st + i * TILE_BYTES + off), bd = sdesc(st + (NSP + j) * TILE_BYTES + off);
              const bool is_big = (i == 0 && j == 0);
              const bool first_in_acc = first && k == 0 && (is_big || (i == 0 && j == 1));
              mma_bf16(is_big ? dbig : dsmall, ad, bd, first_in_acc ? 0u : 1u);
            }
        }
        mma_commit(empty[s]);
        if ((kb % CHUNK) == CHUNK - 1 || kb == nk - 1) mma_commit(acc_full[buf]);
      }
    }
  } else {
    // ---------------- drain warps 0-3
#pragma unroll
    for (int j = 0; j < BN; ++j) acc[j] = 0.f;
    for (int c = 0; c < nchunks; ++c) {
      const int buf = c & 1;
      ok = mbar_wait(acc_full[buf], (c >> 1) & 1, err, 3);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int q = 0; q < BN / 32; ++q) {
        uint32_t v[32], w[32];
        const uint32_t col = (uint32_t)(buf * 2 * BN + q * 32);
        tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + col, v);
        tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16) + col + BN, w);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[q * 32 + j] += __uint_as_float(v[j]) + __uint_as_float(w[j]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty[buf]) : "memory");
    }
  }
  __syncwarp();
  const bool all_ok = __syncthreads_and(ok && !s_abort) != 0;
  // drain copies still in flight if the pipeline was aborted
  if (!all_ok && warp == 4 && lane == 0)
    for (int kb = 0; kb < issued; ++kb) mbar_wait(full[kb % STAGES], (kb / STAGES) & 1, err, 4);
  __syncthreads();
  float* stg = reinterpret_cast<float*>(smem);     // [BM][BN + 1], reuses the operand ring
  if (all_ok && warp < 4) {
    const int r = warp * 32 + lane;
#pragma unroll
    for (int j = 0; j < BN; ++j) stg[r * (BN + 1) + j] = acc[j];
  }
  __syncthreads();
  if (all_ok) epilogue<BN, THREADS>(ep, stg, stg + BM * (BN + 1), m0, n0, M, N, b, err);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------ 128 x 256 tiles
// The same product in M128 N256 instructions.  What bounds it: L2 -> SM traffic (about 37 B a clock and SM on this
// chip) and shared-memory reads; a 128 x 128 tile moves 64 (three parts) or 85 B a clock at full tensor rate, this one
// 47 or 62, and reads 12 KiB of shared memory per 128 clocks instead of 16.
// Accumulators: TMEM columns [0, 256) the hi*hi sum of BIGC k-blocks (of 32), [256, 512) the cross terms of SMALLC.
// A k-block's cross terms are issued first, so the drain of the previous hi*hi sum runs beside them; the cross terms are
// 2^-8 of the sum, so their accumulator may run four times as long for the same error.  Eight drain warps (TMEM lane
// quarter = warp & 3, column half = warp >> 2) add both into FP32 registers, rounded to nearest.
constexpr int WN = 256, WK = 32;
template <int NSP>
struct WideCfg {
  static constexpr int BIGC = NSP == 2 ? 8 : 2, SMALLC = 4 * BIGC;
  static constexpr int STAGES = NSP == 2 ? 4 : 3;
  static constexpr int A_TILE = BM * WK * 2, B_TILE = WN * WK * 2;
  static constexpr int STAGE_BYTES = NSP * (A_TILE + B_TILE);
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
  static_assert(BM * (WN + 1) * 4 + 3 * (WN + BM / 2) * 4 <= STAGES * STAGE_BYTES, "the staged tile reuses the ring");
};
constexpr long kWideMinTiles = 120;
constexpr int WDRAIN = 8, WTHREADS = 32 * (WDRAIN + 2);
constexpr uint32_t WIDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(WN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

template <int NSP>
__global__ void __launch_bounds__(WTHREADS, 1)
    tc_gemm_wide_kernel(const __grid_constant__ TcMaps maps, int M, int N, int K, int b_batched, const TcEpi ep,
                        int* __restrict__ err) {
  using C = WideCfg<NSP>;
  constexpr int STAGES = C::STAGES;
  if (ep.run_if && *ep.run_if == 0) return;     // uniform over the grid: nothing is allocated yet
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  const uint32_t bar0 = base + STAGES * C::STAGE_BYTES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + STAGES * C::STAGE_BYTES + 128);
  auto full = [bar0](int s) { return bar0 + 8u * (uint32_t)s; };
  auto empty = [bar0](int s) { return bar0 + 8u * (uint32_t)(STAGES + s); };
  const uint32_t acc_full = bar0 + 8u * (2 * STAGES), big_empty = acc_full + 8u, small_empty = acc_full + 16u,
                 fin = acc_full + 24u;
  __shared__ int s_abort;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nbn = (N + WN - 1) / WN;
  const int m0 = (blockIdx.x / nbn) * BM, n0 = (blockIdx.x % nbn) * WN, b = blockIdx.y;
  const int nk = (K + WK - 1) / WK;

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(big_empty, WDRAIN);
    mbar_init(small_empty, WDRAIN);
    mbar_init(fin, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  float acc[128];
  bool ok = true;
  if (warp == WDRAIN) {
    if (lane == 0) {
      // ---------------- TMA producer
      int issued = 0;
      bool go = true;
      for (int kb = 0; kb < nk && go; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES;
        if (u > 0 && !mbar_wait(empty(s), (u - 1) & 1, err, 1)) go = false;
        if (!go || *(volatile int*)&s_abort) { go = false; break; }
        const uint32_t st = base + s * C::STAGE_BYTES;
        mbar_expect_tx(full(s), C::STAGE_BYTES);
#pragma unroll
        for (int i = 0; i < NSP; ++i) tma_load_3d(st + i * C::A_TILE, &maps.a[i], kb * WK, m0, b, full(s));
#pragma unroll
        for (int j = 0; j < NSP; ++j)
          tma_load_3d(st + NSP * C::A_TILE + j * C::B_TILE, &maps.b[j], kb * WK, n0, b_batched ? b : 0, full(s));
        issued = kb + 1;
      }
      if (!go) {
        s_abort = 1;
        for (int kb = issued > STAGES ? issued - STAGES : 0; kb < issued; ++kb)
          mbar_wait(full(kb % STAGES), (kb / STAGES) & 1, err, 4);
      }
    }
  } else if (warp == WDRAIN + 1) {
    if (lane == 0) {
      // ---------------- MMA issuer
      bool go = true;
      uint32_t nbig = 0, nsmall = 0;
      const uint64_t dA = ptx::sdesc(base, 8 * 64, 4), dB = ptx::sdesc(base + NSP * C::A_TILE, 8 * 64, 4);
      for (int kb = 0; kb < nk; ++kb) {
        const int s = kb % STAGES, u = kb / STAGES;
        const bool bfirst = kb % C::BIGC == 0, sfirst = kb % C::SMALLC == 0;
        if (!mbar_wait(full(s), u & 1, err, 2)) { go = false; break; }
        if (*(volatile int*)&s_abort) { go = false; break; }
        if (sfirst && kb > 0) {
          if (!mbar_wait(small_empty, nsmall & 1u, err, 6)) { go = false; break; }
          ++nsmall;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t a0 = dA + (uint64_t)((s * C::STAGE_BYTES) >> 4), b0 = dB + (uint64_t)((s * C::STAGE_BYTES) >> 4);
#pragma unroll
        for (int k = 0; k < WK / 16; ++k)
#pragma unroll
          for (int i = 0; i < NSP; ++i)
#pragma unroll
            for (int j = 0; j + i < NSP; ++j)
              if (i + j > 0)
                ptx::mma_bf16(tmem + WN, a0 + (uint64_t)((i * C::A_TILE) >> 4) + 2 * k,
                              b0 + (uint64_t)((j * C::B_TILE) >> 4) + 2 * k, WIDESC,
                              (sfirst && k == 0 && i == 0 && j == 1) ? 0u : 1u);
        if (bfirst && kb > 0) {
          if (!mbar_wait(big_empty, nbig & 1u, err, 5)) { go = false; break; }
          ++nbig;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
#pragma unroll
        for (int k = 0; k < WK / 16; ++k)
          ptx::mma_bf16(tmem, a0 + 2 * k, b0 + 2 * k, WIDESC, (bfirst && k == 0) ? 0u : 1u);
        mma_commit(empty(s));
        if (kb % C::BIGC == C::BIGC - 1 || kb == nk - 1) mma_commit(acc_full);
      }
      if (!go) s_abort = 1;
      mma_commit(fin);             // every product issued above has completed once this flips
      mbar_wait(fin, 0, err, 7);
    }
  } else {
    // ---------------- drain warps
    const uint32_t addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 128);
#pragma unroll
    for (int j = 0; j < 128; ++j) acc[j] = 0.f;
    const int nchunks = (nk + C::BIGC - 1) / C::BIGC;
    for (int c = 0; c < nchunks; ++c) {
      ok = !*(volatile int*)&s_abort && mbar_wait(acc_full, c & 1, err, 3);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        uint32_t v[32];
        tmem_ld32(addr + (uint32_t)(g * 32), v);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[g * 32 + j] += __uint_as_float(v[j]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(big_empty) : "memory");
      if (c % (C::SMALLC / C::BIGC) == C::SMALLC / C::BIGC - 1 || c == nchunks - 1) {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint32_t v[32];
          tmem_ld32(addr + (uint32_t)(WN + g * 32), v);
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[g * 32 + j] += __uint_as_float(v[j]);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(small_empty) : "memory");
      }
    }
    if (!ok) s_abort = 1;
  }
  __syncwarp();
  const bool all_ok = __syncthreads_and(ok && !*(volatile int*)&s_abort) != 0;
  float* stg = reinterpret_cast<float*>(smem);     // [BM][WN + 1], reuses the operand ring
  if (all_ok && warp < WDRAIN) {
    const int r = (warp & 3) * 32 + lane, c = (warp >> 2) * 128;
#pragma unroll
    for (int j = 0; j < 128; ++j) stg[r * (WN + 1) + c + j] = acc[j];
  }
  __syncthreads();
  if (all_ok) epilogue<WN, WTHREADS>(ep, stg, stg + BM * (WN + 1), m0, n0, M, N, b, err);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

typedef CUresult (*PFN_encodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

PFN_encodeTiled get_encode() {
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

bool make_map(CUtensorMap* map, const void* ptr, int rows, int K, int ld, int batch, int box_k, int box_rows,
              CUtensorMapSwizzle swz) {
  PFN_encodeTiled enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)ld * 2 * rows};
  cuuint32_t box[3] = {(cuuint32_t)box_k, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, batch > 0 ? 3 : 2, const_cast<void*>(ptr), dims, strides,
                   box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace

int tc_ld(int K) { return (K + 7) / 8 * 8; }

cudaError_t tc_gemm_ex(const TcOperand& A, int batch, const TcOperand& B, int b_batched, int nsplit, int M, int N,
                       int K, const TcEpi& ep, int* err, cudaStream_t s) {
  const int ld = tc_ld(K);
  TcMaps maps;
  const int bb = b_batched ? batch : 1;
  if (nsplit != 2 && nsplit != 3) return cudaErrorInvalidValue;
  // 128 x 256 tiles wherever they are enough CTAs for the chip; products of fewer tiles and split-K products run in
  // 128 x 128 tiles, twice the CTAs
  const long nbm = (M + BM - 1) / BM, wide_tiles = nbm * ((N + WN - 1) / WN);
  const bool wide = ep.kind != TC_EPI_PART && N > BN && wide_tiles * batch >= kWideMinTiles;
  for (int i = 0; i < nsplit; ++i)
    if (!A.p[i] || !B.p[i] ||
        !make_map(&maps.a[i], A.p[i], M, K, ld, batch, wide ? WK : BK, BM,
                  wide ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map(&maps.b[i], B.p[i], N, K, ld, bb, wide ? WK : BK, wide ? WN : BN,
                  wide ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
  static PerDevice attr;
  const cudaError_t ae = attr.run([] {
    cudaError_t e = cudaFuncSetAttribute(tc_gemm_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         TcCfg<2>::SMEM_BYTES);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(tc_gemm_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcCfg<3>::SMEM_BYTES);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(tc_gemm_wide_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               WideCfg<2>::SMEM_BYTES);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(tc_gemm_wide_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               WideCfg<3>::SMEM_BYTES);
    return e;
  });
  if (ae != cudaSuccess) return ae;
  if (wide) {
    const dim3 grid((unsigned)wide_tiles, batch);
    if (nsplit == 2)
      tc_gemm_wide_kernel<2><<<grid, WTHREADS, WideCfg<2>::SMEM_BYTES, s>>>(maps, M, N, K, b_batched, ep, err);
    else
      tc_gemm_wide_kernel<3><<<grid, WTHREADS, WideCfg<3>::SMEM_BYTES, s>>>(maps, M, N, K, b_batched, ep, err);
    return cudaGetLastError();
  }
  const dim3 grid((unsigned)(nbm * ((N + BN - 1) / BN)), batch, ep.kind == TC_EPI_PART ? std::max(1, ep.ksplit) : 1);
  if (nsplit == 2)
    tc_gemm_kernel<2><<<grid, THREADS, TcCfg<2>::SMEM_BYTES, s>>>(maps, M, N, K, b_batched, ep, err);
  else
    tc_gemm_kernel<3><<<grid, THREADS, TcCfg<3>::SMEM_BYTES, s>>>(maps, M, N, K, b_batched, ep, err);
  return cudaGetLastError();
}

// out[r][c] = s (mode 0) or the embedding (r odd ? -vin : vin) - s (mode 1), s = the ksplit partial products in order.
__global__ void __launch_bounds__(256) tc_part_reduce_kernel(const float* __restrict__ part, int ksplit, long N, int n,
                                                             const float* __restrict__ vin, int mode,
                                                             float* __restrict__ out, const int* __restrict__ run_if) {
  if (run_if && *run_if == 0) return;
  for (long i = blockIdx.x * 256L + threadIdx.x; i < N; i += gridDim.x * 256L) {
    float s = 0.f;
    for (int q = 0; q < ksplit; ++q) s += part[q * N + i];
    if (mode == 1) s = (((i / n) & 1) ? -vin[i] : vin[i]) - s;
    out[i] = s;
  }
}

cudaError_t tc_part_reduce(const float* part, int ksplit, int rows, int n, const float* vin, int mode, float* out,
                           const int* run_if, cudaStream_t s) {
  const long N = (long)rows * n;
  if (N > 0)
    tc_part_reduce_kernel<<<(unsigned)std::min<long>((N + 255) / 256, 2048), 256, 0, s>>>(part, ksplit, N, n, vin, mode,
                                                                                          out, run_if);
  return cudaGetLastError();
}

// K ranges for a product of few tiles: about one wave of CTAs, each with at least eight k-blocks.
int tc_ksplit(int M, int N, int K) {
  const int tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN), nk = (K + BK - 1) / BK;
  return std::max(1, std::min(nk / 8, 152 / std::max(1, tiles)));
}

// B^T split: out[k][m] = B[m][k] as BF16 hi/lo, rows of length tc_ld(M).  32 x 32 tiles through shared memory.
__global__ void transpose_split_kernel(const float* __restrict__ B, int M, int K, long ldb, int ld,
                                       __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                       __nv_bfloat16* __restrict__ lo2) {
  __shared__ float t[32][33];
  const int k0 = blockIdx.x * 32, m0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int m = m0 + r, k = k0 + threadIdx.x;
    t[r][threadIdx.x] = (m < M && k < K) ? B[(long)m * ldb + k] : 0.f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = k0 + r, m = m0 + threadIdx.x;
    if (k < K && m < ld) split_store(m < M ? t[threadIdx.x][r] : 0.f, hi, lo, (long)k * ld + m, lo2);
  }
}

__global__ void split_rows_kernel(const float* __restrict__ src, int cols, int lds, __nv_bfloat16* __restrict__ hi,
                                  __nv_bfloat16* __restrict__ lo, __nv_bfloat16* __restrict__ lo2, int ldh) {
  const long r = blockIdx.y + (long)blockIdx.z * gridDim.y;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ldh; c += gridDim.x * blockDim.x)
    split_store(c < cols ? src[r * lds + c] : 0.f, hi, lo, r * ldh + c, lo2);
}

cudaError_t tc_split_rows(const float* src, int rows, int cols, int lds, __nv_bfloat16* hi, __nv_bfloat16* lo,
                          cudaStream_t s, __nv_bfloat16* lo2) {
  const int ldh = tc_ld(cols);
  if (rows <= 0) return cudaSuccess;
  int gy = rows, gz = 1;
  while (gy > 65535) { gz *= 2; gy = (rows + gz - 1) / gz; }
  if ((long)gy * gz != rows) {
    // rows not a multiple of the z split: run the tail separately
    const int main = (rows / gz) * gz;
    if (main > 0) split_rows_kernel<<<dim3((ldh + 255) / 256, main / gz, gz), 256, 0, s>>>(src, cols, lds, hi, lo, lo2, ldh);
    const int tail = rows - main;
    split_rows_kernel<<<dim3((ldh + 255) / 256, tail, 1), 256, 0, s>>>(src + (long)main * lds, cols, lds,
                                                                     hi + (long)main * ldh, lo + (long)main * ldh,
                                                                     lo2 ? lo2 + (long)main * ldh : nullptr, ldh);
    return cudaGetLastError();
  }
  split_rows_kernel<<<dim3((ldh + 255) / 256, gy, gz), 256, 0, s>>>(src, cols, lds, hi, lo, lo2, ldh);
  return cudaGetLastError();
}

// Power iterations for the spectrum of SPD matrices A_b (n x n FP32, batch stride n*n), many CTAs per matrix:
//   gemv:      y_b = A_b v_b (mode 0)  or  y_b = s_b v_b - A_b v_b (mode 1), one warp per row;
//   normalise: q_b = v_b . y_b (the Rayleigh quotient of the unit vector v_b), v_b = y_b / |y_b|.
__global__ void spec_gemv_kernel(const float* __restrict__ A, int n, const float* __restrict__ v,
                                 const float* __restrict__ shift, int mode, float* __restrict__ y) {
  const int b = blockIdx.y, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = blockIdx.x * (blockDim.x >> 5) + wid;
  if (r >= n) return;
  const float* Ar = A + ((long)b * n + r) * n;
  const float* vb = v + (long)b * n;
  float a = 0.f;
  for (int c = lane; c < n; c += 32) a += Ar[c] * vb[c];
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) y[(long)b * n + r] = mode ? shift[b] * vb[r] - a : a;
}

__global__ void spec_normalise_kernel(int n, float* __restrict__ v, const float* __restrict__ y,
                                      float* __restrict__ q) {
  __shared__ float red[2][32];
  const int b = blockIdx.x;
  float* vb = v + (long)b * n;
  const float* yb = y + (long)b * n;
  float yy = 0.f, vy = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    yy += yb[i] * yb[i];
    vy += vb[i] * yb[i];
  }
  for (int o = 16; o > 0; o >>= 1) {
    yy += __shfl_xor_sync(0xffffffffu, yy, o);
    vy += __shfl_xor_sync(0xffffffffu, vy, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = yy;
    red[1][threadIdx.x >> 5] = vy;
  }
  __syncthreads();
  float tyy = 0.f, tvy = 0.f;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    tyy += red[0][w];
    tvy += red[1][w];
  }
  __syncthreads();
  const float inv = tyy > 0.f ? rsqrtf(tyy) : 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) vb[i] = yb[i] * inv;
  if (threadIdx.x == 0) q[b] = tvy;
}

__global__ void spec_start_kernel(int n, int batch, float* __restrict__ v) {
  const long N = (long)n * batch;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x)
    v[i] = rsqrtf((float)n) * (1.f + 0.25f * (float)((i % n) & 1));   // not orthogonal to any eigenvector
}

__global__ void spec_shift_kernel(int batch, const float* __restrict__ hi, float pad, float* __restrict__ s) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < batch) s[b] = pad * hi[b];
}

cudaError_t tc_spectrum_bounds(const float* A, int n, int batch, int iters, float pad, float* hi, float* lo,
                               float* shift, float* v, float* y, cudaStream_t s) {
  if (batch <= 0) return cudaSuccess;
  const dim3 gg((n + 7) / 8, batch);
  for (int phase = 0; phase < 2; ++phase) {
    spec_start_kernel<<<256, 256, 0, s>>>(n, batch, v);
    if (phase == 1) spec_shift_kernel<<<(batch + 255) / 256, 256, 0, s>>>(batch, hi, pad, shift);
    for (int it = 0; it < iters; ++it) {
      spec_gemv_kernel<<<gg, 256, 0, s>>>(A, n, v, shift, phase, y);
      spec_normalise_kernel<<<batch, 1024, 0, s>>>(n, v, y, phase == 0 ? hi : lo);
    }
  }
  return cudaGetLastError();
}

__global__ void ns_init_kernel(const float* __restrict__ A, int n, const float* __restrict__ ab, float* __restrict__ X,
                               __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                               __nv_bfloat16* __restrict__ lo2, int ldh) {
  const int r = blockIdx.y, b = blockIdx.z;
  const float a = ab[b];
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ldh; c += gridDim.x * blockDim.x) {
    float y = 0.f;
    if (c < n) {
      y = -a * a * A[((long)b * n + r) * n + c] + (r == c ? 2.f * a : 0.f);
      X[((long)b * n + r) * n + c] = y;
    }
    split_store(y, hi, lo, ((long)b * n + r) * ldh + c, lo2);
  }
}

cudaError_t tc_ns_init(const float* A, int n, int batch, const float* ab, float* X, __nv_bfloat16* hi,
                       __nv_bfloat16* lo, cudaStream_t s, __nv_bfloat16* lo2) {
  const int ldh = tc_ld(n);
  dim3 grid((ldh + 255) / 256, n, batch);
  if (batch > 0) ns_init_kernel<<<grid, 256, 0, s>>>(A, n, ab, X, hi, lo, lo2, ldh);
  return cudaGetLastError();
}

// Y_b = (X_b + X_b^T)/2 (FP32, out of place) and its split parts; one thread per element.
__global__ void sym_split_kernel(const float* __restrict__ X, int n, float* __restrict__ Y, __nv_bfloat16* __restrict__ hi,
                                 __nv_bfloat16* __restrict__ lo, __nv_bfloat16* __restrict__ lo2, int ldh) {
  const int r = blockIdx.y, b = blockIdx.z;
  const float* Xb = X + (long)b * n * n;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ldh; c += gridDim.x * blockDim.x) {
    float v = 0.f;
    if (c < n) {
      v = 0.5f * (Xb[(long)r * n + c] + Xb[(long)c * n + r]);
      Y[((long)b * n + r) * n + c] = v;
    }
    split_store(v, hi, lo, ((long)b * n + r) * ldh + c, lo2);
  }
}

cudaError_t tc_sym_split(const float* X, int n, int batch, float* Y, __nv_bfloat16* hi, __nv_bfloat16* lo,
                         __nv_bfloat16* lo2, cudaStream_t s) {
  const int ldh = tc_ld(n);
  dim3 grid((ldh + 255) / 256, n, batch);
  if (batch > 0) sym_split_kernel<<<grid, 256, 0, s>>>(X, n, Y, hi, lo, lo2, ldh);
  return cudaGetLastError();
}

cudaError_t tc_transpose_split(const float* B, int M, int K, __nv_bfloat16* hi, __nv_bfloat16* lo, cudaStream_t s,
                               __nv_bfloat16* lo2, long ldb) {
  const int ld = tc_ld(M);
  dim3 grid((K + 31) / 32, (ld + 31) / 32);
  transpose_split_kernel<<<grid, dim3(32, 8), 0, s>>>(B, M, K, ldb > 0 ? ldb : K, ld, hi, lo, lo2);
  return cudaGetLastError();
}

}  // namespace gw
