// Weighted symmetric rank-K products on the tcgen05 tensor cores with the weight applied inside the kernel:
//
//   out_b = f( B diag(w_b) B^T ),   B = B_ia [n][K] (BF16 hi + lo), w_b = row b of a weight table [nb][ldw] (FP32),
//
// with B in the K-panel layout [P][n][KP] (hi and lo parts): panel p holds columns [p KP, p KP + KP)
// of every row, so that a TMA box of 128 or 256 rows reads one contiguous stretch of memory.  In the plain row
// layout the rows of B_ia at N_ov = 778240 are 1.5-3 MB apart, every row of a box sits in its own page, and the
// address translation of the CTAs' boxes (tens of thousands of pages at every K position) held the kernel to half
// its speed; the panel layout touches a handful of pages per K position.
//
// for every batch entry b, over the lower triangle (computed tiles mirrored into the upper triangle).  This is
//   * Pi(i xi) on the imaginary grid (Sec. 3.3, equation after "wauxbas"): w = -4 D_ia/(D_ia^2 + xi^2);
//   * the dense real-axis Pi(x) of the residue fallback (same section, Pi(z) with +i eta in both pole terms):
//     w = Re c(x) and Im c(x), c = 2[1/(x - D + i eta) + 1/(-x - D + i eta)], as two entries;
//   * the difference-form products Pi(i xi) - Pi(0): w = 4 xi^2/(D (D^2 + xi^2)).
//
// Design (one CTA per SM, persistent over work items = (128 x 256 tile, batch entry), entries fastest so that the
// CTAs running at the same time read the same rows of B):
//   * One thread streams by TMA, per 32-wide k-block, the hi/lo rows of the weighted side (2 x 128 x 32) with the
//     entry's weight row into a 4-stage A ring that the transform releases; another the BF16 hi/lo tiles of the
//     unweighted side (2 x 256 x 32) into a 3-stage B ring that the tensor core releases; the transformed tiles go
//     through a 4-stage T ring, also released by the tensor core.  With one thread for both rings the weighted side
//     could not run ahead of a B stage's release, and the loads alone (transform, drain and two of three products
//     left out) took 7.0 ms of the 10.0 of 38 entries at N_aux 1800, K 26496; they take 5.8 with two.
//   * Two transform groups of four warps take the k-blocks in turn, one thread per row: form b = hi + lo in FP32
//     (exact: 16 significant bits), multiply by the weights and split the products into BF16 hi/lo tiles (64-byte
//     swizzle, the tensor core's K-major layout).  The weight never round-trips through HBM.  A k-block's transform
//     is a chain of waits, conversions and a proxy fence that is longer than its MMAs; two groups overlap two of
//     them (a third group gains nothing and costs a B stage's room).
//   * One thread issues tcgen05.mma M128 N256 K16 (BF16 in, FP32 accumulate in TMEM): hi*hi + hi*lo + lo*hi.
//     The tensor core queues little work ahead of the issuing thread, so an instruction that takes 128 cycles
//     (N = 256) leaves that thread the time for its barrier waits and commits without idling the tensor core;
//     with N = 128 those waits showed up as idle tensor-core time.
//   * Accumulation precision: the tensor core's FP32 accumulator loses up to an ulp per accumulate, so no
//     partial sum runs through more than CHUNK k-blocks (6 CHUNK accumulates) before the drain warps add it,
//     rounded to nearest, into an FP32 running sum.  TMEM columns [256, 512) hold the sum (the first chunk of an
//     item accumulates there directly), [0, 256) the partial of the later chunks.  The tensor core waits while a
//     chunk is drained, so eight warps share it (128 columns each): four took 0.9 of the 10.0 ms, eight 0.4.
//   Together 9.95 to 8.99 ms (38 entries, N_aux 1800, K 26496) and 1.52 to 1.37 (N_aux 1008, K 12160): what remains is
//   shared-memory and L2 traffic (48 KiB in and 32 KiB through the transform per 6 MMAs).
// Every mbarrier wait is bounded; on timeout the kernel records a code in *err, stops every role, waits for its
// copies and tensor-core work in flight, frees TMEM and returns.
#include "pi_tc.cuh"
#include "gw_internal.cuh"
#include "tc_ptx.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

namespace gw {
namespace {
using namespace ptx;

constexpr int BM = 128, BN = 256, BK = 32;
constexpr int TR_GROUPS = 2, TR_GROUP = 4;       // transform: groups of four warps taking the k-blocks in turn
constexpr int A_STAGES = 4, B_STAGES = 3, T_STAGES = 4;
// a stage of the A and T rings always belongs to the same transform group, which then sees every phase of its barriers
// (a wait by parity passes too early for a thread that is two phases behind)
static_assert(A_STAGES % TR_GROUPS == 0 && T_STAGES % TR_GROUPS == 0, "stages of the transform groups");
constexpr int A_BYTES = 2 * BM * BK * 2;        // hi/lo rows of the weighted side: 16 KiB
constexpr int W_BYTES = BK * 4;                 // the entry's weight row [BK] FP32
constexpr int HB_BYTES = BN * BK * 2;           // one BF16 tile of the unweighted side (256 rows x 64 bytes)
constexpr int HA_BYTES = BM * BK * 2;           // one transformed BF16 tile (128 rows x 64 bytes)
constexpr int BS_BYTES = 2 * HB_BYTES;          // B stage: hi, lo (32 KiB)
constexpr int TS_BYTES = 2 * HA_BYTES;          // T stage: hi, lo (16 KiB)
constexpr int A_TX = A_BYTES + W_BYTES;
constexpr int B_TX = BS_BYTES;
// shared memory: A ring, B ring, T ring, weight rows, barriers (every tile 1 KiB aligned)
constexpr int B_OFF = A_STAGES * A_BYTES, T_OFF = B_OFF + B_STAGES * BS_BYTES, W_OFF = T_OFF + T_STAGES * TS_BYTES,
              BAR_OFF = W_OFF + A_STAGES * W_BYTES;
// mbarrier indices: A ring full/empty, B ring full/empty, T ring full/empty, accumulator full/empty, final
constexpr int BAR_AF = 0, BAR_AE = BAR_AF + A_STAGES, BAR_BF = BAR_AE + A_STAGES, BAR_BE = BAR_BF + B_STAGES,
              BAR_TF = BAR_BE + B_STAGES, BAR_TE = BAR_TF + T_STAGES, BAR_ACCF = BAR_TE + T_STAGES,
              BAR_ACCE = BAR_ACCF + 1, BAR_FIN = BAR_ACCE + 1, N_BARS = BAR_FIN + 1;
static_assert(N_BARS * 8 + 4 <= 256, "barrier area");
constexpr int SMEM_BYTES = BAR_OFF + 256 + 1024;
static_assert(SMEM_BYTES + 1024 <= 232448, "shared memory per block (dynamic + static)");
// warps: drain + epilogue (two per TMEM lane quarter, 128 columns each), transform, TMA of the weighted side, MMA, TMA of
// the unweighted side
constexpr int DR_WARPS = 8, TR_WARP0 = DR_WARPS, A_WARP = TR_WARP0 + TR_GROUPS * TR_GROUP, MMA_WARP = A_WARP + 1,
              B_WARP = A_WARP + 2, THREADS = 32 * (A_WARP + 3);
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t COL_P = 0, COL_S = 256;      // TMEM columns of the partial and of the running sum
constexpr uint32_t SBO64 = 8 * 64;              // 8-row groups of 64-byte rows
constexpr uint32_t SWZ64 = 4;                   // descriptor swizzle mode: 64-byte
// kind::f16 instruction descriptor: D = F32, A = B = BF16, both K-major, N = 256, M = 128
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                           ((uint32_t)(BM >> 4) << 24);
constexpr int CHUNK = 16;                       // k-blocks per partial sum
constexpr int KP = 256;                         // panel width of the K-panel layout [P][n][KP]

struct PfMaps {
  CUtensorMap ah, al, bh, bl, w;
};

// Lower tiles, row-major: 128-row block bm holds the 256-column blocks bn2 = 0 .. floor(bm / 2); the first
// C(bm) = sum_{r < bm} (floor(r / 2) + 1) tiles precede row block bm, C(2Q) = Q (Q + 1), C(2Q + 1) = (Q + 1)^2.
__host__ __device__ __forceinline__ long tiles_before(int bm) {
  const long q = bm / 2;
  return (bm & 1) ? (q + 1) * (q + 1) : q * (q + 1);
}

// Work item -> (tile (bm, bn2), entry b, K split ks); items run entry-fastest within a tile, tiles in the order of
// the table `tiles` (bm | bn2 << 16).
__device__ __forceinline__ void decode_item(long item, int nb, int ksplit, const uint32_t* __restrict__ tiles,
                                            int& bm, int& bn2, int& b, int& ks) {
  ks = (int)(item % ksplit);
  item /= ksplit;
  b = (int)(item % nb);
  const uint32_t v = __ldg(tiles + item / nb);
  bm = (int)(v & 0xffffu);
  bn2 = (int)(v >> 16);
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Two FP32 operations in one instruction, each rounded to nearest.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "add.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t"
      "mul.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

// Chunk bookkeeping of an item with nki k-blocks: chunk c = kb / CHUNK accumulates into the running sum (c = 0)
// or into the partial (c >= 1).  The drain warps act at the end of every chunk c >= 1 (sum += partial, or the
// epilogue at the item's last k-block) and at the end of a single-chunk item (epilogue).
__device__ __forceinline__ bool chunk_end(int kb, int nki) { return kb % CHUNK == CHUNK - 1 || kb == nki - 1; }
__device__ __forceinline__ bool drain_event(int kb, int nki) {
  return chunk_end(kb, nki) && (kb >= CHUNK || kb == nki - 1);
}

// With ksplit > 1 the k-blocks of every (tile, entry) are cut into ksplit contiguous ranges, each a work item of
// its own, which writes its raw partial product (lower and mirrored) to part [ksplit][nb][n][n]; pf_reduce_kernel
// then adds the partials in a fixed order (deterministic) and applies the output mode.
__global__ void __launch_bounds__(THREADS, 1)
    pi_fused_kernel(const __grid_constant__ PfMaps maps, const uint32_t* __restrict__ tiles, int n, int K, int nb,
                    int mode_even, int mode_odd,
                    float* __restrict__ out, long out_bstride, int ldo, int ksplit, float* __restrict__ part,
                    long out_limit, long part_limit, int* __restrict__ err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (base - raw);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + BAR_OFF + N_BARS * 8);
  const uint32_t bar0 = base + BAR_OFF;
  // barrier i at bar0 + 8 i (addresses computed, not held in an indexed array)
  auto bar = [bar0](int i) { return bar0 + 8u * (uint32_t)i; };
  __shared__ int s_abort;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nbt = (n + BM - 1) / BM;
  const long n_tiles = tiles_before(nbt);
  const long items = n_tiles * nb * ksplit;
  const int nk = (K + BK - 1) / BK;

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < A_STAGES; ++s) {
      mbar_init(bar(BAR_AF + s), 1);
      mbar_init(bar(BAR_AE + s), TR_GROUP);    // one arrival per transform warp of a group
    }
    for (int s = 0; s < B_STAGES; ++s) {
      mbar_init(bar(BAR_BF + s), 1);              // the producer's expect_tx arrival
      mbar_init(bar(BAR_BE + s), 1);              // the MMA thread's commit
    }
    for (int s = 0; s < T_STAGES; ++s) {
      mbar_init(bar(BAR_TF + s), TR_GROUP);       // one arrival per transform warp of a group
      mbar_init(bar(BAR_TE + s), 1);              // the MMA thread's commit
    }
    mbar_init(bar(BAR_ACCF), 1);
    mbar_init(bar(BAR_ACCE), DR_WARPS);        // one arrival per drain warp
    mbar_init(bar(BAR_FIN), 1);
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

  if (warp == A_WARP) {
    if (lane == 0) {
      // ------------------------------------------------------------ TMA producer, weighted side
      // rows + weight row, released by the transform warps.  Ring positions are stage indices and phase bits.
      long issued = 0;
      uint32_t sa = 0, pa = 0;
      bool wrapped = false, ok = true;
      for (long it = blockIdx.x; it < items && ok; it += gridDim.x) {
        int bm, bn2, b, ks;
        decode_item(it, nb, ksplit, tiles, bm, bn2, b, ks);
        const int kb0 = (int)((long)nk * ks / ksplit), nki = (int)((long)nk * (ks + 1) / ksplit) - kb0;
        for (int kb = 0; kb < nki; ++kb) {
          const int kx = (kb0 + kb) * BK;
          if (wrapped && !mbar_wait(bar(BAR_AE + sa), pa ^ 1u, err, 11)) { ok = false; break; }
          if (*(volatile int*)&s_abort) { ok = false; break; }
          mbar_expect_tx(bar(BAR_AF + sa), A_TX);
          tma_load_3d(base + sa * A_BYTES, &maps.ah, kx % KP, bm * BM, kx / KP, bar(BAR_AF + sa));
          tma_load_3d(base + sa * A_BYTES + HA_BYTES, &maps.al, kx % KP, bm * BM, kx / KP, bar(BAR_AF + sa));
          tma_load_2d(base + W_OFF + sa * W_BYTES, &maps.w, kx, b, bar(BAR_AF + sa));
          ++issued;
          if (++sa == A_STAGES) { sa = 0; pa ^= 1u; wrapped = true; }
        }
      }
      if (!ok) {
        s_abort = 1;
        // wait for the copies that may still be in flight (the latest phase of each stage)
        for (long q = issued > A_STAGES ? issued - A_STAGES : 0; q < issued; ++q)
          mbar_wait(bar(BAR_AF + (int)(q % A_STAGES)), (uint32_t)((q / A_STAGES) & 1), err, 12);
      }
    }
  } else if (warp == B_WARP) {
    if (lane == 0) {
      // ------------------------------------------------------------ TMA producer, unweighted side
      // BF16 hi/lo rows, released by the tensor core.
      long issued = 0;
      uint32_t sb = 0, pb = 0;
      bool wrapped = false, ok = true;
      for (long it = blockIdx.x; it < items && ok; it += gridDim.x) {
        int bm, bn2, b, ks;
        decode_item(it, nb, ksplit, tiles, bm, bn2, b, ks);
        const int kb0 = (int)((long)nk * ks / ksplit), nki = (int)((long)nk * (ks + 1) / ksplit) - kb0;
        for (int kb = 0; kb < nki; ++kb) {
          const int kx = (kb0 + kb) * BK;
          if (wrapped && !mbar_wait(bar(BAR_BE + sb), pb ^ 1u, err, 13)) { ok = false; break; }
          if (*(volatile int*)&s_abort) { ok = false; break; }
          const uint32_t bs = base + B_OFF + sb * BS_BYTES;
          mbar_expect_tx(bar(BAR_BF + sb), B_TX);
          tma_load_3d(bs, &maps.bh, kx % KP, bn2 * BN, kx / KP, bar(BAR_BF + sb));
          tma_load_3d(bs + HB_BYTES, &maps.bl, kx % KP, bn2 * BN, kx / KP, bar(BAR_BF + sb));
          ++issued;
          if (++sb == B_STAGES) { sb = 0; pb ^= 1u; wrapped = true; }
        }
      }
      if (!ok) {
        s_abort = 1;
        for (long q = issued > B_STAGES ? issued - B_STAGES : 0; q < issued; ++q)
          mbar_wait(bar(BAR_BF + (int)(q % B_STAGES)), (uint32_t)((q / B_STAGES) & 1), err, 14);
      }
    }
  } else if (warp == MMA_WARP) {
    if (lane == 0) {
      // ------------------------------------------------------------ MMA issuer
      // Per k-block: two waits (B tiles landed, transformed tiles written), six M128 N256 K16 MMAs, two commits
      // that free the B and T stages.  Before the first MMA of chunk c >= 2 it waits for the drain of chunk c - 1 (which
      // reads the partial), and before an item's first MMA for the previous item's epilogue (which reads both).
      uint32_t sb = 0, pb = 0, st = 0, pt = 0;
      uint32_t n_acc_waits = 0;
      bool first_item = true;
      const uint64_t dB = sdesc(base + B_OFF, SBO64, SWZ64), dT = sdesc(base + T_OFF, SBO64, SWZ64);
      bool ok = true;
      for (long it = blockIdx.x; it < items && ok; it += gridDim.x) {
        int bm, bn2, b, ks;
        decode_item(it, nb, ksplit, tiles, bm, bn2, b, ks);
        const int nki = (int)((long)nk * (ks + 1) / ksplit) - (int)((long)nk * ks / ksplit);
        for (int kb = 0; kb < nki; ++kb) {
          if (!mbar_wait(bar(BAR_BF + sb), pb, err, 21) || !mbar_wait(bar(BAR_TF + st), pt, err, 22)) {
            ok = false;
            break;
          }
          const bool first = kb % CHUNK == 0;
          if (first && (kb >= 2 * CHUNK || (kb == 0 && !first_item))) {
            if (!mbar_wait(bar(BAR_ACCE), n_acc_waits & 1u, err, 23)) { ok = false; break; }
            ++n_acc_waits;
          }
          tc_fence_after();
          const uint32_t d = tmem + (kb < CHUNK ? COL_S : COL_P);
          const uint64_t bh = dB + (uint64_t)((sb * BS_BYTES) >> 4), bl = bh + (uint64_t)(HB_BYTES >> 4);
          const uint64_t ah = dT + (uint64_t)((st * TS_BYTES) >> 4), al = ah + (uint64_t)(HA_BYTES >> 4);
          mma_bf16(d, ah, bh, IDESC, first ? 0u : 1u);
          mma_bf16(d, ah, bl, IDESC, 1u);
          mma_bf16(d, al, bh, IDESC, 1u);
          mma_bf16(d, ah + 2, bh + 2, IDESC, 1u);        // second K16 step: 32 bytes further along each row
          mma_bf16(d, ah + 2, bl + 2, IDESC, 1u);
          mma_bf16(d, al + 2, bh + 2, IDESC, 1u);
          if (drain_event(kb, nki)) mma_commit(bar(BAR_ACCF));
          mma_commit(bar(BAR_BE + sb));
          mma_commit(bar(BAR_TE + st));
          if (++sb == B_STAGES) { sb = 0; pb ^= 1u; }
          if (++st == T_STAGES) { st = 0; pt ^= 1u; }
        }
        first_item = false;
        if (*(volatile int*)&s_abort) ok = false;
      }
      if (!ok) s_abort = 1;
      // every tensor-core operation issued above has completed once the final barrier flips
      mma_commit(bar(BAR_FIN));
      mbar_wait(bar(BAR_FIN), 0, err, 24);
    }
  } else if (warp >= TR_WARP0) {
    // -------------------------------------------------------------- transform: one thread per row of the tile; the
    // groups take the k-blocks in turn, so that one's waits and latencies overlap another's work
    const int r = threadIdx.x & (BM - 1), grp = (warp - TR_WARP0) / TR_GROUP;
    uint32_t sa = grp, pa = 0, st = grp, pt = 0;       // this group's next stages (every TR_GROUPS-th)
    long cnt = grp, total = 0;                         // its next k-block, k-blocks before the current item
    bool ok = true;
    for (long it = blockIdx.x; it < items && ok; it += gridDim.x) {
      const int ks = (int)(it % ksplit);
      const int nki = (int)((long)nk * (ks + 1) / ksplit) - (int)((long)nk * ks / ksplit);
      for (; cnt < total + nki; cnt += TR_GROUPS) {
        bool w_ok = !*(volatile int*)&s_abort && mbar_wait(bar(BAR_AF + sa), pa, err, 31);
        if (w_ok && cnt >= T_STAGES) w_ok = mbar_wait(bar(BAR_TE + st), pt ^ 1u, err, 32);
        if (!__all_sync(0xffffffffu, w_ok)) { ok = false; break; }
        const uint8_t* sp = smem + sa * A_BYTES;
        const float* wrow = reinterpret_cast<const float*>(smem + W_OFF + sa * W_BYTES);
        uint8_t* tp = smem + T_OFF + st * TS_BYTES;
#pragma unroll
        for (int j = 0; j < BK / 8; ++j) {   // 64-byte swizzle: 16-byte chunk j of row r sits at j ^ ((r >> 1) & 3)
          const int off = r * 64 + ((j ^ ((r >> 1) & 3)) << 4);
          const uint4 vh = *reinterpret_cast<const uint4*>(sp + off);
          const uint4 vl = *reinterpret_cast<const uint4*>(sp + HA_BYTES + off);
          const float4 w0 = *reinterpret_cast<const float4*>(wrow + 8 * j);              // broadcast reads
          const float4 w1 = *reinterpret_cast<const float4*>(wrow + 8 * j + 4);
          const uint32_t hw4[4] = {vh.x, vh.y, vh.z, vh.w}, lw4[4] = {vl.x, vl.y, vl.z, vl.w};
          const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
          uint32_t hi[4], lo[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162*>(&hw4[e]);
            const __nv_bfloat162 y = *reinterpret_cast<const __nv_bfloat162*>(&lw4[e]);
            float2 v = make_float2(__low2float(x), __high2float(x));
            v = mul2(add2(v, make_float2(__low2float(y), __high2float(y))), make_float2(wv[2 * e], wv[2 * e + 1]));
            hi[e] = pack_bf16(v.x, v.y);
            const __nv_bfloat162 hh = *reinterpret_cast<const __nv_bfloat162*>(&hi[e]);
            v = add2(v, make_float2(-__low2float(hh), -__high2float(hh)));
            lo[e] = pack_bf16(v.x, v.y);
          }
          *reinterpret_cast<uint4*>(tp + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          *reinterpret_cast<uint4*>(tp + HA_BYTES + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(bar(BAR_TF + st));
          mbar_arrive(bar(BAR_AE + sa));
        }
        if ((sa += TR_GROUPS) >= A_STAGES) { sa -= A_STAGES; pa ^= 1u; }
        if ((st += TR_GROUPS) >= T_STAGES) { st -= T_STAGES; pt ^= 1u; }
      }
      total += nki;
    }
    if (!ok) s_abort = 1;
  } else {
    // -------------------------------------------------------------- drain + epilogue (TMEM lane quarter = warp mod 4)
    const int q = warp & 3, g0 = (warp >> 2) * (BN / 64);
    uint32_t n_events = 0;
    bool ok = true;
    for (long it = blockIdx.x; it < items && ok; it += gridDim.x) {
      int bm, bn2, b, ks;
      decode_item(it, nb, ksplit, tiles, bm, bn2, b, ks);
      const int nki = (int)((long)nk * (ks + 1) / ksplit) - (int)((long)nk * ks / ksplit);
      const int m0 = bm * BM, n0 = bn2 * BN;
      const int row = m0 + q * 32 + lane;
      // split K: the raw partial goes to its slot of `part` (mode 0, row length n); the reduction applies the mode
      const bool raw = ksplit > 1;
      const int mode = raw ? 0 : ((b & 1) ? mode_odd : mode_even);
      const long ob0 = raw ? ((long)ks * nb + b) * n * n : (long)b * out_bstride;
      float* ob = (raw ? part : out) + ob0;
      const int ld = raw ? n : ldo;
      const long lim = (raw ? part_limit : out_limit) - ob0;   // elements writable from ob
      // drain events: the ends of chunks 1, 2, ... and the item's last k-block
      for (int kb = nki > CHUNK ? 2 * CHUNK - 1 : nki - 1;; kb += CHUNK) {
        if (kb > nki - 1) kb = nki - 1;
        const bool final = kb == nki - 1, with_p = kb >= CHUNK;
        const bool w_ok = !*(volatile int*)&s_abort && mbar_wait(bar(BAR_ACCF), n_events & 1u, err, 41);
        if (!__all_sync(0xffffffffu, w_ok)) { ok = false; break; }
        tc_fence_after();
        const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
        for (int g = g0; g < g0 + BN / 64; ++g) {
          uint32_t v[32], w[32];
          tmem_ld32(lane_addr + COL_S + (uint32_t)(g * 32), v);
          if (with_p) tmem_ld32(lane_addr + COL_P + (uint32_t)(g * 32), w);
          tmem_wait_ld();
          if (with_p) {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(w[j]));
          }
          if (!final) {
            tmem_st32(lane_addr + COL_S + (uint32_t)(g * 32), v);
            continue;
          }
          // epilogue: lower element (row, col <= row) in place, mirrored element (col, row) for col < row
          const int c0 = n0 + g * 32;
          if (row < n) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const int col = c0 + j;
              if (col > row || col >= n) continue;
              const float x = __uint_as_float(v[j]);
              const long o = (long)row * ld + col;
              if (o >= lim) { atomicCAS(err, 0, 51); continue; }    // outside the caller's buffer: record, skip
              ob[o] = mode == 0 ? x : (mode == 1 ? ((col == row ? 1.f : 0.f) - x) : -x);
            }
          }
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const int col = c0 + j;
            if (row < n && col < row && col < n) {
              const float x = __uint_as_float(v[j]);
              const long o = (long)col * ld + row;
              if (o >= lim) { atomicCAS(err, 0, 52); continue; }
              ob[o] = mode == 0 ? x : -x;
            }
          }
        }
        if (!final) tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(BAR_ACCE));
        ++n_events;
        if (final) break;
      }
    }
    if (!ok) s_abort = 1;
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// out_b[i][j] = mode(sum_s part[s][b][i][j]) in the fixed order s = 0, 1, ... (split-K reduction).
__global__ void pf_reduce_kernel(const float* __restrict__ part, int ksplit, int nb, int n, int mode_even,
                                 int mode_odd, float* __restrict__ out, long out_bstride, int ldo, long out_limit,
                                 long part_limit, int* __restrict__ err) {
  const long nn = (long)n * n, N = nn * nb;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < N; idx += (long)gridDim.x * blockDim.x) {
    const int b = (int)(idx / nn);
    const long e = idx - (long)b * nn;
    const int i = (int)(e / n), j = (int)(e - (long)i * n);
    if (((long)(ksplit - 1) * nb + b) * nn + e >= part_limit) { atomicCAS(err, 0, 53); continue; }
    float v = 0.f;
    for (int s = 0; s < ksplit; ++s) v += part[((long)s * nb + b) * nn + e];
    const int mode = (b & 1) ? mode_odd : mode_even;
    const long o = (long)b * out_bstride + (long)i * ldo + j;
    if (o >= out_limit) { atomicCAS(err, 0, 54); continue; }
    out[o] = mode == 0 ? v : (mode == 1 ? ((i == j ? 1.f : 0.f) - v) : -v);
  }
}

// w[b][k] for k < K, in FP64 rounded to FP32 (one evaluation per entry and pair).  Kinds: 0 Pi(i xi):
// -4D/(D^2 + xi^2); 1 Re c(x); 2 Im c(x) (broadening eta); 3 unit weight; 4 Pi(i xi) - Pi(0): 4 xi^2/(D (D^2+xi^2)).
__device__ __forceinline__ double pair_weight(int kind, double D, double p, double eta) {
  if (kind == 0) return -4.0 * D / (D * D + p * p);
  if (kind == 3) return 1.0;
  if (kind == 4) return 4.0 * p * p / (D * (D * D + p * p));
  const double a1 = p - D, a2 = -p - D, e2 = eta * eta;
  const double d1 = a1 * a1 + e2, d2 = a2 * a2 + e2;
  if (kind == 1) return 2.0 * (a1 / d1 + a2 / d2);
  return -2.0 * eta * (1.0 / d1 + 1.0 / d2);
}

__global__ void pf_weight_kernel(const double* __restrict__ Dk, int K, const int* __restrict__ kinds,
                                 const double* __restrict__ params, double eta, float* __restrict__ w, int ldw) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x, b = blockIdx.y;
  if (k >= ldw) return;
  w[(long)b * ldw + k] = k < K ? (float)pair_weight(kinds[b], Dk[k], params[b], eta) : 0.f;
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

bool map2d(CUtensorMap* map, CUtensorMapDataType dt, int esize, const void* ptr, int cols, int rows, long ld,
           int box_cols, int box_rows, CUtensorMapSwizzle swz) {
  PFN_encodeTiled enc = encoder();
  if (!enc || (reinterpret_cast<uintptr_t>(ptr) & 15) || ((ld * esize) & 15)) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * esize)};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  return enc(map, dt, 2, const_cast<void*>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3D map of a K-panel array [P][n][KP] with boxes of BK columns x box_rows rows of one panel.
bool map_panel(CUtensorMap* map, CUtensorMapDataType dt, int esize, const void* ptr, int n, int P, int box_rows,
               CUtensorMapSwizzle swz) {
  PFN_encodeTiled enc = encoder();
  if (!enc || (reinterpret_cast<uintptr_t>(ptr) & 15)) return false;
  cuuint64_t dims[3] = {(cuuint64_t)KP, (cuuint64_t)n, (cuuint64_t)P};
  cuuint64_t strides[2] = {(cuuint64_t)KP * esize, (cuuint64_t)KP * esize * n};
  cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return enc(map, dt, 3, const_cast<void*>(ptr), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Row layout -> K-panel layout of the BF16 hi/lo split: hp/lp[p][r][c] from B[r][p KP + c] (zero beyond K).
__global__ void panel_split_kernel(const float* __restrict__ B, long ldb, int n, int K, int P,
                                   __nv_bfloat16* __restrict__ hp, __nv_bfloat16* __restrict__ lp) {
  const long r = blockIdx.y;
  if (r >= n) return;
  for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < (long)P * KP; k += (long)gridDim.x * blockDim.x) {
    const float v = k < K ? B[r * ldb + k] : 0.f;
    const long o = ((k / KP) * n + r) * KP + (k % KP);
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    hp[o] = h;
    lp[o] = __float2bfloat16_rn(v - __bfloat162float(h));
  }
}

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess)
      n = 148;
  }
  return n;
}

}  // namespace

int pf_ldw(int K) { return (K + 3) / 4 * 4; }

long tc_pi_panel_cols(int K) { return (long)(K + KP - 1) / KP * KP; }

cudaError_t tc_pi_panel_split(const float* B, long ldb, int n, int K, __nv_bfloat16* hp, __nv_bfloat16* lp,
                              cudaStream_t s) {
  if (n <= 0 || K <= 0) return cudaSuccess;
  if (n > 65535) return cudaErrorInvalidValue;
  const int P = (K + KP - 1) / KP;
  panel_split_kernel<<<dim3(64, n), 256, 0, s>>>(B, ldb, n, K, P, hp, lp);
  return cudaGetLastError();
}

long tc_pi_fused_items(int n, int nb) { return tiles_before((n + BM - 1) / BM) * nb; }

// Column panels of PANEL 256-column blocks, each swept over the 128-row blocks: the tiles that run at the same time
// then read a few row blocks of the weighted side and PANEL column blocks of the unweighted side, a working set
// per k-block small enough for L2 to serve every CTA from one HBM read (row-major order would sweep all of B).
void tc_pi_fused_tile_order(int n, std::vector<uint32_t>& tiles) {
  constexpr int PANEL = 4;
  const int nbt = (n + BM - 1) / BM, nbn = (nbt + 1) / 2;
  tiles.clear();
  tiles.reserve((size_t)tiles_before(nbt));
  for (int c0 = 0; c0 < nbn; c0 += PANEL)
    for (int bm = 2 * c0; bm < nbt; ++bm)
      for (int bn2 = c0; bn2 < c0 + PANEL && bn2 <= bm / 2; ++bn2) tiles.push_back((uint32_t)bm | ((uint32_t)bn2 << 16));
}

cudaError_t tc_pair_weights(const double* Dk, int K, const int* kinds, const double* params, double eta, int nb,
                            float* w, cudaStream_t s) {
  const int ldw = pf_ldw(K);
  if (nb <= 0) return cudaSuccess;
  pf_weight_kernel<<<dim3((ldw + 255) / 256, nb), 256, 0, s>>>(Dk, K, kinds, params, eta, w, ldw);
  return cudaGetLastError();
}

namespace {

cudaError_t pf_launch(const PfMaps& maps, const uint32_t* tiles, int n, int K, int nb, int mode_even, int mode_odd, float* out,
                      long out_bstride, int ldo, int ksplit, float* part, size_t part_bytes, int* err, cudaStream_t s,
                      int max_ctas) {
  const long items = tiles_before((n + BM - 1) / BM) * nb * ksplit;
  int grid = sm_count();
  if (max_ctas > 0 && max_ctas < grid) grid = max_ctas;
  if (items < grid) grid = (int)items;
  // elements the kernels may write: the nb output matrices, and the capacity of the partials buffer
  const long out_limit = (long)(nb - 1) * out_bstride + (long)n * ldo;
  const long part_limit = part ? (long)(part_bytes / sizeof(float)) : 0;
  if (ksplit > 1 && (long)ksplit * nb * n * n > part_limit) return cudaErrorInvalidValue;
  pi_fused_kernel<<<grid, THREADS, SMEM_BYTES, s>>>(maps, tiles, n, K, nb, mode_even, mode_odd, out, out_bstride, ldo,
                                                     ksplit, part, out_limit, part_limit, err);
  if (ksplit > 1) {
    const long N = (long)n * n * nb;
    pf_reduce_kernel<<<(int)std::min<long>((N + 255) / 256, 4096), 256, 0, s>>>(
        part, ksplit, nb, n, mode_even, mode_odd, out, out_bstride, ldo, out_limit, part_limit, err);
  }
  return cudaGetLastError();
}

// Split-K choices measured per problem shape (n, K, nb, grid cap) and largest split the caller's partials buffer
// allows (a choice made with a larger buffer is never reused with a smaller one), kept for the process.
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int, int, int>, int> g_tune;

}  // namespace

int tc_pi_fused_ksplit(int n, int K, int nb, int max_ctas, int max_split) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto it = g_tune.find(std::make_tuple(n, K, nb, max_ctas, max_split));
  return it == g_tune.end() ? 0 : it->second;
}

cudaError_t tc_pi_fused(int n, int K, const float* w, int nb, const uint32_t* tiles,
                        const __nv_bfloat16* Bhi,
                        const __nv_bfloat16* Blo, int mode_even, int mode_odd, float* out, long out_bstride, int ldo,
                        int* err, cudaStream_t s, int max_ctas, int ksplit, float* part, size_t part_bytes,
                        int* chosen) {
  if (nb <= 0 || n <= 0 || K <= 0) return cudaSuccess;
  if (!tiles || n > 65535 * BM) return cudaErrorInvalidValue;
  PfMaps maps;
  const int ldw = pf_ldw(K);
  const int P = (K + KP - 1) / KP;
  if (!map_panel(&maps.ah, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Bhi, n, P, BM, CU_TENSOR_MAP_SWIZZLE_64B) ||
      !map_panel(&maps.al, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Blo, n, P, BM, CU_TENSOR_MAP_SWIZZLE_64B) ||
      !map_panel(&maps.bh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Bhi, n, P, BN, CU_TENSOR_MAP_SWIZZLE_64B) ||
      !map_panel(&maps.bl, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Blo, n, P, BN, CU_TENSOR_MAP_SWIZZLE_64B) ||
      !map2d(&maps.w, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, w, K, nb, ldw, BK, 1, CU_TENSOR_MAP_SWIZZLE_NONE))
    return cudaErrorInvalidValue;
  static PerDevice attr;
  const cudaError_t ae = attr.run(
      [] { return cudaFuncSetAttribute(pi_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES); });
  if (ae != cudaSuccess) return ae;
  const int nk = (K + BK - 1) / BK;
  const size_t per_split = (size_t)nb * n * n * sizeof(float);
  auto feasible = [&](int ks) {
    return ks == 1 || (part && (size_t)ks * per_split <= part_bytes && nk / ks >= 4);
  };
  if (ksplit > 0) {                        // forced: the largest feasible split not above the request
    while (ksplit > 1 && !feasible(ksplit)) ksplit /= 2;
    if (chosen) *chosen = ksplit;
    return pf_launch(maps, tiles, n, K, nb, mode_even, mode_odd, out, out_bstride, ldo, ksplit, part, part_bytes, err, s,
                     max_ctas);
  }
  // Autotuning over the K split: the persistent grid only fills the GPU when (tiles x entries) reaches the SM
  // count, so small problems (few tiles) split K; each feasible split is timed once per shape (the result of
  // every trial is the same product) and the fastest is kept.
  const long items1 = tiles_before((n + BM - 1) / BM) * nb;
  std::vector<int> cand{1};
  for (int ks : {2, 4, 8})
    if (items1 * (ks / 2) < 2L * sm_count() && feasible(ks)) cand.push_back(ks);
  const int max_split = cand.back();
  int best = tc_pi_fused_ksplit(n, K, nb, max_ctas, max_split);
  if (best == 0) {
    if (cand.size() == 1) {
      best = 1;
    } else {
      cudaEvent_t e0, e1;
      if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) return cudaErrorUnknown;
      float best_ms = 1e30f;
      for (int ks : cand) {
        float ms = 0.f;
        for (int rep = 0; rep < 2; ++rep) {          // the first launch of a configuration warms it up
          cudaEventRecord(e0, s);
          cudaError_t e = pf_launch(maps, tiles, n, K, nb, mode_even, mode_odd, out, out_bstride, ldo, ks, part, part_bytes,
                                    err, s, max_ctas);
          cudaEventRecord(e1, s);
          if (e != cudaSuccess) { cudaEventDestroy(e0); cudaEventDestroy(e1); return e; }
          if (cudaEventSynchronize(e1) != cudaSuccess) { cudaEventDestroy(e0); cudaEventDestroy(e1); return cudaErrorUnknown; }
          cudaEventElapsedTime(&ms, e0, e1);
        }
        if (ms < best_ms) { best_ms = ms; best = ks; }
      }
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
    }
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune[std::make_tuple(n, K, nb, max_ctas, max_split)] = best;
  }
  if (chosen) *chosen = best;
  return pf_launch(maps, tiles, n, K, nb, mode_even, mode_odd, out, out_bstride, ldo, best, part, part_bytes, err, s,
                   max_ctas);
}

}  // namespace gw
