// C ABI of libgw (include/gw.h): plan lifetime, device memory, and the host-side orchestration of
// Algorithm 1 (imaginary-axis screening, then the per-state QP loop with batched residue solves).
#include "gw.h"
#include "gw_internal.cuh"
#include "oz_gemm.cuh"
#include "pi_tc.cuh"

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

using gw::MinresState;
using gw::QPState;

namespace {

thread_local std::string g_create_error;

struct DevBuf {
  void* p = nullptr;
  size_t bytes = 0;
  bool grown = false;        // it has been allocated before
};

}  // namespace

struct gw_plan {
  gw_config cfg{};
  int n_bas = 0, n_ov = 0, n_t = 0, n_g = 0;
  unsigned flags = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  std::vector<double> h_eps, h_xi, h_wt, h_shift, h_sx, h_en;
  // open shell: n_spin = 2, per-spin KS energies and occupations, each target's spin; closed shell: n_spin = 1
  int n_spin = 1;
  int occ_s[2] = {0, 0};
  std::vector<double> h_eps_s[2];
  std::vector<int> h_spin;
  int* d_spin = nullptr;        // [n_targets] (open shell only)
  int* d_occ_t = nullptr;       // [n_targets] occupied states of each target's spin (open shell only)
  std::vector<double> h_eps_g[2];   // poles of G per spin (the KS energies, or the updated ones inside gw_evgw)
  double* d_eps_g = nullptr;        // [n_spin][n_bas]
  std::vector<int> h_targets;
  double* d_eps = nullptr;     // energies of W: the pair energies D_ia of Pi
  double* d_B_ia = nullptr;
  double* d_B_nm = nullptr;
  bool own_B = true;
  double* d_xi = nullptr;     // [n_g + 1], last entry 0 (static point)
  double* d_wt = nullptr;     // [n_g]
  double* d_sx = nullptr;
  double* d_shift = nullptr;
  double* d_en = nullptr;
  double* d_W = nullptr;      // [n_t][n_bas][n_g + 1]
  float* d_B_ia_f = nullptr;  // mixed: FP32 copy of B_ia, rows of ld_f elements (16-byte rows for TMA)
  long ld_f = 0;
  float* d_B_nm_f = nullptr;  // mixed: FP32 copy of B_nm
  __nv_bfloat16* d_Bhi = nullptr;   // mixed: BF16 hi/lo split of B_ia, [n_aux][tc_ld(n_ov)]
  __nv_bfloat16* d_Blo = nullptr;
  __nv_bfloat16* d_BThi = nullptr;  // mixed: BF16 hi/lo split of B_ia^T, [n_ov][tc_ld(n_aux)]
  __nv_bfloat16* d_BTlo = nullptr;
  __nv_bfloat16* d_Blo2 = nullptr;  // mixed: third split parts of B_ia and B_ia^T (refinement operator)
  __nv_bfloat16* d_Bp_hi = nullptr; // mixed: BF16 hi/lo split of B_ia in the K-panel layout of the Pi kernel,
                                    // [P][n_aux][256]
  __nv_bfloat16* d_Bp_lo = nullptr;
  __nv_bfloat16* d_BTlo2 = nullptr;
  double* d_D = nullptr;            // pair energies D_ia [n_ov]
  double* d_Dsort = nullptr;        // mixed: D_ia ascending, with the pair index of each entry in d_Dkidx
  int* d_Dkidx = nullptr;
  double D_min = 0.0;               // smallest pair energy
  __nv_bfloat16* d_Bnhi = nullptr;  // mixed: BF16 hi/lo split of the B_nm rows, [n_t*n_bas][tc_ld(n_aux)]
  __nv_bfloat16* d_Bnlo = nullptr;
  __nv_bfloat16* d_Bnlo2 = nullptr;
  bool screening_done = false;
  std::vector<char*> slabs;         // kSlab bytes each, the last one used up to slab_used (plan_alloc)
  size_t slab_used = 0;
  // spectral-decomposition route (gw_sigma_sd): Casida matrix and eigenvectors, pole weights; valid while sd_done
  DevBuf sd_M, sd_T, sd_cs, sd_off, sd_Om, sd_V, sd_w2, sd_tmap, sd_om, sd_S, sd_dS, sd_part, sd_x[5], sd_vec;
  bool sd_done = false;
  int sd_sweeps = 0;
  // sharding across ranks (gw_set_shard): frequency positions [sh_p0, sh_p1) of the imaginary-axis stage and the
  // residue right-hand sides j with j % sh_world == sh_rank; sums across ranks through sh_reduce
  int sh_rank = 0, sh_world = 1;
  gw_allreduce_fn sh_reduce = nullptr;
  void* sh_ctx = nullptr;
  std::vector<double> sh_buf;
  int ns_iters_last = 0;
  int ns_kmax = 0;
  int ns_ndiff = 0;           // positions 1 .. ns_ndiff of the imaginary-axis stage are difference columns
  gw::FreqNodes nodes;        // mixed: grid points the stage is computed at, for the smallest pair energy nodes_D
  double nodes_D = -1.0;
  bool nodes_ok = false;
  DevBuf sk_C;                // device copy of nodes.C
  std::vector<DevBuf*> bufs;
  int tc_tiles_n = 0;          // N_aux the tile-order table of the Pi kernel was built for
  DevBuf oz_A, oz_B, oz_X, oz_sc, oz_w, oz_part, op_BT, op_sc, op_V;
    // FP64 products on the tensor cores: digits, inverse factors, scales, weights
  DevBuf ws_mat, ws_info, ws_gout, ws_xi, tc_part, tc_kind, tc_par, tc_err, tc_w, tc_tiles, ns_E, ns_X, ns_X2, ns_Xa, ns_Xb, ns_T, ns_lam,
      ns_E0, ns_vec;
  DevBuf mr_V, mr_U, mr_S, mr_vprev, mr_v, mr_d1, mr_d2, mr_x, mr_st, mr_rt, mr_rm, mr_xf, mr_wre, mr_wim,
      mr_dwre, mr_it, mr_res, mr_cnt, mr_Vhi, mr_Vlo, mr_Uhi, mr_Ulo, mr_Vlo2, mr_Ulo2, mr_V64, mr_part;
  DevBuf sg_I, sg_dI, sg_R, sg_dR, sg_om, sg_start, sg_coef, sg_act, sg_tmap, qp_st, qp_om0;
  DevBuf fb_A, fb_y, fb_piv, fb_info, fb_idx, fb_y64, fb_V32, fb_S32, fb_Vp, fb_Up, fb_x, fb_V64, fb_U64, fb_S64, fb_sel,
      fb_pos, fb_rho, fb_xs, fb_Bl, fb_part, fb_lu, fb_sw, fb_linv, fb_lus;
  std::string err;
  gw_stats stats{};
  cudaEvent_t ev0 = nullptr, ev1 = nullptr, ev2 = nullptr;
  // per-kernel-class timing: events recorded around launches, resolved after each call's final sync
  std::vector<cudaEvent_t> tpool;
  size_t tused = 0;
  struct Mark { int cls; size_t a, b; double flops; };
  std::vector<Mark> marks;

  gw_plan() {
    DevBuf* all[] = {&oz_A, &oz_B, &oz_X, &oz_sc, &oz_w, &oz_part, &op_BT, &op_sc, &op_V, &ws_mat, &ws_info, &ws_gout, &ws_xi, &tc_part, &tc_kind, &tc_par, &tc_err, &tc_w, &tc_tiles, &ns_E, &ns_X, &ns_X2, &ns_Xa, &ns_Xb, &ns_T, &ns_lam, &ns_E0, &ns_vec, &sk_C, &mr_V, &mr_U, &mr_S, &mr_vprev,
                     &mr_v, &mr_d1, &mr_d2, &mr_x, &mr_st, &mr_rt, &mr_rm, &mr_xf, &mr_wre, &mr_wim,
                     &mr_dwre, &mr_it, &mr_res, &mr_cnt, &mr_Vhi, &mr_Vlo, &mr_Uhi, &mr_Ulo, &mr_Vlo2, &mr_Ulo2, &mr_V64, &mr_part, &sg_I, &sg_dI, &sg_R, &sg_dR, &sg_om, &sg_start,
                     &sg_coef, &sg_act, &sg_tmap, &qp_st, &qp_om0, &fb_A, &fb_y, &fb_piv, &fb_info, &fb_idx, &fb_y64, &fb_V32, &fb_S32, &fb_Vp, &fb_Up, &fb_x, &fb_V64, &fb_U64, &fb_S64, &fb_sel, &fb_pos, &fb_rho, &fb_xs, &fb_Bl, &fb_part, &fb_lu, &fb_sw, &fb_linv, &fb_lus, &sd_M, &sd_T, &sd_cs, &sd_off, &sd_Om, &sd_V, &sd_w2, &sd_tmap, &sd_om, &sd_S, &sd_dS, &sd_part, &sd_x[0], &sd_x[1], &sd_x[2], &sd_x[3], &sd_x[4], &sd_vec};
    bufs.assign(all, all + sizeof(all) / sizeof(all[0]));
    static_assert(sizeof(all) / sizeof(all[0]) + 32 <= 160, "kPlanBufs: these and the plan's other arrays");
  }
};

namespace {

gw_status fail(gw_plan* p, gw_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  if (p) p->err = buf; else g_create_error = buf;
  return st;
}

#define CK(call)                                                                                   \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess) {                                                                       \
      if (e_ == cudaErrorMemoryAllocation) { cudaGetLastError(); return fail(P, GW_ERR_OOM, "%s: %s", #call, cudaGetErrorString(e_)); } \
      return fail(P, GW_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_));                        \
    }                                                                                              \
  } while (0)

#define LAUNCH(expr)                                                                               \
  do {                                                                                             \
    expr;                                                                                          \
    P->stats.n_kernel_launches++;                                                                  \
    cudaError_t e_ = cudaGetLastError();                                                           \
    if (e_ != cudaSuccess) return fail(P, GW_ERR_CUDA, "launch %s: %s", #expr, cudaGetErrorString(e_)); \
  } while (0)

#define TRY(call)                                                                                  \
  do {                                                                                             \
    gw_status s_ = (call);                                                                         \
    if (s_ != GW_OK) return s_;                                                                    \
  } while (0)

void count_bytes(gw_plan* P, long long delta) {
  P->stats.bytes_device += delta;
  P->stats.bytes_device_peak = std::max(P->stats.bytes_device_peak, P->stats.bytes_device);
}

// Device allocations of a plan, counted in gw_stats.bytes_device: a buffer's first allocation, up to kSmallBuf, comes out
// of slabs that the plan holds until it is destroyed; larger ones and a buffer that has outgrown its share are the
// driver's.  A cudaMalloc with its cudaFree takes 40 to 130 us and a small job has some 60 buffers: a (H2O)_1 job takes
// 3.70 ms with one each, 3.48 with 4 MiB slabs, 3.25 with these; a (H2O)_5 one 15.2, 14.8 and 14.1.
// A slab is left when a buffer of at most kSmallBuf does not fit, so at least 3/4 of it are first allocations, one per
// buffer: slab_bound follows.
constexpr size_t kSlab = 32u << 20, kSmallBuf = 8u << 20;
constexpr size_t kPlanBufs = 160;              // buffers a plan has, work space and others

// Bytes of slabs that a plan may hold beside its other buffers, all of them `bytes` at their final sizes.
unsigned long long slab_bound(unsigned long long bytes) {
  const unsigned long long first = std::min<unsigned long long>(bytes, kPlanBufs * kSmallBuf) + 512 * kPlanBufs;
  return first / 3 * 4 + kSlab;
}

gw_status plan_alloc(gw_plan* P, void** p, size_t bytes, bool first = true) {
  if (bytes > kSmallBuf || !first) {
    CK(cudaMalloc(p, bytes));
    count_bytes(P, (long long)bytes);
    return GW_OK;
  }
  const size_t need = (bytes + 511) & ~(size_t)511;
  if (P->slabs.empty() || P->slab_used + need > kSlab) {
    void* q = nullptr;
    CK(cudaMalloc(&q, kSlab));
    P->slabs.push_back(static_cast<char*>(q));
    count_bytes(P, (long long)kSlab);
    P->slab_used = 0;
  }
  *p = P->slabs.back() + P->slab_used;
  P->slab_used += need;
  return GW_OK;
}

bool in_slab(const gw_plan* P, const void* p) {
  for (const char* q : P->slabs)
    if (p >= q && p < q + kSlab) return true;
  return false;
}

// Gives back a buffer of plan_alloc (bytes as asked for; a slab keeps its share until the plan ends).
void plan_free(gw_plan* P, void* p, size_t bytes) {
  if (!p || in_slab(P, p)) return;
  cudaFree(p);
  count_bytes(P, -(long long)bytes);
}

template <typename T>
gw_status dmalloc(gw_plan* P, T** p, size_t bytes) {
  return plan_alloc(P, reinterpret_cast<void**>(p), bytes);
}

gw_status ensure(gw_plan* P, DevBuf& b, size_t bytes) {
  if (b.bytes >= bytes && b.p) return GW_OK;
  const bool first = !b.p && !b.grown;
  if (b.p) {
    CK(cudaStreamSynchronize(P->stream));
    plan_free(P, b.p, b.bytes);
    b.p = nullptr;
    b.bytes = 0;
    b.grown = true;
  }
  if (bytes == 0) bytes = 16;
  TRY(plan_alloc(P, &b.p, bytes, first));
  b.bytes = bytes;
  return GW_OK;
}

// Gives a buffer's memory back to the driver (one in a slab keeps it); the stream must have finished with it.
void release(gw_plan* P, DevBuf& b) {
  if (!b.p || in_slab(P, b.p)) return;
  plan_free(P, b.p, b.bytes);
  b.p = nullptr;
  b.bytes = 0;
}

template <typename T>
T* as(DevBuf& b) { return reinterpret_cast<T*>(b.p); }

size_t ws_bytes(const gw_plan* P) {
  return (size_t)(P->cfg.workspace_mb > 0 ? P->cfg.workspace_mb : 8192) << 20;
}

size_t tick(gw_plan* P) {
  if (P->tused == P->tpool.size()) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return (size_t)-1;
    P->tpool.push_back(e);
  }
  cudaEventRecord(P->tpool[P->tused], P->stream);
  return P->tused++;
}

void mark(gw_plan* P, int cls, size_t a, double flops) {
  size_t b = tick(P);
  if (a != (size_t)-1 && b != (size_t)-1) P->marks.push_back({cls, a, b, flops});
  P->stats.launches_kernel[cls]++;
}

// Accumulate the recorded intervals (the stream must be synchronised).
void resolve_marks(gw_plan* P) {
  for (const auto& m : P->marks) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, P->tpool[m.a], P->tpool[m.b]) == cudaSuccess) {
      P->stats.ms_kernel[m.cls] += ms;
      P->stats.flops_kernel[m.cls] += m.flops;
    }
  }
  P->marks.clear();
  P->tused = 0;
  cudaGetLastError();
}

double now_ms(gw_plan* P, cudaEvent_t a, cudaEvent_t b) {
  float ms = 0.f;
  cudaEventElapsedTime(&ms, a, b);
  return (double)ms;
}

// Tensor-core weighted SYRK for `nb` batch entries: out_b = f(B diag(w_b) B^T) with (kind, param) per entry,
// the weights applied inside the kernel (tc_pi_fused).  reset_err = false keeps a bounded-wait code that earlier
// launches of the caller left in tc_err, so that the check at the end reports it.
gw_status tc_weighted_syrk(gw_plan* P, const int* kinds, const double* params, int nb, int mode_even, int mode_odd,
                           float* out, int cls, bool reset_err = true) {
  const int n = P->cfg.n_aux, K = P->n_ov;
  TRY(ensure(P, P->tc_kind, sizeof(int) * nb));
  TRY(ensure(P, P->tc_par, sizeof(double) * nb));
  TRY(ensure(P, P->tc_err, sizeof(int)));
  TRY(ensure(P, P->tc_w, sizeof(float) * (size_t)nb * gw::pf_ldw(K)));
  if (P->tc_tiles_n != n) {                  // tile order of the Pi kernel, uploaded once per plan
    std::vector<uint32_t> order;
    gw::tc_pi_fused_tile_order(n, order);
    TRY(ensure(P, P->tc_tiles, sizeof(uint32_t) * order.size()));
    CK(cudaMemcpy(P->tc_tiles.p, order.data(), sizeof(uint32_t) * order.size(), cudaMemcpyHostToDevice));
    P->tc_tiles_n = n;
  }
  CK(cudaMemcpyAsync(P->tc_kind.p, kinds, sizeof(int) * nb, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->tc_par.p, params, sizeof(double) * nb, cudaMemcpyHostToDevice, P->stream));
  if (reset_err) CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
  const size_t t0 = tick(P);
  CK(gw::tc_pair_weights(P->d_D, K, as<int>(P->tc_kind), as<double>(P->tc_par),
                         P->cfg.eta, nb, as<float>(P->tc_w), P->stream));
  // split-K partials (only small problems, whose tiles x entry pairs do not fill the GPU, consider a split)
  float* part = nullptr;
  size_t part_bytes = 0;
  if (P->cfg.pi_ksplit != 1 && gw::tc_pi_fused_items(n, nb) < 2L * 152) {
    part_bytes = std::min(ws_bytes(P), (size_t)(P->cfg.pi_ksplit > 0 ? P->cfg.pi_ksplit : 8) * nb * n * n * 4);
    TRY(ensure(P, P->tc_part, part_bytes));
    part = as<float>(P->tc_part);
  }
  int chosen = 1;
  CK(gw::tc_pi_fused(n, K, as<float>(P->tc_w), nb, as<uint32_t>(P->tc_tiles), P->d_Bp_hi, P->d_Bp_lo, mode_even, mode_odd,
                     out, (long)n * n, n, as<int>(P->tc_err), P->stream, P->cfg.tc_max_ctas, P->cfg.pi_ksplit, part,
                     part_bytes, &chosen));
  P->stats.pi_ksplit_last = chosen;
  mark(P, cls, t0, (double)nb * n * n * K);     // symmetric rank-K update: n^2 K flops per entry
  P->stats.n_kernel_launches += 2;
  int herr = 0;
  CK(cudaMemcpyAsync(&herr, P->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  if (herr != 0) return fail(P, GW_ERR_TIMEOUT, "tensor-core GEMM: bounded wait ran out (code %d)", herr);
  return GW_OK;
}

// W table on the tensor cores (mixed precision) for nc frequency matrices eps_b = 1 - Pi_b held FP32 in ws_mat:
// Newton-Schulz X <- 2X - (X eps) X from the closed-form first iterate 2a I - a^2 eps (a = 2/(1 + lambda_max)),
// converging quadratically because the spectrum of eps lies in [1, lambda_max]; the last iterate is written as
// eps^-1 - 1, and W[r][g] = b_r^T (eps_g^-1 - 1) b_r is reduced straight out of one more GEMM.
// Positions [g0, g0 + nc) of the stage, at the frequencies xi_pos[0 .. nc).
gw_status ns_w_table(gw_plan* P, int g0, int nc, const double* xi_pos) {
  const int n = P->cfg.n_aux, ldn = gw::tc_ld(n);
  const int R = P->n_t * P->n_bas, n_g1 = P->n_g + 1;
  const size_t mat = (size_t)n * n, smat = (size_t)n * ldn, sz = smat * nc;
  // three split parts per operand: the cheap iterations use two, the last iteration and the W reduction three
  TRY(ensure(P, P->ns_E, 3 * sizeof(__nv_bfloat16) * sz));
  TRY(ensure(P, P->ns_Xa, 3 * sizeof(__nv_bfloat16) * sz));
  TRY(ensure(P, P->ns_Xb, 3 * sizeof(__nv_bfloat16) * sz));
  TRY(ensure(P, P->ns_T, 3 * sizeof(__nv_bfloat16) * sz));
  TRY(ensure(P, P->ns_X, sizeof(float) * mat * nc));
  TRY(ensure(P, P->ns_X2, sizeof(float) * mat * nc));
  TRY(ensure(P, P->ns_lam, sizeof(float) * 4 * nc));         // per matrix: lambda estimates, shift, a_b
  TRY(ensure(P, P->ns_vec, sizeof(float) * 2 * (size_t)nc * n));
  TRY(ensure(P, P->tc_err, sizeof(int)));
  CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
  const float* eps = reinterpret_cast<const float*>(P->ws_mat.p);
  auto parts = [&](DevBuf& b) {
    __nv_bfloat16* p0 = as<__nv_bfloat16>(b);
    return gw::TcOperand{{p0, p0 + sz, p0 + 2 * sz}};
  };
  const gw::TcOperand E = parts(P->ns_E), T = parts(P->ns_T);
  const gw::TcOperand Xs[2] = {parts(P->ns_Xa), parts(P->ns_Xb)};
  float* X = as<float>(P->ns_X);
  const size_t t0 = tick(P);
  // Spectrum of each eps_b = 1 - Pi(i xi_b) in [L_b, H_b]: H_b = 1.25 x the power-iteration estimate of
  // lambda_max (power iteration approaches it from below), L_b = max(1, 0.75 x the estimate of lambda_min from the
  // shifted iteration, which approaches it from above); eps >= 1 because -Pi is positive semidefinite.  With
  // a_b = 2/(L_b + H_b) the first iterate X = 2 a I - a^2 eps leaves I - X eps = (I - a eps)^2, every eigenvalue in
  // [0, rho_b^2], rho_b = (H_b - L_b)/(H_b + L_b), and each Newton-Schulz step squares it.  An eigenvalue outside
  // the estimates still converges (0 < a lambda < 2 for lambda < L_b + H_b), only more slowly.
  // One iteration count for every frequency: the first chunk (xi = 0 and the lowest grid points, the widest
  // spectra) fixes it; a later chunk that needs more takes more.
  float* f_hi = as<float>(P->ns_lam);
  float* f_lo = f_hi + nc;
  float* f_ab = f_hi + 3 * nc;
  CK(gw::tc_spectrum_bounds(eps, n, nc, 20, 1.25f, f_hi, f_lo, f_hi + 2 * nc, as<float>(P->ns_vec),
                            as<float>(P->ns_vec) + (size_t)nc * n, P->stream));
  P->stats.n_kernel_launches += 2 + 2 * 2 * 20 + 1;
  std::vector<float> hl(2 * nc);
  CK(cudaMemcpyAsync(hl.data(), f_hi, sizeof(float) * 2 * nc, cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  std::vector<float> ab(nc);
  double rho = 0.0;
  for (int b = 0; b < nc; ++b) {
    const double H = 1.25 * std::max(1.0f, hl[b]);
    const double L = std::max(1.0, 0.75 * (H - hl[nc + b]));
    ab[b] = (float)(2.0 / (L + H));
    rho = std::max(rho, (H - L) / (H + L));
  }
  CK(cudaMemcpyAsync(f_ab, ab.data(), sizeof(float) * nc, cudaMemcpyHostToDevice, P->stream));
  // two-part iterations until rho^(2^k) <= e^-11.5 (about 1e-5), then one three-part iteration (quadratic: to
  // the FP32 floor)
  int k = 2;
  if (rho > 0.0) k = std::max(2, (int)std::ceil(std::log2(11.5 / -std::log(rho))) + 1);
  k = std::min(k, 24);
  if (g0 == 0 || P->ns_kmax == 0) P->ns_kmax = k;
  const int kmax = std::max(k, P->ns_kmax);
  CK(gw::tc_split_rows(eps, nc * n, n, n, const_cast<__nv_bfloat16*>(E.p[0]), const_cast<__nv_bfloat16*>(E.p[1]),
                       P->stream, const_cast<__nv_bfloat16*>(E.p[2])));
  CK(gw::tc_ns_init(eps, n, nc, f_ab, X, const_cast<__nv_bfloat16*>(Xs[0].p[0]),
                    const_cast<__nv_bfloat16*>(Xs[0].p[1]), P->stream, const_cast<__nv_bfloat16*>(Xs[0].p[2])));
  int cur = 0;
  float* Xf[2] = {X, as<float>(P->ns_X2)};
  int xf = 0;
  for (int k = 1; k < kmax; ++k) {
    const bool last = (k == kmax - 1);
    const int ns = last ? 3 : 2;
    if (last) {
      // the products below take X as its own transpose: make the iterate exactly symmetric before the
      // high-precision step, so that its error F maps to -F eps F (quadratic) for any F
      CK(gw::tc_sym_split(Xf[xf], n, nc, Xf[1 - xf], const_cast<__nv_bfloat16*>(Xs[cur].p[0]),
                          const_cast<__nv_bfloat16*>(Xs[cur].p[1]), const_cast<__nv_bfloat16*>(Xs[cur].p[2]),
                          P->stream));
      xf = 1 - xf;
    }
    gw::TcEpi et{};
    et.kind = gw::TC_EPI_AXPBY;
    et.gamma = 1.f;
    et.ldo = n;
    et.ohi = const_cast<__nv_bfloat16*>(T.p[0]);
    et.olo = const_cast<__nv_bfloat16*>(T.p[1]);
    et.olo2 = const_cast<__nv_bfloat16*>(T.p[2]);
    et.ldh = ldn;
    et.oh_bstride = (long)smat;
    // S = X eps   (eps is symmetric, so it is its own K-major B operand)
    CK(gw::tc_gemm_ex(Xs[cur], nc, E, 1, ns, n, n, n, et, as<int>(P->tc_err), P->stream));
    gw::TcEpi ex{};
    ex.kind = gw::TC_EPI_AXPBY;
    ex.xin = Xf[xf];
    ex.x_bstride = (long)mat;
    ex.alpha = 2.f;
    ex.gamma = -1.f;
    ex.beta = last ? -1.f : 0.f;
    ex.out = Xf[xf];
    ex.out_bstride = (long)mat;
    ex.ldo = n;
    ex.ohi = const_cast<__nv_bfloat16*>(Xs[1 - cur].p[0]);
    ex.olo = const_cast<__nv_bfloat16*>(Xs[1 - cur].p[1]);
    ex.olo2 = const_cast<__nv_bfloat16*>(Xs[1 - cur].p[2]);
    ex.ldh = ldn;
    ex.oh_bstride = (long)smat;
    // X <- 2X - S X = 2X - X eps X  (X symmetric: X is its own transpose as the B operand); the last iterate is
    // written as X - I
    CK(gw::tc_gemm_ex(T, nc, Xs[cur], 1, ns, n, n, n, ex, as<int>(P->tc_err), P->stream));
    cur = 1 - cur;
    P->stats.n_kernel_launches += 2;
  }
  mark(P, 2, t0, 2.0 * 2.0 * (double)(kmax - 1) * nc * (double)n * n * n);
  // W table, reduced in the epilogue of one more GEMM into the table zeroed before the chunks:
  //   static point and grid points g >= ns_ndiff:  W[r][g] = b_r^T (eps_g^-1 - 1) b_r
  //   grid points g < ns_ndiff (xi_g well below every D_ia):
  //     W[r][g] - W[r][n_g] = b_r^T eps_g^-1 M_g eps_0^-1 b_r,  M_g = Pi(i xi_g) - Pi(0)
  //                         = 4 xi_g^2 sum_ia B_ia B_ia^T / (D_ia (D_ia^2 + xi_g^2))   (eps_g = eps_0 - M_g).
  // The I term's omega-derivative weighs W_g - W_0 of the diagonal state by w_g/xi_g^2 at the first nodes; there
  // the difference is O(xi^2) and, formed from two separately computed columns, it would carry their rounding
  // error; in this form its error is relative to itself.  W[r][n_g] is added to those columns after the chunks.
  const gw::TcOperand Bn{{P->d_Bnhi, P->d_Bnlo, P->d_Bnlo2}};
  auto wred = [&](const gw::TcOperand& A, int nb, int pos) {
    gw::TcEpi ew{};
    ew.kind = gw::TC_EPI_WRED;
    ew.W = P->d_W;
    ew.wld = n_g1;
    ew.gidx = as<int>(P->ws_gout) + pos;
    ew.bvec = P->d_B_nm_f;
    ew.ldb = n;
    return gw::tc_gemm_ex(A, nb, Bn, 0, 3, n, R, n, ew, as<int>(P->tc_err), P->stream);
  };
  auto shift = [&](const gw::TcOperand& op, int b) {
    return gw::TcOperand{{op.p[0] + b * smat, op.p[1] + b * smat, op.p[2] + b * smat}};
  };
  int b0 = 0;
  if (g0 == 0) {
    if (P->ns_ndiff > 0) {   // keep eps_0^-1 - 1 (split) for the difference columns of later chunks
      TRY(ensure(P, P->ns_E0, 3 * sizeof(__nv_bfloat16) * smat));
      __nv_bfloat16* e0 = as<__nv_bfloat16>(P->ns_E0);
      for (int i = 0; i < 3; ++i)
        CK(cudaMemcpyAsync(e0 + i * smat, Xs[cur].p[i], sizeof(__nv_bfloat16) * smat, cudaMemcpyDeviceToDevice,
                           P->stream));
    }
    b0 = 1;
  }
  // positions [b0, b1) of this chunk are difference columns
  const int b1 = std::max(b0, std::min(nc, P->ns_ndiff + 1 - g0));
  const size_t t1 = tick(P);
  if (b0 > 0) CK(wred(Xs[cur], 1, g0));
  if (nc > b1) CK(wred(shift(Xs[cur], b1), nc - b1, g0 + b1));
  mark(P, 3, t1, 2.0 * (b0 + nc - b1) * (double)n * n * R);
  const int nb = b1 - b0;
  if (nb > 0) {
    __nv_bfloat16* e0 = as<__nv_bfloat16>(P->ns_E0);
    const gw::TcOperand E0{{e0, e0 + smat, e0 + 2 * smat}};
    std::vector<int> kinds(nb, 4);
    std::vector<double> xis(nb);
    for (int b = 0; b < nb; ++b) xis[b] = xi_pos[b0 + b];
    // M_b in FP32 (ws_mat: eps is no longer needed) and split (ns_E)
    float* Mf = as<float>(P->ws_mat);
    TRY(tc_weighted_syrk(P, kinds.data(), xis.data(), nb, 0, 0, Mf, 0, /*reset_err=*/false));
    const size_t t2 = tick(P);
    CK(gw::tc_split_rows(Mf, nb * n, n, n, const_cast<__nv_bfloat16*>(E.p[0]), const_cast<__nv_bfloat16*>(E.p[1]),
                         P->stream, const_cast<__nv_bfloat16*>(E.p[2])));
    // C_b = M_b eps_0^-1 = M_b E_0 + M_b   (E_0 = eps_0^-1 - 1 is symmetric: its own K-major operand)
    float* C = Xf[1 - xf];
    gw::TcEpi e1{};
    e1.kind = gw::TC_EPI_AXPBY;
    e1.gamma = 1.f;
    e1.alpha = 1.f;
    e1.xin = Mf;
    e1.x_bstride = (long)mat;
    e1.out = C;
    e1.out_bstride = (long)mat;
    e1.ldo = n;
    CK(gw::tc_gemm_ex(E, nb, E0, 0, 3, n, n, n, e1, as<int>(P->tc_err), P->stream));
    // C_b^T = eps_0^-1 M_b, split, as the K-major operand of the next product
    for (int b = 0; b < nb; ++b)
      CK(gw::tc_transpose_split(C + b * mat, n, n, const_cast<__nv_bfloat16*>(T.p[0]) + b * smat,
                                const_cast<__nv_bfloat16*>(T.p[1]) + b * smat, P->stream,
                                const_cast<__nv_bfloat16*>(T.p[2]) + b * smat));
    // K_b = eps_b^-1 M_b eps_0^-1 = E_b C_b + C_b, written split for the reduction
    gw::TcEpi e2{};
    e2.kind = gw::TC_EPI_AXPBY;
    e2.gamma = 1.f;
    e2.alpha = 1.f;
    e2.xin = C;
    e2.x_bstride = (long)mat;
    e2.ldo = n;
    e2.ohi = const_cast<__nv_bfloat16*>(Xs[1 - cur].p[0]);
    e2.olo = const_cast<__nv_bfloat16*>(Xs[1 - cur].p[1]);
    e2.olo2 = const_cast<__nv_bfloat16*>(Xs[1 - cur].p[2]);
    e2.ldh = ldn;
    e2.oh_bstride = (long)smat;
    CK(gw::tc_gemm_ex(shift(Xs[cur], b0), nb, T, 1, 3, n, n, n, e2, as<int>(P->tc_err), P->stream));
    mark(P, 2, t2, 2.0 * 2.0 * nb * (double)n * n * n);
    const size_t t3 = tick(P);
    CK(wred(Xs[1 - cur], nb, g0 + b0));
    mark(P, 3, t3, 2.0 * nb * (double)n * n * R);
    P->stats.n_kernel_launches += 4 + nb;
  }
  P->stats.n_kernel_launches += 5;
  int herr = 0;
  CK(cudaMemcpyAsync(&herr, P->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  if (herr != 0) return fail(P, GW_ERR_TIMEOUT, "tensor-core W table: bounded wait ran out (code %d)", herr);
  P->ns_iters_last = kmax;
  return GW_OK;
}

// ---------------------------------------------------------------- FP64 products by digits (oz_gemm.cu)
constexpr int kSmall64 = 128;        // FP64 plans up to here keep the imaginary axis on the FP64 pipe
// Bytes a digit buffer may take (at least one matrix's smallest piece).
size_t oz_cap(const gw_plan* P) { return std::min<size_t>(ws_bytes(P), (size_t)1 << 30); }

gw_status oz_check(gw_plan* P) {
  int herr = 0;
  CK(cudaMemcpyAsync(&herr, P->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  if (herr != 0) return fail(P, GW_ERR_TIMEOUT, "tensor-core FP64 product: bounded wait ran out (code %d)", herr);
  return GW_OK;
}

// K columns a weighted product holds at once: all of them, or as many (a multiple of 128) as the cap allows for the
// digits of one entry's two operands.
int oz_slab(size_t cap, int n, int K) {
  const size_t per_col = 2 * (size_t)gw::OZ_S * n * sizeof(__nv_bfloat16);
  if (per_col * gw::oz_ld(K) <= cap) return K;
  return (int)std::min<size_t>(K, std::max<size_t>(128, cap / per_col / 128 * 128));
}

// out_b = f(B diag(w_b) B^T) in FP64 for nb entries (weights of kind 0, 1, 2 as in tc_pair_weights).  checked (kind 0,
// f = v): tiles whose elements the digits cannot give as accurately as an FP64 sum are computed again (oz_cover).
gw_status oz_weighted_syrk(gw_plan* P, const int* kinds, const double* params, int nb, int mode_even, int mode_odd,
                           double* out, bool checked = false) {
  const int n = P->cfg.n_aux, K = P->n_ov;
  const size_t cap = oz_cap(P);
  const int slab = oz_slab(cap, n, K);
  const size_t one = gw::oz_elems(n, slab);
  // entries at once: their digits within the cap, pairs kept together (even and odd entries have their own modes)
  int eg = (int)std::min<size_t>(nb, std::max<size_t>(1, cap / (2 * one * sizeof(__nv_bfloat16))));
  eg = std::min(eg, 32768);
  if (eg > 1 && eg < nb) eg &= ~1;
  const int tiles = gw::oz_cover_tiles(n);
  TRY(ensure(P, P->oz_A, sizeof(__nv_bfloat16) * one * eg));
  TRY(ensure(P, P->oz_B, sizeof(__nv_bfloat16) * one * eg));
  TRY(ensure(P, P->oz_w, (sizeof(double) + sizeof(int)) * (size_t)K * eg));
  TRY(ensure(P, P->oz_sc, sizeof(double) * 2 * (size_t)n * eg));
  if (checked) TRY(ensure(P, P->oz_part, sizeof(int) * (size_t)tiles * eg));
  TRY(ensure(P, P->tc_kind, sizeof(int) * nb));
  TRY(ensure(P, P->tc_par, sizeof(double) * nb));
  TRY(ensure(P, P->tc_err, sizeof(int)));
  CK(cudaMemcpyAsync(P->tc_kind.p, kinds, sizeof(int) * nb, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->tc_par.p, params, sizeof(double) * nb, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
  double* scB = as<double>(P->oz_sc);
  double* scA = scB + (size_t)n * eg;
  double* f = as<double>(P->oz_w);
  int* h = reinterpret_cast<int*>(f + (size_t)K * eg);
  __nv_bfloat16* dB = as<__nv_bfloat16>(P->oz_B);
  __nv_bfloat16* dA = as<__nv_bfloat16>(P->oz_A);
  for (int b0 = 0; b0 < nb; b0 += eg) {
    const int ne = std::min(eg, nb - b0);
    CK(gw::oz_pair_weights(P->d_D, K, as<int>(P->tc_kind) + b0, as<double>(P->tc_par) + b0, P->cfg.eta, ne, f, h,
                           P->stream));
    if (checked) CK(cudaMemsetAsync(P->oz_part.p, 0, sizeof(int) * (size_t)tiles * ne, P->stream));
    for (int k0 = 0; k0 < K; k0 += slab) {
      const int kc = std::min(slab, K - k0);
      CK(gw::oz_split_weighted(P->d_B_ia, n, k0, kc, K, f, h, K, ne, dA, scA, dB, scB, P->stream));
      const gw::OzOperand A{dA, scA, 1}, B{dB, scB, 1};
      if (checked) CK(gw::oz_cover(A, B, n, kc, ne, as<int>(P->oz_part), P->stream));
      gw::OzEpi ep{};
      ep.kind = gw::OZ_EPI_STORE;
      ep.lower = 1;
      ep.mode_even = (b0 & 1) ? mode_odd : mode_even;
      ep.mode_odd = (b0 & 1) ? mode_even : mode_odd;
      ep.accumulate = k0 > 0;
      ep.out = out + (size_t)b0 * n * n;
      ep.out_bstride = (long)n * n;
      ep.ldo = n;
      CK(gw::oz_gemm(A, B, ne, n, n, kc, ep, as<int>(P->tc_err), P->stream));
      P->stats.n_kernel_launches += checked ? 3 : 2;
    }
    P->stats.n_kernel_launches += 1;
    if (checked)
      LAUNCH(gw::launch_pi_syrk(P->d_B_ia, P->d_D, K, n, as<double>(P->tc_par) + b0, ne, out + (size_t)b0 * n * n, 0,
                                P->stream, as<int>(P->oz_part)));
  }
  return GW_OK;
}

// Matrices and rows of B_nm of one product of oz_w_columns: the inverse factors with their digits, the rows' digits and
// the tiles' sums each within the cap.
void oz_w_blocks(size_t cap, int n, long R, int nc, int* sub, int* rows) {
  const size_t per = gw::oz_elems(n, n) * sizeof(__nv_bfloat16);
  *sub = (int)std::min<size_t>(nc, std::max<size_t>(1, cap / (per + sizeof(double) * n * n)));
  const size_t part = sizeof(double) * gw::oz_sumsq_tiles(n) * (size_t)*sub;
  *rows = (int)std::min<size_t>((size_t)R, std::max<size_t>(128, std::min(cap / (per / n), cap / part)));
}

// W[r][gidx[b]] += |L_b^-1 b_r|^2 for nc Cholesky factors L (ws_mat) and every row of B_nm: the inverse factors, their
// digits and one digit product per block of rows, squares summed per tile in its epilogue and over the tiles after it.
gw_status oz_w_columns(gw_plan* P, const double* L, int nc, const int* gidx) {
  const int n = P->cfg.n_aux, n_g1 = P->n_g + 1;
  const long R = (long)P->n_t * P->n_bas;
  const size_t per = gw::oz_elems(n, n) * sizeof(__nv_bfloat16);
  const int tiles = gw::oz_sumsq_tiles(n);
  int sub, rc;
  oz_w_blocks(oz_cap(P), n, R, nc, &sub, &rc);
  TRY(ensure(P, P->oz_part, sizeof(double) * (size_t)tiles * rc * sub));
  TRY(ensure(P, P->oz_X, sizeof(double) * (size_t)n * n * sub));
  TRY(ensure(P, P->oz_A, sizeof(__nv_bfloat16) * gw::oz_elems(rc, n)));
  TRY(ensure(P, P->oz_B, per * sub));
  TRY(ensure(P, P->oz_sc, sizeof(double) * ((size_t)R + (size_t)n * sub)));
  TRY(ensure(P, P->tc_err, sizeof(int)));
  CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
  double* scR = as<double>(P->oz_sc);
  double* scX = scR + R;
  double* X = as<double>(P->oz_X);
  CK(gw::oz_row_scale(P->d_B_nm, (int)R, n, n, scR, P->stream));
  for (int b0 = 0; b0 < nc; b0 += sub) {
    const int nb = std::min(sub, nc - b0);
    CK(gw::launch_tri_inv(L + (size_t)b0 * n * n, (long)n * n, n, nb, X, (long)n * n, P->stream));
    CK(gw::oz_row_scale(X, n * nb, n, n, scX, P->stream));
    CK(gw::oz_split(X, (long)n * n, n, 0, n, n, scX, nb, as<__nv_bfloat16>(P->oz_B), P->stream));
    for (long r0 = 0; r0 < R; r0 += rc) {
      const int nr = (int)std::min<long>(rc, R - r0);
      if (b0 == 0 || rc < R)
        CK(gw::oz_split(P->d_B_nm + r0 * n, 0, nr, 0, n, n, scR + r0, 1, as<__nv_bfloat16>(P->oz_A), P->stream));
      gw::OzEpi ep{};
      ep.kind = gw::OZ_EPI_SUMSQ;
      ep.part = as<double>(P->oz_part);
      CK(gw::oz_gemm(gw::OzOperand{as<__nv_bfloat16>(P->oz_A), scR + r0, 0},
                     gw::OzOperand{as<__nv_bfloat16>(P->oz_B), scX, 1}, nb, nr, n, n, ep, as<int>(P->tc_err),
                     P->stream));
      CK(gw::oz_sumsq_add(as<double>(P->oz_part), nb, tiles, nr, P->d_W + r0 * n_g1, n_g1, gidx + b0, P->stream));
      P->stats.n_kernel_launches += 3;
    }
    P->stats.n_kernel_launches += 3;
  }
  return GW_OK;
}

// ---------------------------------------------------------------- imaginary-axis screening
template <typename T>
gw_status screening_T(gw_plan* P) {
  const int n = P->cfg.n_aux;
  const int n_g1 = P->n_g + 1;
  const int R = P->n_t * P->n_bas;
  const bool use_tc = (P->cfg.precision == GW_PREC_MIXED);
  // FP64 plans of one digit tile stay on the FP64 pipe: a tile's padding takes the digits' advantage (n_aux 84, 95 pairs,
  // 129 points: Pi 0.35 ms and W 0.24, the job by the step tree 6.3 ms either way), and these plans run the QP searches
  // whose roots, near poles of Sigma, move by 1e-8 with the order in which W is summed.
  const bool small64 = !use_tc && n <= kSmall64;
  // difference-form columns: grid points with xi_g below a tenth of the smallest pair energy (there
  // |Pi(i xi_g) - Pi(0)| <= 1% of |Pi(0)|)
  int n_diff = 0;
  if (use_tc)
    while (n_diff < P->n_g && P->h_xi[n_diff] < 0.1 * P->D_min) ++n_diff;
  // frequency matrices held at once: <= 8 GiB (and the split-operand budget on the tensor-core path)
  const size_t per = (size_t)n * n * sizeof(T);
  int chunk = (int)std::max<size_t>(1, std::min<size_t>((size_t)n_g1, ws_bytes(P) / per));
  if (use_tc) {
    const size_t per_ns = (size_t)n * gw::tc_ld(n) * 24 + (size_t)n * n * 8;   // split E, Xa, Xb, T; FP32 X, eps
    chunk = (int)std::max<size_t>(1, std::min<size_t>((size_t)chunk, ws_bytes(P) / per_ns));
  }
  // mixed precision, one rank: the stage runs at the nodes of the grid (FreqNodes, 35 to 40 of 129 points) and the
  // other columns follow from them; the nodes' 2e-8 is far below the BF16-part products' error.  FP64 plans and sharded
  // plans (each rank owns a block of columns) run at every grid point, so do plans whose caller left room for fewer than
  // three matrices (no need of theirs: the chunked form of the every-point stage, which sharded plans share, is checked
  // against the oracle there) and plans of one 128-row tile a matrix, whose 129 points are one wave and cost less than the
  // search for the nodes (a (H2O)_1 job took 4.68 ms with nodes, 4.48 without; a (H2O)_3 one 4.6 with, 6.8 without).
  const bool use_nodes = use_tc && n > 128 && P->sh_world == 1 && !(P->cfg.workspace_mb > 0 && chunk < 3);
  if (use_nodes && P->nodes_D != P->D_min) {
    P->nodes_D = -1.0;
    P->nodes_ok = gw::freq_nodes(P->h_xi, n_diff, P->D_min, P->nodes);
    if (P->nodes_ok) {
      TRY(ensure(P, P->sk_C, sizeof(double) * P->nodes.C.size()));
      CK(cudaMemcpyAsync(P->sk_C.p, P->nodes.C.data(), sizeof(double) * P->nodes.C.size(), cudaMemcpyHostToDevice,
                         P->stream));
    }
    P->nodes_D = P->D_min;
  }
  const bool nodes = use_nodes && P->nodes_ok;
  P->ns_ndiff = nodes ? P->nodes.n_diff : n_diff;
  // processing order: the static point xi = 0 first, then the grid ascending; gout maps position -> W column
  std::vector<int> gout;
  if (nodes) {
    gout = P->nodes.col;
  } else {
    gout.resize(n_g1);
    gout[0] = P->n_g;
    for (int g = 0; g < P->n_g; ++g) gout[g + 1] = g;
  }
  const int n_pos = (int)gout.size();
  chunk = std::min(chunk, n_pos);
  TRY(ensure(P, P->ws_mat, per * chunk));
  TRY(ensure(P, P->ws_info, sizeof(int) * chunk));
  TRY(ensure(P, P->ws_gout, sizeof(int) * n_pos));
  CK(cudaMemcpyAsync(P->ws_gout.p, gout.data(), sizeof(int) * n_pos, cudaMemcpyHostToDevice, P->stream));
  std::vector<double> xi_all(n_pos);
  for (int i = 0; i < n_pos; ++i) xi_all[i] = gout[i] < P->n_g ? P->h_xi[gout[i]] : 0.0;
  TRY(ensure(P, P->ws_xi, sizeof(double) * n_pos));
  CK(cudaMemcpyAsync(P->ws_xi.p, xi_all.data(), sizeof(double) * n_pos, cudaMemcpyHostToDevice, P->stream));
  P->ns_kmax = 0;
  // positions this rank computes: its block [p0, p1), from position 0 when the block holds difference-form
  // columns (they need eps(0)^-1); columns outside the block are zeroed before the sum across ranks
  int p0 = 0, p1 = n_pos;
  if (P->sh_world > 1) gw_shard_columns(P->n_g, P->sh_rank, P->sh_world, &p0, &p1);
  const int p_begin = (use_tc && p0 > 0 && p0 <= P->ns_ndiff) ? 0 : p0;
  if (use_tc || (small64 && P->sh_world > 1))
    CK(cudaMemsetAsync(P->d_W, 0, sizeof(double) * (size_t)R * n_g1, P->stream));   // W is accumulated / summed
  else if (!small64)
    LAUNCH(CK(gw::launch_w_minus_norm(P->d_B_nm, n, R, n_g1, P->d_W, P->stream)));
  std::vector<int> info(chunk);
  double ms_pi = 0.0;
  for (int g0 = p_begin; g0 < p1; g0 += chunk) {
    const int nc = std::min(chunk, p1 - g0);
    CK(cudaEventRecord(P->ev0, P->stream));
    if (use_tc) {
      std::vector<int> kinds(nc, 0);
      TRY(tc_weighted_syrk(P, kinds.data(), xi_all.data() + g0, nc, 1, 1, reinterpret_cast<float*>(P->ws_mat.p), 0));
    } else {
      const size_t t0 = tick(P);
      if (small64) {
        LAUNCH(gw::launch_pi_syrk(P->d_B_ia, P->d_D, P->n_ov, n, as<double>(P->ws_xi) + g0, nc, as<double>(P->ws_mat),
                                  1, P->stream));
      } else {
        std::vector<int> kinds(nc, 0);
        TRY(oz_weighted_syrk(P, kinds.data(), xi_all.data() + g0, nc, 1, 1, as<double>(P->ws_mat)));
      }
      mark(P, 1, t0, (double)nc * n * n * P->n_ov);
      if (!small64) TRY(oz_check(P));
    }
    CK(cudaEventRecord(P->ev1, P->stream));
    if (use_tc) {
      CK(cudaStreamSynchronize(P->stream));
      ms_pi += now_ms(P, P->ev0, P->ev1);
      TRY(ns_w_table(P, g0, nc, xi_all.data() + g0));
      continue;
    }
    size_t t1 = tick(P);
    LAUNCH(gw::launch_cholesky<double>(as<double>(P->ws_mat), n, (long)n * n, nc, as<int>(P->ws_info), P->stream));
    mark(P, 2, t1, (double)nc * n * n * (double)n / 3.0);
    t1 = tick(P);
    if (small64) {
      const int n_cta = gw::trsm_w_default_ctas();
      TRY(ensure(P, P->oz_X, sizeof(double) * gw::trsm_w_scratch_elems<double>(n, n_cta)));
      LAUNCH(gw::launch_trsm_w<double>(as<double>(P->ws_mat), (long)n * n, n, nc, as<int>(P->ws_gout) + g0, P->d_B_nm,
                                       R, P->d_W, n_g1, as<double>(P->oz_X), n_cta, P->stream));
    } else {
      TRY(oz_w_columns(P, as<double>(P->ws_mat), nc, as<int>(P->ws_gout) + g0));
    }
    mark(P, 3, t1, (double)nc * (double)n * n * R);
    if (!small64) TRY(oz_check(P));
    CK(cudaMemcpyAsync(info.data(), P->ws_info.p, sizeof(int) * nc, cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    ms_pi += now_ms(P, P->ev0, P->ev1);
    for (int i = 0; i < nc; ++i)
      if (info[i] != 0)
        return fail(P, GW_ERR_NUMERIC, "Cholesky of eps(i xi) failed at frequency %d, pivot %d", g0 + i, info[i]);
  }
  if (nodes)
    LAUNCH(CK(gw::launch_w_expand(P->d_W, R, P->n_g, n_pos, as<int>(P->ws_gout), as<double>(P->sk_C), P->stream)));
  else if (use_tc && P->ns_ndiff > 0)
    LAUNCH(gw::launch_w_add_static(P->d_W, R, P->n_g, P->ns_ndiff, P->stream));
  P->stats.ms_pi = ms_pi;
  if (P->sh_world > 1) {
    // keep the owned columns (positions [p0, p1): position 0 is column n_g, position p > 0 is column p - 1), then
    // sum the tables of all ranks: every column comes from exactly one rank
    LAUNCH(gw::launch_w_keep_positions(P->d_W, R, P->n_g, p0, p1, P->stream));
    const size_t cnt = (size_t)R * n_g1;
    P->sh_buf.resize(cnt);
    CK(cudaMemcpyAsync(P->sh_buf.data(), P->d_W, sizeof(double) * cnt, cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    if (P->sh_reduce(P->sh_buf.data(), (long long)cnt, P->sh_ctx) != 0)
      return fail(P, GW_ERR_CUDA, "shard all-reduce of the W table failed");
    CK(cudaMemcpyAsync(P->d_W, P->sh_buf.data(), sizeof(double) * cnt, cudaMemcpyHostToDevice, P->stream));
    CK(cudaStreamSynchronize(P->stream));
  }
  return GW_OK;
}

gw_status ensure_screening(gw_plan* P) {
  if (P->screening_done) return GW_OK;
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  CK(cudaEventRecord(a, P->stream));
  gw_status st;
  if (P->cfg.precision == GW_PREC_MIXED)
    st = screening_T<float>(P);
  else
    st = screening_T<double>(P);
  if (st != GW_OK) { cudaEventDestroy(a); cudaEventDestroy(b); return st; }
  CK(cudaEventRecord(b, P->stream));
  CK(cudaEventSynchronize(b));
  P->stats.ms_screening = now_ms(P, a, b);
  resolve_marks(P);
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  P->screening_done = true;
  return GW_OK;
}

gw_status tc_operator3(gw_plan* P, int nf, const double* xf, const float* V32, float* S32);
gw_status ensure_third_parts(gw_plan* P);

// Half-width (Ha) of the window around each resonance x = +-D_ia whose derivative terms are computed in FP64.
constexpr double kResonantCut = 0.1;

// BF16 elements of the blocked LU's panel operands for a fallback batch of fb matrices: the whole batch, or as many
// matrices as fit in the work space ws, 1 GiB at most (at least one); the LU then runs in sub-batches.
size_t lu_work_elems(int n, long fb, bool fp64, size_t ws) {
  const size_t one = gw::zlu_operand_elems(n, 1, fp64);
  const size_t cap = std::max(one, std::min<size_t>((size_t)1 << 29, ws / 2) / std::max<size_t>(one, 1) * one);
  return std::min(one * (size_t)std::max(1L, fb), cap);
}

// Dense solves for the MINRES batch slots in `need` (Sec. 3.3: build the dielectric matrix and factorise).
// A_j = 1 - Pi(x_j) is built on the tensor cores (mixed) or by the FP64 SIMT kernel, then factorised by the
// batched complex LU; W and the derivative-pass vectors are written into the slot.
template <typename T>
gw_status dense_fallback(gw_plan* P, const std::vector<int>& need, const int* rt, const int* rm, const double* xf,
                         double* w_re, double* w_im, double* resnorm) {
  const int n = P->cfg.n_aux;
  const size_t mat = (size_t)n * n;
  const int nneed = (int)need.size();
  // batch of dense matrices: A planes <= 8 GiB (one LU launch fills the GPU); the tensor-core build runs in
  // sub-batches sized by the split-operand budget
  int fb = (int)std::max<size_t>(1, ws_bytes(P) / (2 * mat * sizeof(T)));
  fb = std::min(fb, nneed);
  const int sub = fb;
  TRY(ensure(P, P->fb_A, sizeof(T) * 2 * mat * fb));
  TRY(ensure(P, P->fb_y, sizeof(T) * 2 * (size_t)n * fb));
  TRY(ensure(P, P->fb_piv, sizeof(int) * (size_t)n * fb));
  TRY(ensure(P, P->fb_info, sizeof(int) * fb));
  TRY(ensure(P, P->fb_idx, sizeof(int) * nneed));
  if (sizeof(T) == 4) {
    TRY(ensure(P, P->fb_y64, sizeof(double) * 2 * (size_t)n * fb));
    TRY(ensure(P, P->fb_V32, sizeof(float) * 2 * (size_t)n * fb));
    TRY(ensure(P, P->fb_S32, sizeof(float) * 2 * (size_t)n * fb));
    TRY(ensure(P, P->fb_Vp, 3 * sizeof(__nv_bfloat16) * 2 * (size_t)gw::tc_ld(n) * fb));
    TRY(ensure(P, P->fb_Up, 3 * sizeof(__nv_bfloat16) * 2 * (size_t)gw::tc_ld(P->n_ov) * fb));
    TRY(ensure(P, P->tc_err, sizeof(int)));
    TRY(ensure(P, P->fb_x, sizeof(double) * fb));
    TRY(ensure(P, P->fb_xs, sizeof(double) * fb));
    TRY(ensure(P, P->fb_rho, sizeof(double) * fb));
    TRY(ensure(P, P->fb_sel, sizeof(int) * fb));
    TRY(ensure(P, P->fb_pos, sizeof(int) * fb));
  }
  TRY(ensure(P, P->fb_lu, sizeof(__nv_bfloat16) * lu_work_elems(n, fb, sizeof(T) == 8, ws_bytes(P))));
  TRY(ensure(P, P->fb_sw, sizeof(int) * gw::zlu_index_ints(fb)));
  TRY(ensure(P, P->fb_linv, sizeof(T) * gw::zlu_linv_elems(fb)));
  if (sizeof(T) == 8) TRY(ensure(P, P->fb_lus, sizeof(double) * gw::zlu_scale_elems(n, fb)));
  CK(cudaMemcpyAsync(P->fb_idx.p, need.data(), sizeof(int) * nneed, cudaMemcpyHostToDevice, P->stream));
  std::vector<double> hx(nneed);
  {
    int mx = 0;
    for (int j : need) mx = std::max(mx, j);
    std::vector<double> xs(mx + 1);
    CK(cudaMemcpyAsync(xs.data(), xf, sizeof(double) * (mx + 1), cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    for (int k = 0; k < nneed; ++k) hx[k] = xs[need[k]];
  }
  std::vector<int> info(fb);
  for (int k0 = 0; k0 < nneed; k0 += fb) {
    const int nf = std::min(fb, nneed - k0);
    T* A = as<T>(P->fb_A);
    if (sizeof(T) == 4) {
      for (int s0 = 0; s0 < nf; s0 += sub) {
        const int ns = std::min(sub, nf - s0);
        std::vector<int> kinds(2 * ns);
        std::vector<double> par(2 * ns);
        for (int k = 0; k < ns; ++k) {
          kinds[2 * k] = 1;
          kinds[2 * k + 1] = 2;
          par[2 * k] = par[2 * k + 1] = hx[k0 + s0 + k];
        }
        TRY(tc_weighted_syrk(P, kinds.data(), par.data(), 2 * ns, 1, 2,
                             reinterpret_cast<float*>(A) + 2 * mat * (size_t)s0, 6));
      }
    } else {
      const size_t t0 = tick(P);
      std::vector<int> kinds(2 * nf);
      std::vector<double> par(2 * nf);
      for (int k = 0; k < nf; ++k) {
        kinds[2 * k] = 1;
        kinds[2 * k + 1] = 2;
        par[2 * k] = par[2 * k + 1] = hx[k0 + k];
      }
      TRY(oz_weighted_syrk(P, kinds.data(), par.data(), 2 * nf, 1, 2, reinterpret_cast<double*>(A)));
      mark(P, 6, t0, 2.0 * nf * (double)mat * P->n_ov);
      TRY(oz_check(P));
    }
    LAUNCH(gw::launch_fallback_rhs<T>(P->d_B_nm, P->n_bas, n, rt, rm, as<int>(P->fb_idx) + k0, nf, as<T>(P->fb_y),
                                      P->stream));
    const size_t tl = tick(P);
    // trailing updates on the tensor cores (FP32: about FP32-accurate six-product split; FP64: exact digits); a bounded
    // wait that runs out in them is reported by the check below (FP64) or by the refinement operator's (mixed)
    CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
    CK(gw::launch_zlu<T>(A, (long)(2 * mat), (long)mat, n, nf, as<int>(P->fb_piv), as<int>(P->fb_info),
                         as<__nv_bfloat16>(P->fb_lu), P->fb_lu.bytes / sizeof(__nv_bfloat16), as<int>(P->fb_sw),
                         as<T>(P->fb_linv), as<double>(P->fb_lus), as<int>(P->tc_err), P->stream));
    P->stats.n_kernel_launches += 4 * ((n + 63) / 64);
    LAUNCH(CK(gw::launch_zlu_solve<T>(A, A + mat, (long)(2 * mat), n, nf, as<int>(P->fb_piv), as<T>(P->fb_y),
                                      as<T>(P->fb_y) + n, 2L * n, P->stream)));
    mark(P, 7, tl, nf * (8.0 / 3.0 * (double)n * n * n + 8.0 * (double)n * n));
    if (sizeof(T) == 4) {
      // iterative refinement with the FP32 factors (matrix-free residuals), solution accumulated in FP64
      float* y32 = reinterpret_cast<float*>(P->fb_y.p);
      const int* idx = as<int>(P->fb_idx) + k0;
      std::vector<double> xk(hx.begin() + k0, hx.begin() + k0 + nf);
      CK(cudaMemcpyAsync(P->fb_x.p, xk.data(), sizeof(double) * nf, cudaMemcpyHostToDevice, P->stream));
      LAUNCH(gw::launch_refine(0, P->d_B_nm, P->n_bas, n, rt, rm, idx, nf, y32, as<double>(P->fb_y64),
                               as<float>(P->fb_V32), nullptr, P->stream));
      // step 1: residual from the three-part tensor-core operator (about FP32-accurate), FP32 LU correction
      {
        const size_t tr = tick(P);
        TRY(tc_operator3(P, nf, as<double>(P->fb_x), as<float>(P->fb_V32), as<float>(P->fb_S32)));
        mark(P, 8, tr, 2.0 * 2.0 * (2.0 * nf) * n * (double)P->n_ov);
        LAUNCH(gw::launch_refine(1, P->d_B_nm, P->n_bas, n, rt, rm, idx, nf, y32, as<double>(P->fb_y64),
                                 as<float>(P->fb_V32), as<float>(P->fb_S32), P->stream));
        LAUNCH(CK(gw::launch_zlu_solve<T>(A, A + mat, (long)(2 * mat), n, nf, as<int>(P->fb_piv), as<T>(P->fb_y),
                                          as<T>(P->fb_y) + n, 2L * n, P->stream)));
        LAUNCH(gw::launch_refine(2, P->d_B_nm, P->n_bas, n, rt, rm, idx, nf, y32, as<double>(P->fb_y64),
                                 as<float>(P->fb_V32), nullptr, P->stream, nullptr, nullptr,
                                 P->cfg.refine_tol > 0.0 ? as<double>(P->fb_rho) : nullptr));
      }
      // step 2, for the solves the first correction shows to be ill-conditioned (|dy|/|y| > refine_tol: a
      // near-resonant x_j, where the operator's FP32-level error limits step 1): residual from the FP64 operator
      if (P->cfg.refine_tol >= 0.0) {
        std::vector<int> sel, pos(nf, -1);
        std::vector<double> xs;
        if (P->cfg.refine_tol > 0.0) {
          std::vector<double> rho(nf);
          CK(cudaMemcpyAsync(rho.data(), P->fb_rho.p, sizeof(double) * nf, cudaMemcpyDeviceToHost, P->stream));
          CK(cudaStreamSynchronize(P->stream));
          for (int k = 0; k < nf; ++k)
            if (!(rho[k] <= P->cfg.refine_tol)) sel.push_back(k);   // NaN selects too
        } else {
          for (int k = 0; k < nf; ++k) sel.push_back(k);
        }
        const int m = (int)sel.size();
        if (m > 0) {
          for (int q = 0; q < m; ++q) {
            pos[sel[q]] = q;
            xs.push_back(hx[k0 + sel[q]]);
          }
          TRY(ensure(P, P->fb_V64, sizeof(double) * 2 * (size_t)n * m));
          TRY(ensure(P, P->fb_S64, sizeof(double) * 2 * (size_t)n * m));
          TRY(ensure(P, P->fb_U64, sizeof(double) * 2 * (size_t)P->n_ov * m));
          CK(cudaMemcpyAsync(P->fb_sel.p, sel.data(), sizeof(int) * m, cudaMemcpyHostToDevice, P->stream));
          CK(cudaMemcpyAsync(P->fb_pos.p, pos.data(), sizeof(int) * nf, cudaMemcpyHostToDevice, P->stream));
          CK(cudaMemcpyAsync(P->fb_xs.p, xs.data(), sizeof(double) * m, cudaMemcpyHostToDevice, P->stream));
          const size_t tr = tick(P);
          LAUNCH(gw::launch_refine_v64(m, n, as<int>(P->fb_sel), as<double>(P->fb_y64), as<double>(P->fb_V64),
                                       P->stream));
          if (P->cfg.refine_df) {
            // double-float (FP32 pair) residual: 48-bit products and sums on the FP32 pipes
            // the hi part of the split is the FP32 copy of B_ia already held by the plan; only the lo part is made
            if (!P->fb_Bl.p) {
              const size_t nb = (size_t)n * P->n_ov;
              TRY(ensure(P, P->fb_Bl, sizeof(float) * nb));
              LAUNCH(gw::launch_df_split(P->d_B_ia, (long)nb, nullptr, as<float>(P->fb_Bl), P->stream));
            }
            LAUNCH(gw::launch_op_gemm1_df(as<double>(P->fb_V64), P->d_B_ia_f, as<float>(P->fb_Bl), P->ld_f, P->d_D,
                                          P->n_ov, n, as<double>(P->fb_xs), P->cfg.eta, m, as<double>(P->fb_U64),
                                          P->stream));
            const int ks = gw::op_gemm2_df_ranges(n, P->n_ov, m);
            if (ks > 1) TRY(ensure(P, P->fb_part, sizeof(double) * 2 * (size_t)n * m * ks));
            LAUNCH(gw::launch_op_gemm2_df(as<double>(P->fb_U64), P->d_B_ia_f, as<float>(P->fb_Bl), P->ld_f, n,
                                          P->n_ov, m, as<double>(P->fb_V64), as<double>(P->fb_S64),
                                          as<double>(P->fb_part), P->stream));
          } else {
            LAUNCH(gw::launch_op_gemm1(as<double>(P->fb_V64), P->d_B_ia, P->d_D, P->n_ov, n, as<double>(P->fb_xs),
                                       P->cfg.eta, m, as<double>(P->fb_U64), P->stream));
            LAUNCH(gw::launch_op_gemm2(as<double>(P->fb_U64), P->d_B_ia, n, P->n_ov, m, as<double>(P->fb_V64),
                                       as<double>(P->fb_S64), 1, P->stream));
          }
          mark(P, 8, tr, 2.0 * 2.0 * (2.0 * m) * n * (double)P->n_ov);
          LAUNCH(gw::launch_refine(1, P->d_B_nm, P->n_bas, n, rt, rm, idx, nf, y32, as<double>(P->fb_y64),
                                   as<float>(P->fb_V32), nullptr, P->stream, as<double>(P->fb_S64),
                                   as<int>(P->fb_pos)));
          LAUNCH(CK(gw::launch_zlu_solve<T>(A, A + mat, (long)(2 * mat), n, nf, as<int>(P->fb_piv), as<T>(P->fb_y),
                                            as<T>(P->fb_y) + n, 2L * n, P->stream)));
          LAUNCH(gw::launch_refine(2, P->d_B_nm, P->n_bas, n, rt, rm, idx, nf, y32, as<double>(P->fb_y64),
                                   as<float>(P->fb_V32), nullptr, P->stream));
          P->stats.n_refine_fp64 += m;
        }
      }
      LAUNCH(gw::launch_fallback_finish64<T>(P->d_B_nm, P->n_bas, n, rt, rm, idx, nf, as<double>(P->fb_y64), w_re,
                                             w_im, resnorm, as<T>(P->mr_V), P->stream, as<double>(P->mr_V64)));
    } else {
      LAUNCH(gw::launch_fallback_finish<T>(P->d_B_nm, P->n_bas, n, rt, rm, as<int>(P->fb_idx) + k0, nf,
                                           as<T>(P->fb_y), w_re, w_im, resnorm, as<T>(P->mr_V), P->stream));
      TRY(oz_check(P));
    }
    CK(cudaMemcpyAsync(info.data(), P->fb_info.p, sizeof(int) * nf, cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    for (int k = 0; k < nf; ++k)
      if (info[k] != 0) return fail(P, GW_ERR_NUMERIC, "dense residue solve: zero pivot at column %d", info[k]);
    P->stats.n_fallback += nf;
  }
  return GW_OK;
}

// Residue operator on the tensor cores (mixed precision), for nr right-hand sides held in V32 [2nr][n]:
// GEMM1 t = B^T z with the complex weights c_ia(x_j) fused into its epilogue (written as split BF16),
// GEMM2 B w with either the plain store (mode 0: [Re; Im] of Pi z) or the 2n embedding of (1 - Pi) z (mode 1).
gw_status tc_operator(gw_plan* P, int nr, const double* xf, const float* V32, float* S32, int mode,
                      const int* run_if = nullptr) {
  const int n = P->cfg.n_aux, n_ov = P->n_ov;
  if (nr <= gw::kSkinnyRhs) {
    LAUNCH(gw::launch_op_skinny(V32, P->d_B_ia_f, P->ld_f, P->d_D, n_ov, n, xf, (float)P->cfg.eta, nr,
                                as<float>(P->mr_U), S32, mode, P->stream, run_if));
    P->stats.n_kernel_launches++;
    return GW_OK;
  }
  const int ldov = gw::tc_ld(n_ov);
  const bool three = P->cfg.op_parts >= 3;
  if (three) TRY(ensure_third_parts(P));
  __nv_bfloat16* vlo2 = three ? as<__nv_bfloat16>(P->mr_Vlo2) : nullptr;
  __nv_bfloat16* ulo2 = three ? as<__nv_bfloat16>(P->mr_Ulo2) : nullptr;
  CK(gw::tc_split_rows(V32, 2 * nr, n, n, as<__nv_bfloat16>(P->mr_Vhi), as<__nv_bfloat16>(P->mr_Vlo), P->stream,
                       vlo2));
  gw::TcEpi e1{};
  e1.kind = gw::TC_EPI_CPAIR;
  e1.Dk = P->d_D;
  e1.x = xf;
  e1.eta = (float)P->cfg.eta;
  e1.ohi = as<__nv_bfloat16>(P->mr_Uhi);
  e1.olo = as<__nv_bfloat16>(P->mr_Ulo);
  e1.olo2 = ulo2;
  e1.ldh = ldov;
  e1.run_if = run_if;
  const gw::TcOperand Vop{{as<__nv_bfloat16>(P->mr_Vhi), as<__nv_bfloat16>(P->mr_Vlo), vlo2}};
  const gw::TcOperand BT{{P->d_BThi, P->d_BTlo, three ? P->d_BTlo2 : nullptr}};
  const int ns = three ? 3 : 2;
  CK(gw::tc_gemm_ex(Vop, 1, BT, 0, ns, 2 * nr, n_ov, n, e1, as<int>(P->tc_err), P->stream));
  gw::TcEpi e2{};
  // the second product's contraction is the long one: over few output tiles it is split in K ranges (at 50 rows,
  // 629 x 4675, 62 us on 5 CTAs before)
  const int ks = gw::tc_ksplit(2 * nr, n, n_ov);
  e2.kind = ks > 1 ? gw::TC_EPI_PART : (mode == 0 ? gw::TC_EPI_STORE : gw::TC_EPI_EMBED);
  e2.out = ks > 1 ? as<float>(P->mr_part) : S32;
  e2.ksplit = ks;
  e2.ldo = n;
  e2.vin = V32;
  e2.ldv = n;
  e2.run_if = run_if;
  const gw::TcOperand Uop{{as<__nv_bfloat16>(P->mr_Uhi), as<__nv_bfloat16>(P->mr_Ulo), ulo2}};
  const gw::TcOperand Bop{{P->d_Bhi, P->d_Blo, three ? P->d_Blo2 : nullptr}};
  CK(gw::tc_gemm_ex(Uop, 1, Bop, 0, ns, 2 * nr, n, n_ov, e2, as<int>(P->tc_err), P->stream));
  P->stats.n_kernel_launches += 3;
  if (ks > 1) {
    CK(gw::tc_part_reduce(as<float>(P->mr_part), ks, 2 * nr, n, V32, mode, S32, run_if, P->stream));
    P->stats.n_kernel_launches++;
  }
  return GW_OK;
}

// Three-part (about FP32-accurate) residue operator for the refinement of dense fallback solves: the embedding
// output S32 = [Re; Im]((1 - Pi(x)) z) for nf right-hand sides z held as (u, v) rows in V32.
gw_status tc_operator3(gw_plan* P, int nf, const double* xf, const float* V32, float* S32) {
  TRY(ensure_third_parts(P));
  const int n = P->cfg.n_aux, n_ov = P->n_ov;
  const size_t sv = 2 * (size_t)nf * gw::tc_ld(n), su = 2 * (size_t)nf * gw::tc_ld(n_ov);
  __nv_bfloat16* vp = as<__nv_bfloat16>(P->fb_Vp);
  __nv_bfloat16* up = as<__nv_bfloat16>(P->fb_Up);
  // tc_err is not reset here: the caller clears it before the blocked LU, whose bounded waits this check covers too
  CK(gw::tc_split_rows(V32, 2 * nf, n, n, vp, vp + sv, P->stream, vp + 2 * sv));
  gw::TcEpi e1{};
  e1.kind = gw::TC_EPI_CPAIR;
  e1.Dk = P->d_D;
  e1.x = xf;
  e1.eta = (float)P->cfg.eta;
  e1.ohi = up;
  e1.olo = up + su;
  e1.olo2 = up + 2 * su;
  e1.ldh = gw::tc_ld(n_ov);
  const gw::TcOperand Vop{{vp, vp + sv, vp + 2 * sv}};
  const gw::TcOperand BT{{P->d_BThi, P->d_BTlo, P->d_BTlo2}};
  CK(gw::tc_gemm_ex(Vop, 1, BT, 0, 3, 2 * nf, n_ov, n, e1, as<int>(P->tc_err), P->stream));
  gw::TcEpi e2{};
  e2.kind = gw::TC_EPI_EMBED;
  e2.out = S32;
  e2.ldo = n;
  e2.vin = V32;
  e2.ldv = n;
  const gw::TcOperand Uop{{up, up + su, up + 2 * su}};
  const gw::TcOperand Bop{{P->d_Bhi, P->d_Blo, P->d_Blo2}};
  CK(gw::tc_gemm_ex(Uop, 1, Bop, 0, 3, 2 * nf, n, n_ov, e2, as<int>(P->tc_err), P->stream));
  P->stats.n_kernel_launches += 3;
  int herr = 0;
  CK(cudaMemcpyAsync(&herr, P->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  if (herr != 0) return fail(P, GW_ERR_TIMEOUT, "tensor-core refinement operator: bounded wait ran out (code %d)", herr);
  return GW_OK;
}

// ---------------------------------------------------------------- FP64 derivative pass
// dW/dx = y^T Pi'(x) y for the rows V (y) of nr right-hand sides: t = V B by exact digits, then the weighted sum; where
// the digits of B^T (16 bytes an element) do not fit, the fused FP64 product.
bool deriv_digits_fit(size_t ws, int n, long K) { return gw::oz_elems((int)K, n) <= ws / 4 / sizeof(__nv_bfloat16); }

gw_status derivative64(gw_plan* P, int batch, int nr, const double* xf, const double* V, double* dw, bool* have_BT) {
  const int n = P->cfg.n_aux, K = P->n_ov, M = 2 * nr;
  // below 2^23 multiply-adds a digit product has no more than a wave of short tiles to gain
  if ((double)M * n * K < 8388608.0 || !deriv_digits_fit(ws_bytes(P), n, K)) {
    LAUNCH(gw::launch_deriv<double>(V, P->d_B_ia, P->d_D, K, n, xf, P->cfg.eta, nr, dw, 0.0, K, P->stream));
    return GW_OK;
  }
  TRY(ensure(P, P->tc_err, sizeof(int)));
  TRY(ensure(P, P->op_sc, sizeof(double) * (K + 2 * (size_t)batch)));
  TRY(ensure(P, P->op_BT, sizeof(__nv_bfloat16) * gw::oz_elems(K, n)));
  TRY(ensure(P, P->op_V, sizeof(__nv_bfloat16) * gw::oz_elems(2 * batch, n)));
  double* scB = as<double>(P->op_sc);
  double* scV = scB + K;
  if (!*have_BT) {                      // once per residue call
    CK(gw::oz_col_scale(P->d_B_ia, n, K, K, scB, P->stream));
    CK(gw::oz_split_transpose(P->d_B_ia, n, K, K, scB, as<__nv_bfloat16>(P->op_BT), P->stream));
    P->stats.n_kernel_launches += 2;
    *have_BT = true;
  }
  CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
  CK(gw::oz_row_digits(V, M, n, n, scV, as<__nv_bfloat16>(P->op_V), P->stream));
  gw::OzEpi e{};
  e.kind = gw::OZ_EPI_STORE;
  e.out = as<double>(P->mr_U);
  e.ldo = K;
  CK(gw::oz_gemm(gw::OzOperand{as<__nv_bfloat16>(P->op_V), scV, 0}, gw::OzOperand{as<__nv_bfloat16>(P->op_BT), scB, 0},
                 1, M, K, n, e, as<int>(P->tc_err), P->stream));
  CK(gw::oz_pole_derivative(as<double>(P->mr_U), K, P->d_D, xf, P->cfg.eta, nr, dw, P->stream));
  P->stats.n_kernel_launches += 3;
  return oz_check(P);
}

// ---------------------------------------------------------------- batched residue solves
// Device arrays in: rt, rm (target index, state), xf (frequency); out: w_re, w_im, dw_re, iters, resnorm.
template <typename T>
gw_status residues_T(gw_plan* P, int nr_total, const int* d_rt, const int* d_rm, const double* d_xf, double* w_re,
                     double* w_im, double* dw_re, int* iters, double* resnorm, int* h_fallback) {
  const int n = P->cfg.n_aux, n_ov = P->n_ov;
  int batch = P->cfg.max_rhs_batch;
  if (batch <= 0) {
    // keep the U buffer (2 batch x n_ov) within ~4 GiB
    size_t cap = (ws_bytes(P) / 2) / ((size_t)2 * n_ov * sizeof(T));
    batch = (int)std::max<size_t>(1, std::min<size_t>(cap, 2048));
  }
  batch = std::min(batch, std::max(1, nr_total));
  TRY(ensure(P, P->mr_V, sizeof(T) * 2 * (size_t)batch * n));
  TRY(ensure(P, P->mr_S, sizeof(T) * 2 * (size_t)batch * n));
  TRY(ensure(P, P->mr_U, sizeof(T) * 2 * (size_t)batch * (sizeof(T) == 4 ? P->ld_f : n_ov)));
  const bool d64 = (sizeof(T) == 4) && P->cfg.deriv_fp64;
  if (sizeof(T) == 4) TRY(ensure(P, P->mr_V64, sizeof(double) * 2 * (size_t)batch * n));
  double* V64 = (sizeof(T) == 4) ? as<double>(P->mr_V64) : nullptr;
  for (DevBuf* b : {&P->mr_vprev, &P->mr_v, &P->mr_d1, &P->mr_d2, &P->mr_x})
    TRY(ensure(P, *b, sizeof(double) * 2 * (size_t)batch * n));
  TRY(ensure(P, P->mr_st, sizeof(MinresState) * batch));
  TRY(ensure(P, P->mr_cnt, sizeof(int)));
  const bool tcop = (sizeof(T) == 4) && P->d_BThi != nullptr;
  if (tcop) {
    // partial products of the full batch and of the last, smaller one
    const int last = nr_total % batch ? nr_total % batch : batch;
    for (int nr : {batch, last}) {
      const int ks = gw::tc_ksplit(2 * nr, n, n_ov);
      if (nr > gw::kSkinnyRhs && ks > 1) TRY(ensure(P, P->mr_part, sizeof(float) * (size_t)ks * 2 * nr * n));
    }
    TRY(ensure(P, P->mr_Vhi, sizeof(__nv_bfloat16) * 2 * (size_t)batch * gw::tc_ld(n)));
    TRY(ensure(P, P->mr_Vlo, sizeof(__nv_bfloat16) * 2 * (size_t)batch * gw::tc_ld(n)));
    TRY(ensure(P, P->mr_Uhi, sizeof(__nv_bfloat16) * 2 * (size_t)batch * gw::tc_ld(n_ov)));
    TRY(ensure(P, P->mr_Ulo, sizeof(__nv_bfloat16) * 2 * (size_t)batch * gw::tc_ld(n_ov)));
    if (P->cfg.op_parts >= 3) {
      TRY(ensure(P, P->mr_Vlo2, sizeof(__nv_bfloat16) * 2 * (size_t)batch * gw::tc_ld(n)));
      TRY(ensure(P, P->mr_Ulo2, sizeof(__nv_bfloat16) * 2 * (size_t)batch * gw::tc_ld(n_ov)));
    }
    TRY(ensure(P, P->tc_err, sizeof(int)));
    CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
  }
  const double eta = P->cfg.eta;
  bool have_BT = false;
  std::vector<double> h_res;
  for (int j0 = 0; j0 < nr_total; j0 += batch) {
    const int nr = std::min(batch, nr_total - j0);
    const int* rt = d_rt + j0;
    const int* rm = d_rm + j0;
    const double* xf = d_xf + j0;
    LAUNCH(gw::launch_gather_rhs<T>(P->d_B_nm, P->n_bas, n, rt, rm, nr, as<T>(P->mr_V), P->stream));
    // rhs = Pi(x) b
    if (tcop) {
      TRY(tc_operator(P, nr, xf, reinterpret_cast<const float*>(P->mr_V.p), reinterpret_cast<float*>(P->mr_S.p), 0));
    } else {
      LAUNCH(gw::launch_op_gemm1(as<double>(P->mr_V), P->d_B_ia, P->d_D, n_ov, n, xf, eta, nr, as<double>(P->mr_U),
                                 P->stream));
      LAUNCH(gw::launch_op_gemm2(as<double>(P->mr_U), P->d_B_ia, n, n_ov, nr, as<double>(P->mr_V),
                                 as<double>(P->mr_S), 0, P->stream));
    }
    LAUNCH(gw::launch_minres_init<T>(as<T>(P->mr_S), nr, n, as<double>(P->mr_vprev), as<double>(P->mr_v),
                                     as<double>(P->mr_d1), as<double>(P->mr_d2), as<double>(P->mr_x),
                                     as<MinresState>(P->mr_st), as<T>(P->mr_V), P->stream));
    const double op_flops = 2.0 * 2.0 * (2.0 * nr) * n * (double)n_ov;   // two GEMMs, 2nr columns each
    // The minres_maxit iterations (operator, then one MINRES step of every right-hand side) are captured as one
    // CUDA graph and launched without host synchronisation.  mr_cnt holds the number of right-hand sides still
    // active after the last step; once it is 0 the operator launches of the remaining iterations return at once
    // and the step kernel leaves every converged right-hand side frozen.
    int* cnt = as<int>(P->mr_cnt);
    CK(cudaMemcpyAsync(cnt, &nr, sizeof(int), cudaMemcpyHostToDevice, P->stream));
    if (P->cfg.minres_maxit > 0) {
      cudaGraph_t graph = nullptr;
      cudaGraphExec_t exec = nullptr;
      CK(cudaStreamBeginCapture(P->stream, cudaStreamCaptureModeThreadLocal));
      gw_status cap = GW_OK;
      for (int it = 0; it < P->cfg.minres_maxit && cap == GW_OK; ++it) {
        if (tcop) {
          cap = tc_operator(P, nr, xf, reinterpret_cast<const float*>(P->mr_V.p),
                            reinterpret_cast<float*>(P->mr_S.p), 1, cnt);
        } else {
          gw::launch_op_gemm1(as<double>(P->mr_V), P->d_B_ia, P->d_D, n_ov, n, xf, eta, nr, as<double>(P->mr_U),
                              P->stream, cnt);
          gw::launch_op_gemm2(as<double>(P->mr_U), P->d_B_ia, n, n_ov, nr, as<double>(P->mr_V), as<double>(P->mr_S), 1,
                              P->stream, cnt);
          P->stats.n_kernel_launches += 2;
        }
        if (cudaMemsetAsync(cnt, 0, sizeof(int), P->stream) != cudaSuccess) cap = GW_ERR_CUDA;
        gw::launch_minres_step<T>(as<T>(P->mr_S), nr, n, P->cfg.minres_tol, as<double>(P->mr_vprev),
                                  as<double>(P->mr_v), as<double>(P->mr_d1), as<double>(P->mr_d2),
                                  as<double>(P->mr_x), as<MinresState>(P->mr_st), as<T>(P->mr_V), cnt, P->stream);
        P->stats.n_kernel_launches++;
      }
      const cudaError_t ec = cudaStreamEndCapture(P->stream, &graph);
      if (cap != GW_OK) {
        if (graph) cudaGraphDestroy(graph);
        return cap == GW_ERR_CUDA ? fail(P, GW_ERR_CUDA, "MINRES graph capture failed") : cap;
      }
      CK(ec);
      const cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
      cudaGraphDestroy(graph);
      CK(ei);
      const size_t tg = tick(P);
      const cudaError_t el = cudaGraphLaunch(exec, P->stream);
      const size_t tg1 = tick(P);
      if (el != cudaSuccess) {
        cudaGraphExecDestroy(exec);
        CK(el);
      }
      CK(cudaStreamSynchronize(P->stream));
      cudaGraphExecDestroy(exec);
      P->stats.n_graph_launches++;
      // operator iterations that ran: the largest MINRES iteration count of the batch (states of converged
      // right-hand sides are frozen)
      std::vector<MinresState> hst(nr);
      CK(cudaMemcpy(hst.data(), P->mr_st.p, sizeof(MinresState) * nr, cudaMemcpyDeviceToHost));
      int ran = 0;
      for (const auto& x : hst) ran = std::max(ran, x.iters);
      if (tg != (size_t)-1 && tg1 != (size_t)-1) P->marks.push_back({4, tg, tg1, op_flops * ran});
      P->stats.launches_kernel[4] += ran;
    }
    if (tcop) {
      int herr = 0;
      CK(cudaMemcpyAsync(&herr, P->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, P->stream));
      CK(cudaStreamSynchronize(P->stream));
      if (herr != 0) return fail(P, GW_ERR_TIMEOUT, "tensor-core operator GEMM: bounded wait ran out (code %d)", herr);
    }
    LAUNCH(gw::launch_minres_finish<T>(P->d_B_nm, P->n_bas, n, rt, rm, nr, as<double>(P->mr_x),
                                       as<MinresState>(P->mr_st), w_re + j0, w_im + j0, iters + j0, resnorm + j0,
                                       as<T>(P->mr_V), P->stream, V64));
    // dense fallback for right-hand sides above the fallback threshold (Sec. 3.3, MINRES defaults paragraph)
    h_res.resize(nr);
    CK(cudaMemcpyAsync(h_res.data(), resnorm + j0, sizeof(double) * nr, cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    std::vector<int> need;
    for (int j = 0; j < nr; ++j) {
      bool bad = !(h_res[j] <= P->cfg.minres_fallback_tol);
      if (h_fallback) h_fallback[j0 + j] = bad ? 1 : 0;
      if (bad) need.push_back(j);
    }
    if (!need.empty()) TRY(dense_fallback<T>(P, need, rt, rm, xf, w_re + j0, w_im + j0, resnorm + j0));
    // dW/dx = y^T Pi'(x) y, reduced in FP64 inside the GEMM.  Mixed: the FP32 pass leaves out the pairs within
    // kResonantCut of resonance, where c'(x) reaches 2/eta^2 and FP32 rounding of t = B^T y would dominate dW;
    // those are added in FP64.
    CK(cudaMemsetAsync(dw_re + j0, 0, sizeof(double) * nr, P->stream));
    const size_t td = tick(P);
    if (d64) {
      LAUNCH(gw::launch_deriv<double>(V64, P->d_B_ia, P->d_D, n_ov, n, xf, eta, nr, dw_re + j0, 0.0, n_ov, P->stream));
    } else if (sizeof(T) == 4) {
      LAUNCH(gw::launch_deriv<float>(as<float>(P->mr_V), P->d_B_ia_f, P->d_D, n_ov, n, xf, eta, nr, dw_re + j0,
                                     kResonantCut, P->ld_f, P->stream));
      LAUNCH(gw::launch_deriv_resonant(V64, P->d_B_ia, n_ov, n, P->d_Dsort, P->d_Dkidx, xf, nr, eta, kResonantCut,
                                       dw_re + j0, P->stream));
    } else {
      TRY(derivative64(P, batch, nr, xf, as<double>(P->mr_V), dw_re + j0, &have_BT));
    }
    mark(P, 4, td, 2.0 * (2.0 * nr) * n * (double)n_ov);
  }
  return GW_OK;
}

gw_status residues(gw_plan* P, int nr, const int* d_rt, const int* d_rm, const double* d_xf, double* w_re,
                   double* w_im, double* dw_re, int* iters, double* resnorm, int* h_fallback) {
  if (nr <= 0) return GW_OK;
  CK(cudaEventRecord(P->ev2, P->stream));
  gw_status st = (P->cfg.precision == GW_PREC_MIXED)
                     ? residues_T<float>(P, nr, d_rt, d_rm, d_xf, w_re, w_im, dw_re, iters, resnorm, h_fallback)
                     : residues_T<double>(P, nr, d_rt, d_rm, d_xf, w_re, w_im, dw_re, iters, resnorm, h_fallback);
  if (st != GW_OK) return st;
  CK(cudaEventRecord(P->ev1, P->stream));
  CK(cudaEventSynchronize(P->ev1));
  P->stats.ms_residues += now_ms(P, P->ev2, P->ev1);
  resolve_marks(P);
  P->stats.n_rhs_solved += nr;
  std::vector<int> it(nr);
  CK(cudaMemcpy(it.data(), iters, sizeof(int) * nr, cudaMemcpyDeviceToHost));
  for (int v : it) P->stats.n_minres_iters += v;
  return GW_OK;
}

// Residues of eq. "rnn" at omega_t for the active targets: (t, m, x = e_m - omega_t, coef = sign * theta).
// Evaluation points p (target tmap[p], or p without a map) at omega[p]; start[p] .. start[p + 1] are point p's
// entries.
void build_residue_list(gw_plan* P, const std::vector<double>& omega, const std::vector<unsigned char>& active,
                        std::vector<int>& rt, std::vector<int>& rm, std::vector<double>& xf,
                        std::vector<double>& coef, std::vector<int>& start, const std::vector<int>* tmap = nullptr) {
  rt.clear(); rm.clear(); xf.clear(); coef.clear();
  const int np = (int)omega.size();
  start.assign(np + 1, 0);
  for (int pt = 0; pt < np; ++pt) {
    start[pt] = (int)rt.size();
    if (!active[pt]) continue;
    const int t = tmap ? (*tmap)[pt] : pt;
    const int sp = P->h_spin[t];
    const double w = omega[pt];
    for (int m = 0; m < P->n_bas; ++m) {
      const double e = P->h_eps_g[sp][m];
      double th;
      double sg;
      if (m < P->occ_s[sp]) {
        th = (e > w) ? 1.0 : (e == w ? 0.5 : 0.0);
        sg = -1.0;
      } else {
        th = (w > e) ? 1.0 : (w == e ? 0.5 : 0.0);
        sg = 1.0;
      }
      if (th == 0.0) continue;
      rt.push_back(t);
      rm.push_back(m);
      xf.push_back(e - w);
      coef.push_back(sg * th);
    }
  }
  start[np] = (int)rt.size();
}

// Sigma_c = R - I (and derivative) at evaluation points p: target tmap[p] (p itself without a map) at omega[p],
// for the active points, into sg_R/sg_dR/sg_I/sg_dI [n points].  Every point's residues share one batched solve.
gw_status sigma_eval(gw_plan* P, const std::vector<double>& omega, const std::vector<unsigned char>& active,
                     int* n_fallback_out, const std::vector<int>* tmap = nullptr) {
  const int n_t = (int)omega.size();
  TRY(ensure(P, P->sg_I, sizeof(double) * n_t));
  TRY(ensure(P, P->sg_dI, sizeof(double) * n_t));
  TRY(ensure(P, P->sg_R, sizeof(double) * n_t));
  TRY(ensure(P, P->sg_dR, sizeof(double) * n_t));
  TRY(ensure(P, P->sg_om, sizeof(double) * n_t));
  TRY(ensure(P, P->sg_act, n_t));
  TRY(ensure(P, P->sg_start, sizeof(int) * (n_t + 1)));
  CK(cudaMemcpyAsync(P->sg_om.p, omega.data(), sizeof(double) * n_t, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->sg_act.p, active.data(), n_t, cudaMemcpyHostToDevice, P->stream));
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  CK(cudaEventRecord(a, P->stream));
  const int* d_tmap = nullptr;
  if (tmap) {
    TRY(ensure(P, P->sg_tmap, sizeof(int) * n_t));
    CK(cudaMemcpyAsync(P->sg_tmap.p, tmap->data(), sizeof(int) * n_t, cudaMemcpyHostToDevice, P->stream));
    d_tmap = as<int>(P->sg_tmap);
  }
  LAUNCH(gw::launch_sigma_imag(P->d_W, n_t, P->n_bas, P->n_g, P->d_eps_g, P->d_xi, P->d_wt, as<double>(P->sg_om),
                               P->cfg.static_subtraction, as<double>(P->sg_I), as<double>(P->sg_dI),
                               as<unsigned char>(P->sg_act), P->stream, d_tmap, P->d_spin));
  CK(cudaEventRecord(b, P->stream));
  std::vector<int> rt, rm, start;
  std::vector<double> xf, coef;
  build_residue_list(P, omega, active, rt, rm, xf, coef, start, tmap);
  if (P->sh_world > 1) {
    // this rank's right-hand sides: entry j of the full list with j % world == rank (the per-target sums of R
    // and dR are then added across ranks)
    std::vector<int> rt2, rm2, start2(n_t + 1, 0);
    std::vector<double> xf2, coef2;
    for (int t = 0; t < n_t; ++t) {
      start2[t] = (int)rt2.size();
      for (int j = start[t]; j < start[t + 1]; ++j)
        if (j % P->sh_world == P->sh_rank) {
          rt2.push_back(rt[j]);
          rm2.push_back(rm[j]);
          xf2.push_back(xf[j]);
          coef2.push_back(coef[j]);
        }
    }
    start2[n_t] = (int)rt2.size();
    rt.swap(rt2); rm.swap(rm2); xf.swap(xf2); coef.swap(coef2); start.swap(start2);
  }
  const int nr = (int)rt.size();
  TRY(ensure(P, P->mr_rt, sizeof(int) * std::max(1, nr)));
  TRY(ensure(P, P->mr_rm, sizeof(int) * std::max(1, nr)));
  TRY(ensure(P, P->mr_xf, sizeof(double) * std::max(1, nr)));
  TRY(ensure(P, P->sg_coef, sizeof(double) * std::max(1, nr)));
  TRY(ensure(P, P->mr_wre, sizeof(double) * std::max(1, nr)));
  TRY(ensure(P, P->mr_wim, sizeof(double) * std::max(1, nr)));
  TRY(ensure(P, P->mr_dwre, sizeof(double) * std::max(1, nr)));
  TRY(ensure(P, P->mr_it, sizeof(int) * std::max(1, nr)));
  TRY(ensure(P, P->mr_res, sizeof(double) * std::max(1, nr)));
  if (nr > 0) {
    CK(cudaMemcpyAsync(P->mr_rt.p, rt.data(), sizeof(int) * nr, cudaMemcpyHostToDevice, P->stream));
    CK(cudaMemcpyAsync(P->mr_rm.p, rm.data(), sizeof(int) * nr, cudaMemcpyHostToDevice, P->stream));
    CK(cudaMemcpyAsync(P->mr_xf.p, xf.data(), sizeof(double) * nr, cudaMemcpyHostToDevice, P->stream));
    CK(cudaMemcpyAsync(P->sg_coef.p, coef.data(), sizeof(double) * nr, cudaMemcpyHostToDevice, P->stream));
  }
  CK(cudaMemcpyAsync(P->sg_start.p, start.data(), sizeof(int) * (n_t + 1), cudaMemcpyHostToDevice, P->stream));
  std::vector<int> fb(std::max(1, nr), 0);
  TRY(residues(P, nr, as<int>(P->mr_rt), as<int>(P->mr_rm), as<double>(P->mr_xf), as<double>(P->mr_wre),
               as<double>(P->mr_wim), as<double>(P->mr_dwre), as<int>(P->mr_it), as<double>(P->mr_res), fb.data()));
  LAUNCH(gw::launch_residue_reduce(as<int>(P->sg_start), n_t, as<double>(P->sg_coef), as<double>(P->mr_wre),
                                   as<double>(P->mr_dwre), as<double>(P->sg_R), as<double>(P->sg_dR), P->stream));
  if (P->sh_world > 1) {
    // R and dR of every target summed over the ranks' residue subsets (the I term is computed on every rank)
    P->sh_buf.resize(2 * (size_t)n_t);
    CK(cudaMemcpyAsync(P->sh_buf.data(), P->sg_R.p, sizeof(double) * n_t, cudaMemcpyDeviceToHost, P->stream));
    CK(cudaMemcpyAsync(P->sh_buf.data() + n_t, P->sg_dR.p, sizeof(double) * n_t, cudaMemcpyDeviceToHost,
                       P->stream));
    CK(cudaStreamSynchronize(P->stream));
    if (P->sh_reduce(P->sh_buf.data(), 2LL * n_t, P->sh_ctx) != 0)
      return fail(P, GW_ERR_CUDA, "shard all-reduce of the residue terms failed");
    CK(cudaMemcpyAsync(P->sg_R.p, P->sh_buf.data(), sizeof(double) * n_t, cudaMemcpyHostToDevice, P->stream));
    CK(cudaMemcpyAsync(P->sg_dR.p, P->sh_buf.data() + n_t, sizeof(double) * n_t, cudaMemcpyHostToDevice,
                       P->stream));
  }
  CK(cudaStreamSynchronize(P->stream));
  P->stats.ms_sigma_imag += now_ms(P, a, b);
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  int nf = 0;
  for (int j = 0; j < nr; ++j) nf += fb[j];
  if (n_fallback_out) *n_fallback_out = nf;
  for (int t = 0; t < n_t; ++t) P->stats.n_sigma_evals += active[t] ? 1 : 0;
  return GW_OK;
}

// Pair-energy table D [n_ov] (the columns of B_ia) on the device; in mixed precision also its ascending order with
// the pair index of each entry (for the resonance windows of the derivative pass) and its minimum.
gw_status set_pair_table(gw_plan* P, const std::vector<double>& D) {
  CK(cudaMemcpyAsync(P->d_D, D.data(), sizeof(double) * P->n_ov, cudaMemcpyHostToDevice, P->stream));
  double dmin = D.empty() ? 0.0 : D[0];
  for (double v : D) dmin = std::min(dmin, v);
  P->D_min = dmin;
  if (P->d_Dsort) {
    std::vector<int> order((size_t)P->n_ov);
    for (size_t k = 0; k < order.size(); ++k) order[k] = (int)k;
    std::sort(order.begin(), order.end(), [&](int a, int b) { return D[a] < D[b]; });
    std::vector<double> Ds(order.size());
    for (size_t k = 0; k < order.size(); ++k) Ds[k] = D[order[k]];
    CK(cudaMemcpyAsync(P->d_Dsort, Ds.data(), sizeof(double) * P->n_ov, cudaMemcpyHostToDevice, P->stream));
    CK(cudaMemcpyAsync(P->d_Dkidx, order.data(), sizeof(int) * P->n_ov, cudaMemcpyHostToDevice, P->stream));
    CK(cudaStreamSynchronize(P->stream));
  }
  CK(cudaStreamSynchronize(P->stream));
  return GW_OK;
}

// W's energies: d_eps, the pair energies D_ia = e_a - e_i (ia = i n_virt + a) and, in mixed precision, their
// ascending order and the smallest one.
gw_status set_pair_energies(gw_plan* P, const double* eps, const double* eps_b = nullptr) {
  CK(cudaMemcpyAsync(P->d_eps, eps, sizeof(double) * P->n_bas, cudaMemcpyHostToDevice, P->stream));
  std::vector<double> D;
  D.reserve((size_t)P->n_ov);
  for (int sp = 0; sp < P->n_spin; ++sp) {      // spin blocks side by side: the columns of the (open-shell) B_ia
    const double* e = sp == 0 ? eps : eps_b;
    const int n_occ = P->occ_s[sp], n_virt = P->n_bas - n_occ;
    for (int i = 0; i < n_occ; ++i)
      for (int a = 0; a < n_virt; ++a) D.push_back(e[n_occ + a] - e[i]);
  }
  P->sd_done = false;             // the Casida poles follow W's energies
  return set_pair_table(P, D);
}

// G's energies (host copy for the residue list, device copy for the I term).
gw_status set_g_energies(gw_plan* P, int spin, const double* eps) {
  P->h_eps_g[spin].assign(eps, eps + P->n_bas);
  CK(cudaMemcpyAsync(P->d_eps_g + (size_t)spin * P->n_bas, eps, sizeof(double) * P->n_bas, cudaMemcpyHostToDevice,
                     P->stream));
  CK(cudaStreamSynchronize(P->stream));
  return GW_OK;
}

__global__ void convert_f64_f32_kernel(const double* __restrict__ a, float* __restrict__ b, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    b[i] = (float)a[i];
}

__global__ void scale_kernel(double* __restrict__ a, size_t n, double f) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) a[i] *= f;
}

// rows x cols FP64 (contiguous) to FP32 rows of ldb elements, zero padded.
__global__ void convert_rows_kernel(const double* __restrict__ a, int rows, int cols, float* __restrict__ b,
                                    long ldb) {
  for (int r = blockIdx.y; r < rows; r += gridDim.y)
    for (long c = blockIdx.x * (long)blockDim.x + threadIdx.x; c < ldb; c += (long)gridDim.x * blockDim.x)
      b[(long)r * ldb + c] = c < cols ? (float)a[(long)r * cols + c] : 0.f;
}

// Third BF16 parts of B_ia and B_ia^T, made when a three-part operator first needs them (the hi and lo parts are
// rewritten with the same values).
gw_status ensure_third_parts(gw_plan* P) {
  if (P->d_Blo2) return GW_OK;
  const int n = P->cfg.n_aux;
  TRY(dmalloc(P, &P->d_Blo2, sizeof(__nv_bfloat16) * (size_t)n * gw::tc_ld(P->n_ov)));
  TRY(dmalloc(P, &P->d_BTlo2, sizeof(__nv_bfloat16) * (size_t)P->n_ov * gw::tc_ld(n)));
  CK(gw::tc_split_rows(P->d_B_ia_f, n, P->n_ov, (int)P->ld_f, P->d_Bhi, P->d_Blo, P->stream, P->d_Blo2));
  CK(gw::tc_transpose_split(P->d_B_ia_f, n, P->n_ov, P->d_BThi, P->d_BTlo, P->stream, P->d_BTlo2, P->ld_f));
  P->stats.n_kernel_launches += 2;
  return GW_OK;
}

}  // namespace

// ==================================================================== C ABI
extern "C" {

void gw_config_default(gw_config* c) {
  if (!c) return;
  std::memset(c, 0, sizeof(*c));
  c->n_freq = 128;
  c->x0 = 0.5;
  c->eta = 1e-3;
  c->precision = GW_PREC_FP64;
  c->minres_maxit = 25;
  c->minres_tol = 5e-5;
  c->minres_fallback_tol = 1e-4;
  c->qp_maxit = 50;
  c->qp_tol = 1e-8;
  c->static_subtraction = 1;
  c->max_rhs_batch = 0;
  c->refine_tol = 1e-6;
  c->op_parts = 2;
  c->refine_df = 1;
  c->qp_window = 0.5;
  c->qp_window_points = 64;
}

static void free_plan(gw_plan* P) {
  if (!P) return;
  if (P->stream) cudaStreamSynchronize(P->stream);
  for (DevBuf* b : P->bufs)
    plan_free(P, b->p, 0);
  double* owned[] = {P->d_eps, P->d_eps_g, P->d_xi, P->d_wt, P->d_sx, P->d_shift, P->d_en, P->d_W};
  plan_free(P, P->d_spin, 0);
  plan_free(P, P->d_occ_t, 0);
  for (double* p : owned)
    plan_free(P, p, 0);
  if (P->own_B) {
    plan_free(P, P->d_B_ia, 0);
    plan_free(P, P->d_B_nm, 0);
  }
  plan_free(P, P->d_B_ia_f, 0);
  plan_free(P, P->d_B_nm_f, 0);
  plan_free(P, P->d_Bhi, 0);
  plan_free(P, P->d_Blo, 0);
  plan_free(P, P->d_BThi, 0);
  plan_free(P, P->d_BTlo, 0);
  plan_free(P, P->d_Blo2, 0);
  plan_free(P, P->d_Bp_hi, 0);
  plan_free(P, P->d_Bp_lo, 0);
  plan_free(P, P->d_BTlo2, 0);
  plan_free(P, P->d_D, 0);
  plan_free(P, P->d_Dsort, 0);
  plan_free(P, P->d_Dkidx, 0);
  plan_free(P, P->d_Bnhi, 0);
  plan_free(P, P->d_Bnlo, 0);
  plan_free(P, P->d_Bnlo2, 0);
  for (char* q : P->slabs) cudaFree(q);
  if (P->ev0) cudaEventDestroy(P->ev0);
  if (P->ev1) cudaEventDestroy(P->ev1);
  if (P->ev2) cudaEventDestroy(P->ev2);
  for (cudaEvent_t e : P->tpool) cudaEventDestroy(e);
  if (P->own_stream && P->stream) cudaStreamDestroy(P->stream);
  delete P;
}

// Open-shell inputs of gw_plan_create_uks: the beta channel (its energies, occupations and B_ia block) and the
// spin of every target; the alpha channel comes through the closed-shell arguments.
struct UksInput {
  const double* eps_b;
  int n_occ_b;
  const double* B_ia_b;
  const int* spins;
};

static gw_status plan_create_impl(gw_plan* P, const gw_config* cfg, const double* eps, const double* B_ia,
                                  const double* B_nm, const int* targets, int n_targets, const double* vxc,
                                  const double* xi, const double* wt, unsigned flags, void* stream,
                                  const UksInput* uks = nullptr) {
  P->cfg = *cfg;
  P->flags = flags;
  P->n_bas = cfg->n_occ + cfg->n_virt;
  P->n_spin = uks ? 2 : 1;
  P->occ_s[0] = cfg->n_occ;
  P->occ_s[1] = uks ? uks->n_occ_b : cfg->n_occ;
  const long n_ov_a = (long)cfg->n_occ * cfg->n_virt;
  const long n_ov_b = uks ? (long)uks->n_occ_b * (P->n_bas - uks->n_occ_b) : 0;
  P->n_ov = (int)(n_ov_a + n_ov_b);
  P->n_t = n_targets;
  P->n_g = cfg->n_freq;
  if (stream) {
    P->stream = (cudaStream_t)stream;
  } else {
    CK(cudaStreamCreateWithFlags(&P->stream, cudaStreamNonBlocking));
    P->own_stream = true;
  }
  CK(cudaEventCreate(&P->ev0));
  CK(cudaEventCreate(&P->ev1));
  CK(cudaEventCreate(&P->ev2));
  const int n = cfg->n_aux;
  P->h_eps.assign(eps, eps + P->n_bas);
  P->h_eps_s[0] = P->h_eps;
  P->h_eps_s[1] = uks ? std::vector<double>(uks->eps_b, uks->eps_b + P->n_bas) : P->h_eps;
  P->h_eps_g[0] = P->h_eps_s[0];
  P->h_eps_g[1] = P->h_eps_s[1];
  P->h_targets.assign(targets, targets + n_targets);
  P->h_spin.assign(n_targets, 0);
  if (uks)
    for (int t = 0; t < n_targets; ++t) P->h_spin[t] = uks->spins[t];
  // grid
  P->h_xi.resize(P->n_g);
  P->h_wt.resize(P->n_g);
  if (xi && wt) {
    for (int g = 0; g < P->n_g; ++g) { P->h_xi[g] = xi[g]; P->h_wt[g] = wt[g]; }
  } else {
    gw_grid(P->n_g, cfg->x0, P->h_xi.data(), P->h_wt.data());
  }
  std::vector<double> xi_all(P->h_xi);
  xi_all.push_back(0.0);
  TRY(dmalloc(P, &P->d_eps, sizeof(double) * P->n_bas));
  TRY(dmalloc(P, &P->d_eps_g, sizeof(double) * P->n_spin * P->n_bas));
  TRY(dmalloc(P, &P->d_xi, sizeof(double) * (P->n_g + 1)));
  TRY(dmalloc(P, &P->d_wt, sizeof(double) * std::max(1, P->n_g)));
  TRY(dmalloc(P, &P->d_sx, sizeof(double) * std::max(1, n_targets)));
  TRY(dmalloc(P, &P->d_shift, sizeof(double) * std::max(1, n_targets)));
  TRY(dmalloc(P, &P->d_en, sizeof(double) * std::max(1, n_targets)));
  TRY(dmalloc(P, &P->d_W, sizeof(double) * (size_t)n_targets * P->n_bas * (P->n_g + 1)));
  TRY(dmalloc(P, &P->d_D, sizeof(double) * (size_t)P->n_ov));
  for (int sp = 0; sp < P->n_spin; ++sp) TRY(set_g_energies(P, sp, P->h_eps_s[sp].data()));
  CK(cudaMemcpyAsync(P->d_xi, xi_all.data(), sizeof(double) * (P->n_g + 1), cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->d_wt, P->h_wt.data(), sizeof(double) * P->n_g, cudaMemcpyHostToDevice, P->stream));
  if (uks) {
    std::vector<int> occ_t(n_targets);
    for (int t = 0; t < n_targets; ++t) occ_t[t] = P->occ_s[P->h_spin[t]];
    TRY(dmalloc(P, &P->d_spin, sizeof(int) * n_targets));
    TRY(dmalloc(P, &P->d_occ_t, sizeof(int) * n_targets));
    CK(cudaMemcpyAsync(P->d_spin, P->h_spin.data(), sizeof(int) * n_targets, cudaMemcpyHostToDevice, P->stream));
    CK(cudaMemcpyAsync(P->d_occ_t, occ_t.data(), sizeof(int) * n_targets, cudaMemcpyHostToDevice, P->stream));
    CK(cudaStreamSynchronize(P->stream));
  }
  const size_t nB = (size_t)n * P->n_ov, nBn = (size_t)n_targets * P->n_bas * n;
  cudaMemcpyKind kind = (flags & GW_INPUT_ON_DEVICE) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  if (uks) {
    // the two spin channels side by side along the pair axis, each scaled by 1/sqrt(2): the closed-shell formulas
    // (factor 2 for the two spins) then give sum over sigma with factor 1 per channel (Sec. 3.3, Pi with Sigma_s)
    P->own_B = true;
    TRY(dmalloc(P, &P->d_B_ia, sizeof(double) * nB));
    TRY(dmalloc(P, &P->d_B_nm, sizeof(double) * nBn));
    CK(cudaMemcpy2DAsync(P->d_B_ia, sizeof(double) * P->n_ov, B_ia, sizeof(double) * n_ov_a, sizeof(double) * n_ov_a,
                         n, kind, P->stream));
    if (n_ov_b > 0)
      CK(cudaMemcpy2DAsync(P->d_B_ia + n_ov_a, sizeof(double) * P->n_ov, uks->B_ia_b, sizeof(double) * n_ov_b,
                           sizeof(double) * n_ov_b, n, kind, P->stream));
    LAUNCH((scale_kernel<<<1024, 256, 0, P->stream>>>(P->d_B_ia, nB, 0.70710678118654752440)));
    CK(cudaMemcpyAsync(P->d_B_nm, B_nm, sizeof(double) * nBn, kind, P->stream));
  } else if (flags & GW_BORROW_DEVICE_PTRS) {
    P->own_B = false;
    P->d_B_ia = const_cast<double*>(B_ia);
    P->d_B_nm = const_cast<double*>(B_nm);
  } else {
    P->own_B = true;
    TRY(dmalloc(P, &P->d_B_ia, sizeof(double) * nB));
    TRY(dmalloc(P, &P->d_B_nm, sizeof(double) * nBn));
    CK(cudaMemcpyAsync(P->d_B_ia, B_ia, sizeof(double) * nB, kind, P->stream));
    CK(cudaMemcpyAsync(P->d_B_nm, B_nm, sizeof(double) * nBn, kind, P->stream));
  }
  if (cfg->precision == GW_PREC_MIXED) {
    // FP32 B_ia with rows padded to 16 bytes (the fused Pi kernel reads it by TMA)
    P->ld_f = gw::pf_ldw(P->n_ov);
    TRY(dmalloc(P, &P->d_B_ia_f, sizeof(float) * (size_t)n * P->ld_f));
    TRY(dmalloc(P, &P->d_B_nm_f, sizeof(float) * nBn));
    LAUNCH((convert_rows_kernel<<<dim3(64, std::min(n, 65535)), 256, 0, P->stream>>>(P->d_B_ia, n, P->n_ov,
                                                                                   P->d_B_ia_f, P->ld_f)));
    LAUNCH((convert_f64_f32_kernel<<<1024, 256, 0, P->stream>>>(P->d_B_nm, P->d_B_nm_f, nBn)));
    const size_t nsplit = (size_t)n * gw::tc_ld(P->n_ov);
    TRY(dmalloc(P, &P->d_Bhi, sizeof(__nv_bfloat16) * nsplit));
    TRY(dmalloc(P, &P->d_Blo, sizeof(__nv_bfloat16) * nsplit));
    CK(gw::tc_split_rows(P->d_B_ia_f, n, P->n_ov, (int)P->ld_f, P->d_Bhi, P->d_Blo, P->stream));
    const size_t npanel = (size_t)n * gw::tc_pi_panel_cols(P->n_ov);
    TRY(dmalloc(P, &P->d_Bp_hi, sizeof(__nv_bfloat16) * npanel));
    TRY(dmalloc(P, &P->d_Bp_lo, sizeof(__nv_bfloat16) * npanel));
    CK(gw::tc_pi_panel_split(P->d_B_ia_f, P->ld_f, n, P->n_ov, P->d_Bp_hi, P->d_Bp_lo, P->stream));
    const size_t nsplitN = (size_t)n_targets * P->n_bas * gw::tc_ld(n);
    TRY(dmalloc(P, &P->d_Bnhi, sizeof(__nv_bfloat16) * nsplitN));
    TRY(dmalloc(P, &P->d_Bnlo, sizeof(__nv_bfloat16) * nsplitN));
    TRY(dmalloc(P, &P->d_Bnlo2, sizeof(__nv_bfloat16) * nsplitN));
    CK(gw::tc_split_rows(P->d_B_nm_f, n_targets * P->n_bas, n, n, P->d_Bnhi, P->d_Bnlo, P->stream, P->d_Bnlo2));
    const size_t nsplitT = (size_t)P->n_ov * gw::tc_ld(n);
    TRY(dmalloc(P, &P->d_BThi, sizeof(__nv_bfloat16) * nsplitT));
    TRY(dmalloc(P, &P->d_BTlo, sizeof(__nv_bfloat16) * nsplitT));
    CK(gw::tc_transpose_split(P->d_B_ia_f, n, P->n_ov, P->d_BThi, P->d_BTlo, P->stream, nullptr, P->ld_f));
    TRY(dmalloc(P, &P->d_Dsort, sizeof(double) * P->n_ov));
    TRY(dmalloc(P, &P->d_Dkidx, sizeof(int) * P->n_ov));
    CK(cudaStreamSynchronize(P->stream));
  }
  TRY(set_pair_energies(P, P->h_eps_s[0].data(), P->h_eps_s[1].data()));
  LAUNCH(gw::launch_sigma_x(P->d_B_nm, n_targets, P->n_bas, n, cfg->n_occ, P->d_sx, P->stream, P->d_occ_t));
  P->h_sx.resize(n_targets);
  CK(cudaMemcpyAsync(P->h_sx.data(), P->d_sx, sizeof(double) * n_targets, cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  P->h_shift.resize(n_targets);
  P->h_en.resize(n_targets);
  for (int t = 0; t < n_targets; ++t) {
    P->h_shift[t] = vxc ? P->h_sx[t] - vxc[t] : 0.0;
    P->h_en[t] = P->h_eps_s[P->h_spin[t]][targets[t]];
  }
  CK(cudaMemcpyAsync(P->d_shift, P->h_shift.data(), sizeof(double) * n_targets, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->d_en, P->h_en.data(), sizeof(double) * n_targets, cudaMemcpyHostToDevice, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  return GW_OK;
}

gw_status gw_plan_create(const gw_config* cfg, const double* eps, const double* B_ia, const double* B_nm,
                         const int* targets, int n_targets, const double* vxc, const double* xi, const double* wt,
                         unsigned flags, void* stream, gw_plan_t* out) {
  gw_plan* P = nullptr;
  if (!out) return fail(nullptr, GW_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!cfg || !eps || !B_ia || !B_nm || !targets) return fail(nullptr, GW_ERR_ARG, "NULL input pointer");
  if (cfg->n_occ <= 0 || cfg->n_virt <= 0 || cfg->n_aux <= 0 || n_targets <= 0 || cfg->n_freq <= 0)
    return fail(nullptr, GW_ERR_ARG, "sizes must be positive (n_occ %d n_virt %d n_aux %d n_targets %d n_freq %d)",
                cfg->n_occ, cfg->n_virt, cfg->n_aux, n_targets, cfg->n_freq);
  if ((long)cfg->n_occ * cfg->n_virt > 2147483647L) return fail(nullptr, GW_ERR_ARG, "n_occ*n_virt too large");
  if (cfg->precision != GW_PREC_FP64 && cfg->precision != GW_PREC_MIXED)
    return fail(nullptr, GW_ERR_ARG, "unknown precision %d", cfg->precision);
  if ((xi == nullptr) != (wt == nullptr)) return fail(nullptr, GW_ERR_ARG, "xi and wt must both be given or both NULL");
  if (!(cfg->x0 > 0.0) && !xi) return fail(nullptr, GW_ERR_ARG, "x0 must be positive");
  if (!(cfg->eta >= 0.0)) return fail(nullptr, GW_ERR_ARG, "eta must be >= 0");
  if (cfg->minres_maxit < 0 || cfg->qp_maxit <= 0) return fail(nullptr, GW_ERR_ARG, "bad iteration caps");
  if (cfg->tc_max_ctas < 0) return fail(nullptr, GW_ERR_ARG, "tc_max_ctas must be >= 0");
  if (!(cfg->qp_window > 0.0) || cfg->qp_window_points < 2 || !(cfg->qp_cluster_gap >= 0.0))
    return fail(nullptr, GW_ERR_ARG, "bad graphical window (%g Ha, %d points) or cluster gap %g", cfg->qp_window,
                cfg->qp_window_points, cfg->qp_cluster_gap);
  if (cfg->pi_ksplit != 0 && cfg->pi_ksplit != 1 && cfg->pi_ksplit != 2 && cfg->pi_ksplit != 4 && cfg->pi_ksplit != 8)
    return fail(nullptr, GW_ERR_ARG, "pi_ksplit must be 0 (autotune), 1, 2, 4 or 8 (got %d)", cfg->pi_ksplit);
  if (cfg->op_parts != 2 && cfg->op_parts != 3)
    return fail(nullptr, GW_ERR_ARG, "op_parts must be 2 or 3 (got %d)", cfg->op_parts);
  const int n_bas = cfg->n_occ + cfg->n_virt;
  for (int i = 0; i < n_bas; ++i) {
    if (!std::isfinite(eps[i])) return fail(nullptr, GW_ERR_ARG, "eps[%d] is not finite", i);
    if (i > 0 && eps[i] < eps[i - 1]) return fail(nullptr, GW_ERR_ARG, "eps must be ascending (index %d)", i);
  }
  if (eps[cfg->n_occ] <= eps[cfg->n_occ - 1]) return fail(nullptr, GW_ERR_ARG, "no gap between HOMO and LUMO");
  for (int t = 0; t < n_targets; ++t)
    if (targets[t] < 0 || targets[t] >= n_bas) return fail(nullptr, GW_ERR_ARG, "target %d out of range", targets[t]);
  if ((flags & GW_BORROW_DEVICE_PTRS) && cfg->precision == GW_PREC_MIXED) {
    // the FP32 copies are made from the borrowed FP64 arrays; fine
  }
  P = new (std::nothrow) gw_plan();
  if (!P) return fail(nullptr, GW_ERR_OOM, "host allocation failed");
  gw_status st = plan_create_impl(P, cfg, eps, B_ia, B_nm, targets, n_targets, vxc, xi, wt, flags, stream);
  if (st != GW_OK) {
    g_create_error = P->err;
    free_plan(P);
    return st;
  }
  *out = P;
  return GW_OK;
}

gw_status gw_plan_create_uks(const gw_config* cfg, const double* eps_a, const double* eps_b, int n_occ_b,
                             const double* B_ia_a, const double* B_ia_b, const double* B_nm, const int* targets,
                             const int* spins, int n_targets, const double* vxc, const double* xi, const double* wt,
                             unsigned flags, void* stream, gw_plan_t* out) {
  if (!out) return fail(nullptr, GW_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!cfg || !eps_a || !eps_b || !B_ia_a || !B_nm || !targets || !spins)
    return fail(nullptr, GW_ERR_ARG, "NULL input pointer");
  if (flags & GW_BORROW_DEVICE_PTRS) return fail(nullptr, GW_ERR_ARG, "open shell: B cannot be borrowed");
  const int n_bas = cfg->n_occ + cfg->n_virt;
  if (cfg->n_occ <= 0 || cfg->n_virt <= 0 || n_occ_b < 0 || n_occ_b >= n_bas || cfg->n_aux <= 0 || n_targets <= 0 ||
      cfg->n_freq <= 0)
    return fail(nullptr, GW_ERR_ARG, "bad sizes (n_occ %d/%d n_bas %d n_aux %d n_targets %d)", cfg->n_occ, n_occ_b,
                n_bas, cfg->n_aux, n_targets);
  if (n_occ_b > 0 && !B_ia_b) return fail(nullptr, GW_ERR_ARG, "B_ia_b is NULL");
  if ((long)cfg->n_occ * cfg->n_virt + (long)n_occ_b * (n_bas - n_occ_b) > 2147483647L)
    return fail(nullptr, GW_ERR_ARG, "too many pairs");
  if (cfg->precision != GW_PREC_FP64 && cfg->precision != GW_PREC_MIXED)
    return fail(nullptr, GW_ERR_ARG, "unknown precision %d", cfg->precision);
  if ((xi == nullptr) != (wt == nullptr)) return fail(nullptr, GW_ERR_ARG, "xi and wt must both be given or both NULL");
  if (!(cfg->x0 > 0.0) && !xi) return fail(nullptr, GW_ERR_ARG, "x0 must be positive");
  if (!(cfg->eta >= 0.0) || cfg->minres_maxit < 0 || cfg->qp_maxit <= 0 || (cfg->op_parts != 2 && cfg->op_parts != 3))
    return fail(nullptr, GW_ERR_ARG, "bad solver settings");
  const double* e2[2] = {eps_a, eps_b};
  const int occ[2] = {cfg->n_occ, n_occ_b};
  for (int sp = 0; sp < 2; ++sp) {
    for (int i = 0; i < n_bas; ++i) {
      if (!std::isfinite(e2[sp][i])) return fail(nullptr, GW_ERR_ARG, "spin %d: eps[%d] is not finite", sp, i);
      if (i > 0 && e2[sp][i] < e2[sp][i - 1]) return fail(nullptr, GW_ERR_ARG, "spin %d: eps not ascending", sp);
    }
    if (occ[sp] > 0 && e2[sp][occ[sp]] <= e2[sp][occ[sp] - 1])
      return fail(nullptr, GW_ERR_ARG, "spin %d: no gap between HOMO and LUMO", sp);
  }
  for (int t = 0; t < n_targets; ++t) {
    if (targets[t] < 0 || targets[t] >= n_bas) return fail(nullptr, GW_ERR_ARG, "target %d out of range", targets[t]);
    if (spins[t] != 0 && spins[t] != 1) return fail(nullptr, GW_ERR_ARG, "spin of target %d must be 0 or 1", t);
  }
  gw_plan* P = new (std::nothrow) gw_plan();
  if (!P) return fail(nullptr, GW_ERR_OOM, "host allocation failed");
  const UksInput uks{eps_b, n_occ_b, B_ia_b, spins};
  gw_status st = plan_create_impl(P, cfg, eps_a, B_ia_a, B_nm, targets, n_targets, vxc, xi, wt, flags, stream, &uks);
  if (st != GW_OK) {
    g_create_error = P->err;
    free_plan(P);
    return st;
  }
  *out = P;
  return GW_OK;
}

gw_status gw_polarizability(gw_plan_t P, const double* xi, int n_xi, double* pi_out) {
  if (!P) return GW_ERR_ARG;
  if (!xi) {
    if (pi_out) return fail(P, GW_ERR_ARG, "pi_out must be NULL when building the plan grid");
    P->screening_done = false;    // explicit request: rebuild the table
    return ensure_screening(P);
  }
  if (n_xi <= 0) return fail(P, GW_ERR_ARG, "n_xi must be positive");
  const int n = P->cfg.n_aux;
  CK(cudaEventRecord(P->ev0, P->stream));
  if (P->cfg.precision == GW_PREC_MIXED) {
    TRY(ensure(P, P->ws_mat, sizeof(float) * (size_t)n * n * n_xi));
    std::vector<int> kinds(n_xi, 0);
    TRY(tc_weighted_syrk(P, kinds.data(), xi, n_xi, 0, 0, as<float>(P->ws_mat), 0));
    CK(cudaEventRecord(P->ev1, P->stream));
    if (pi_out) {
      std::vector<float> h((size_t)n * n * n_xi);
      CK(cudaMemcpyAsync(h.data(), P->ws_mat.p, sizeof(float) * h.size(), cudaMemcpyDeviceToHost, P->stream));
      CK(cudaStreamSynchronize(P->stream));
      for (size_t i = 0; i < h.size(); ++i) pi_out[i] = h[i];
    }
  } else {
    TRY(ensure(P, P->ws_mat, sizeof(double) * (size_t)n * n * n_xi));
    std::vector<int> kinds(n_xi, 0);
    TRY(oz_weighted_syrk(P, kinds.data(), xi, n_xi, 0, 0, as<double>(P->ws_mat), /*checked=*/true));
    CK(cudaEventRecord(P->ev1, P->stream));
    if (pi_out)
      CK(cudaMemcpyAsync(pi_out, P->ws_mat.p, sizeof(double) * (size_t)n * n * n_xi, cudaMemcpyDeviceToHost,
                         P->stream));
    TRY(oz_check(P));
  }
  CK(cudaStreamSynchronize(P->stream));
  P->stats.ms_pi = now_ms(P, P->ev0, P->ev1);
  resolve_marks(P);
  return GW_OK;
}

gw_status gw_sigma_cd(gw_plan_t P, const double* omega, double* sigma_c, double* dsigma_c, double* sigma_x) {
  if (!P || !omega) return P ? fail(P, GW_ERR_ARG, "omega is NULL") : GW_ERR_ARG;
  TRY(ensure_screening(P));
  const int n_t = P->n_t;
  std::vector<double> om(omega, omega + n_t);
  std::vector<unsigned char> act(n_t, 1);
  int nf = 0;
  TRY(sigma_eval(P, om, act, &nf));
  std::vector<double> R(n_t), dR(n_t), I(n_t), dI(n_t);
  CK(cudaMemcpy(R.data(), P->sg_R.p, sizeof(double) * n_t, cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(dR.data(), P->sg_dR.p, sizeof(double) * n_t, cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(I.data(), P->sg_I.p, sizeof(double) * n_t, cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(dI.data(), P->sg_dI.p, sizeof(double) * n_t, cudaMemcpyDeviceToHost));
  for (int t = 0; t < n_t; ++t) {
    if (sigma_c) sigma_c[t] = R[t] - I[t];
    if (dsigma_c) dsigma_c[t] = dR[t] - dI[t];
    if (sigma_x) sigma_x[t] = P->h_sx[t];
  }
  return GW_OK;
}

// Spectral decomposition (Sec. 2.2, 3.2): the Hermitian Casida matrix M = D^1/2 (D + 4K) D^1/2 (K = B^T B over the
// pairs of every spin channel side by side; an open-shell plan stores each channel scaled by 1/sqrt 2, which turns
// the factor 4 into the 2 of each spin block) diagonalised by cyclic Jacobi sweeps in FP64 until the off-diagonal
// Frobenius norm is below 1e-13 of the diagonal one, then Omega_s and the pole weights of every (target, state).
constexpr long kSdMaxPairs = 16384;       // O(N_ov^3) work and 2 N_ov^2 doubles of storage

// One N_ov x N_ov FP64 product C = X Y^T by digits, in buffers sd_direct has sized; Yt: Y given transposed (C = X Yt).
gw_status sd_product(gw_plan* P, const double* X, const double* Y, const double* Yt, double* C) {
  const int N = P->n_ov;
  double* sa = as<double>(P->oz_sc);
  double* sb = sa + N;
  __nv_bfloat16* da = as<__nv_bfloat16>(P->oz_A);
  __nv_bfloat16* db = as<__nv_bfloat16>(P->oz_B);
  CK(gw::oz_row_digits(X, N, N, N, sa, da, P->stream));
  if (Yt) {
    CK(gw::oz_col_scale(Yt, N, N, N, sb, P->stream));
    CK(gw::oz_split_transpose(Yt, N, N, N, sb, db, P->stream));
  } else if (Y == X) {
    db = da;
    sb = sa;
  } else {
    CK(gw::oz_row_digits(Y, N, N, N, sb, db, P->stream));
  }
  gw::OzEpi ep{};
  ep.kind = gw::OZ_EPI_STORE;
  ep.out = C;
  ep.ldo = N;
  CK(gw::oz_gemm(gw::OzOperand{da, sa, 0}, gw::OzOperand{db, sb, 0}, 1, N, N, N, ep, as<int>(P->tc_err), P->stream));
  P->stats.n_kernel_launches += 3;
  return GW_OK;
}

// Memory of the diagonalisation: the direct route's matrices and digits, and (all) the Casida matrix and eigenvectors.
void sd_release(gw_plan* P, bool all) {
  for (DevBuf& b : P->sd_x) release(P, b);
  for (DevBuf* b : {&P->oz_A, &P->oz_B}) release(P, *b);
  if (all)
    for (DevBuf* b : {&P->sd_M, &P->sd_T, &P->sd_V}) release(P, *b);
}

// Eigenvectors of the Casida matrix by tridiagonalisation and refinement on digit products (kernels_sd.cu); *ok is 0
// where the off-diagonal criterion of the Jacobi sweeps is not met (they then start from the matrix in sd_M).
gw_status sd_direct(gw_plan* P, int Np, bool* ok) {
  *ok = false;
  const int N = P->n_ov, n = P->cfg.n_aux, R = P->n_t * P->n_bas;
  const size_t nn = sizeof(double) * (size_t)N * N;
  TRY(ensure(P, P->tc_err, sizeof(int)));
  // everything up front: where the digits (16 N max(N, n) bytes twice) and the five matrices do not fit, the sweeps run
  // in the memory they have
  const size_t dg_bytes = sizeof(__nv_bfloat16) * std::max(gw::oz_elems(N, N), gw::oz_elems(n, N));
  gw_status fit = GW_OK;
  for (int i = 0; i < 5 && fit == GW_OK; ++i) fit = ensure(P, P->sd_x[i], nn);
  if (fit == GW_OK) fit = ensure(P, P->sd_vec, sizeof(double) * (9 * (size_t)N + 8));
  if (fit == GW_OK) fit = ensure(P, P->oz_A, dg_bytes);
  if (fit == GW_OK) fit = ensure(P, P->oz_B, dg_bytes);
  if (fit == GW_OK) fit = ensure(P, P->oz_sc, sizeof(double) * ((size_t)std::max(N, n) + N));
  if (fit != GW_OK) {
    (void)cudaGetLastError();
    sd_release(P, false);
    return GW_OK;
  }
  CK(cudaMemsetAsync(P->tc_err.p, 0, sizeof(int), P->stream));
  double* M = as<double>(P->sd_x[0]);      // the matrix, row length N
  double* A = as<double>(P->sd_x[1]);      // its working copy; then pivots, S
  double* H = as<double>(P->sd_x[2]);      // reflectors; then G, C
  double* W = as<double>(P->sd_x[3]);      // pivots; then M V^T
  double* V = as<double>(P->sd_x[4]);      // eigenvectors, rows
  double* vec = as<double>(P->sd_vec);
  double *dg = vec, *eg = vec + N, *beta = vec + 2 * (size_t)N, *lam = vec + 3 * (size_t)N, *nrm = vec + 4 * (size_t)N,
         *pb = vec + 5 * (size_t)N, *norms = vec + 9 * (size_t)N;
  unsigned* bar = reinterpret_cast<unsigned*>(norms + 4);
  CK(gw::sd_pack_rows(as<double>(P->sd_M), N, N, Np, M, P->stream));
  CK(cudaMemcpyAsync(A, M, nn, cudaMemcpyDeviceToDevice, P->stream));
  const cudaError_t coop = gw::sd_tridiagonal(A, N, N, H, beta, dg, eg, pb, bar, as<int>(P->tc_err), P->stream);
  if (coop == cudaErrorCooperativeLaunchTooLarge || coop == cudaErrorNotSupported || coop == cudaErrorLaunchOutOfResources) {
    (void)cudaGetLastError();                       // a context with fewer SMs than the device: the sweeps need no grid barrier
    return GW_OK;
  }
  CK(coop);
  CK(gw::sd_tridiagonal_vectors(dg, eg, N, lam, A, W, N, H, beta, N, nrm, V, P->stream));
  P->stats.n_kernel_launches += 5;
  double h[3];
  for (int it = 0; it < 5; ++it) {
    TRY(sd_product(P, V, V, nullptr, H));              // G
    TRY(sd_product(P, V, M, nullptr, W));              // V M (M is symmetric)
    TRY(sd_product(P, W, V, nullptr, A));              // S
    CK(gw::sd_eig_norms(A, H, N, norms, P->stream));
    CK(cudaMemcpyAsync(h, norms, sizeof(h), cudaMemcpyDeviceToHost, P->stream));
    int herr = 0;
    CK(cudaMemcpyAsync(&herr, P->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    if (herr != 0) return GW_OK;                    // a bounded wait ran out: the sweeps have none
    if (!std::isfinite(h[0] + h[1] + h[2]) || h[2] > 0.01) return GW_OK;     // not a basis
    // S is as diagonal as the sweeps leave it and the rows are orthonormal to the same level
    if (it > 0 && h[0] <= 1e-26 * h[1] && h[2] <= 1e-26 * N) {
      *ok = true;
      break;
    }
    CK(gw::sd_eig_update(A, H, N, W, norms, P->stream));
    TRY(sd_product(P, W, nullptr, V, A));              // next rows
    std::swap(V, A);
    P->stats.n_kernel_launches += 2;
  }
  if (!*ok) return GW_OK;
  // V_aux = 2 B D^1/2 T and the pole weights
  double* sA = as<double>(P->oz_sc);
  double* sV = sA + n;
  CK(gw::sd_twice_sqrt(P->d_D, N, dg, P->stream));
  CK(gw::oz_split_weighted(P->d_B_ia, n, 0, N, N, dg, nullptr, N, 1, as<__nv_bfloat16>(P->oz_A), sA, nullptr, nullptr,
                           P->stream));
  CK(gw::oz_row_digits(V, N, N, N, sV, as<__nv_bfloat16>(P->oz_B), P->stream));
  gw::OzEpi ep{};
  ep.kind = gw::OZ_EPI_STORE;
  ep.out = as<double>(P->sd_V);
  ep.ldo = N;
  CK(gw::oz_gemm(gw::OzOperand{as<__nv_bfloat16>(P->oz_A), sA, 0}, gw::OzOperand{as<__nv_bfloat16>(P->oz_B), sV, 0}, 1, n,
                 N, N, ep, as<int>(P->tc_err), P->stream));
  CK(gw::sd_rows_weights(A, H, as<double>(P->sd_V), P->d_B_nm, n, N, R, as<double>(P->sd_Om), as<double>(P->sd_w2),
                         P->stream));
  P->stats.n_kernel_launches += 6;
  return oz_check(P);
}

gw_status ensure_sd(gw_plan* P) {
  if (P->sd_done) return GW_OK;
  const long N = P->n_ov;
  if (N > kSdMaxPairs)
    return fail(P, GW_ERR_ARG, "spectral decomposition needs N_ov <= %ld (got %ld): O(N_ov^3)", kSdMaxPairs, N);
  const int n = P->cfg.n_aux, Np = (int)(N + (N & 1));
  TRY(ensure(P, P->sd_M, sizeof(double) * (size_t)Np * Np));
  TRY(ensure(P, P->sd_T, sizeof(double) * (size_t)Np * Np));
  TRY(ensure(P, P->sd_cs, sizeof(double) * (size_t)Np));
  TRY(ensure(P, P->sd_off, sizeof(double) * 2));
  TRY(ensure(P, P->sd_Om, sizeof(double) * (size_t)N));
  TRY(ensure(P, P->sd_V, sizeof(double) * (size_t)n * N));
  const int R = P->n_t * P->n_bas;
  TRY(ensure(P, P->sd_w2, sizeof(double) * (size_t)R * N));
  LAUNCH(CK(gw::sd_casida_matrix(P->d_B_ia, P->d_D, n, (int)N, Np, as<double>(P->sd_M), as<double>(P->sd_T),
                                 P->stream)));
  if (N >= 8 && N <= gw::sd_direct_max()) {
    bool ok = false;
    TRY(sd_direct(P, Np, &ok));
    sd_release(P, ok);                             // the stream is synchronised
    if (ok) {
      P->sd_sweeps = 0;
      P->sd_done = true;
      return GW_OK;
    }
  }
  double off[2] = {1.0, 1.0};
  int sweeps = 0;
  for (; sweeps < 40; ++sweeps) {
    CK(gw::sd_offdiag(as<double>(P->sd_M), Np, as<double>(P->sd_off), P->stream));
    CK(cudaMemcpyAsync(off, P->sd_off.p, sizeof(off), cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    if (!(off[0] > 1e-26 * off[1])) break;
    CK(gw::sd_jacobi_sweep(as<double>(P->sd_M), as<double>(P->sd_T), Np, as<double>(P->sd_cs), P->stream));
    P->stats.n_kernel_launches += 4 * (Np - 1) + 1;
  }
  if (!(off[0] <= 1e-26 * off[1]))
    return fail(P, GW_ERR_NOT_CONVERGED, "Jacobi sweeps of the Casida matrix did not converge (off/diag %g)",
                std::sqrt(off[0] / off[1]));
  LAUNCH(CK(gw::sd_weights(P->d_B_ia, P->d_D, as<double>(P->sd_M), as<double>(P->sd_T), P->d_B_nm, n, (int)N, Np, R,
                           as<double>(P->sd_Om), as<double>(P->sd_V), as<double>(P->sd_w2), P->stream)));
  CK(cudaStreamSynchronize(P->stream));
  sd_release(P, true);
  P->sd_sweeps = sweeps;
  P->sd_done = true;
  return GW_OK;
}

gw_status gw_sigma_sd(gw_plan_t P, int n_points, const int* target_idx, const double* omega, double* sigma_c,
                      double* dsigma_c) {
  if (!P) return GW_ERR_ARG;
  if (n_points < 0 || (n_points > 0 && !omega)) return fail(P, GW_ERR_ARG, "bad point list");
  if (n_points == 0) return GW_OK;
  std::vector<int> tmap(n_points);
  for (int p = 0; p < n_points; ++p) {
    tmap[p] = target_idx ? target_idx[p] : p;
    if (tmap[p] < 0 || tmap[p] >= P->n_t) return fail(P, GW_ERR_ARG, "target_idx[%d] out of range", p);
    if (!std::isfinite(omega[p])) return fail(P, GW_ERR_ARG, "omega[%d] not finite", p);
  }
  if (!target_idx && n_points != P->n_t) return fail(P, GW_ERR_ARG, "without target_idx, n_points = n_targets");
  TRY(ensure_sd(P));
  TRY(ensure(P, P->sd_tmap, sizeof(int) * n_points));
  TRY(ensure(P, P->sd_om, sizeof(double) * n_points));
  TRY(ensure(P, P->sd_S, sizeof(double) * n_points));
  TRY(ensure(P, P->sd_dS, sizeof(double) * n_points));
  TRY(ensure(P, P->sd_part, sizeof(double) * 2 * (size_t)n_points * gw::sd_sigma_parts(P->n_bas, P->n_ov)));
  CK(cudaMemcpyAsync(P->sd_tmap.p, tmap.data(), sizeof(int) * n_points, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->sd_om.p, omega, sizeof(double) * n_points, cudaMemcpyHostToDevice, P->stream));
  LAUNCH(CK(gw::sd_sigma(as<double>(P->sd_w2), as<double>(P->sd_Om), (int)P->n_ov, P->n_bas, P->d_eps_g,
                         as<int>(P->sd_tmap), P->d_spin, P->d_occ_t, P->cfg.n_occ, as<double>(P->sd_om), n_points,
                         P->cfg.eta, as<double>(P->sd_part), as<double>(P->sd_S), as<double>(P->sd_dS), P->stream)));
  std::vector<double> S(n_points), dS(n_points);
  CK(cudaMemcpyAsync(S.data(), P->sd_S.p, sizeof(double) * n_points, cudaMemcpyDeviceToHost, P->stream));
  CK(cudaMemcpyAsync(dS.data(), P->sd_dS.p, sizeof(double) * n_points, cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  for (int p = 0; p < n_points; ++p) {
    if (sigma_c) sigma_c[p] = S[p];
    if (dsigma_c) dsigma_c[p] = dS[p];
  }
  return GW_OK;
}

gw_status gw_sigma_points(gw_plan_t P, int n_points, const int* target_idx, const double* omega, double* sigma_c,
                          double* dsigma_c) {
  if (!P) return GW_ERR_ARG;
  if (n_points < 0 || (n_points > 0 && (!target_idx || !omega))) return fail(P, GW_ERR_ARG, "bad point list");
  if (n_points == 0) return GW_OK;
  for (int p = 0; p < n_points; ++p) {
    if (target_idx[p] < 0 || target_idx[p] >= P->n_t) return fail(P, GW_ERR_ARG, "target_idx[%d] out of range", p);
    if (!std::isfinite(omega[p])) return fail(P, GW_ERR_ARG, "omega[%d] not finite", p);
  }
  TRY(ensure_screening(P));
  std::vector<double> om(omega, omega + n_points);
  std::vector<int> tmap(target_idx, target_idx + n_points);
  std::vector<unsigned char> act(n_points, 1);
  int nf = 0;
  TRY(sigma_eval(P, om, act, &nf, &tmap));
  std::vector<double> R(n_points), dR(n_points), I(n_points), dI(n_points);
  CK(cudaMemcpy(R.data(), P->sg_R.p, sizeof(double) * n_points, cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(dR.data(), P->sg_dR.p, sizeof(double) * n_points, cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(I.data(), P->sg_I.p, sizeof(double) * n_points, cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(dI.data(), P->sg_dI.p, sizeof(double) * n_points, cudaMemcpyDeviceToHost));
  for (int p = 0; p < n_points; ++p) {
    if (sigma_c) sigma_c[p] = R[p] - I[p];
    if (dsigma_c) dsigma_c[p] = dR[p] - dI[p];
  }
  return GW_OK;
}

gw_status gw_residues_minres(gw_plan_t P, int n_rhs, const int* target_idx, const int* m, const double* x,
                             double* w_re, double* w_im, double* dw_re, int* iters, double* resnorm,
                             int* used_fallback) {
  if (!P) return GW_ERR_ARG;
  if (n_rhs < 0 || (n_rhs > 0 && (!target_idx || !m || !x))) return fail(P, GW_ERR_ARG, "bad right-hand side list");
  if (n_rhs == 0) return GW_OK;
  for (int j = 0; j < n_rhs; ++j) {
    if (target_idx[j] < 0 || target_idx[j] >= P->n_t) return fail(P, GW_ERR_ARG, "target_idx[%d] out of range", j);
    if (m[j] < 0 || m[j] >= P->n_bas) return fail(P, GW_ERR_ARG, "m[%d] out of range", j);
    if (!std::isfinite(x[j])) return fail(P, GW_ERR_ARG, "x[%d] not finite", j);
  }
  TRY(ensure(P, P->mr_rt, sizeof(int) * n_rhs));
  TRY(ensure(P, P->mr_rm, sizeof(int) * n_rhs));
  TRY(ensure(P, P->mr_xf, sizeof(double) * n_rhs));
  TRY(ensure(P, P->mr_wre, sizeof(double) * n_rhs));
  TRY(ensure(P, P->mr_wim, sizeof(double) * n_rhs));
  TRY(ensure(P, P->mr_dwre, sizeof(double) * n_rhs));
  TRY(ensure(P, P->mr_it, sizeof(int) * n_rhs));
  TRY(ensure(P, P->mr_res, sizeof(double) * n_rhs));
  CK(cudaMemcpyAsync(P->mr_rt.p, target_idx, sizeof(int) * n_rhs, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->mr_rm.p, m, sizeof(int) * n_rhs, cudaMemcpyHostToDevice, P->stream));
  CK(cudaMemcpyAsync(P->mr_xf.p, x, sizeof(double) * n_rhs, cudaMemcpyHostToDevice, P->stream));
  std::vector<int> fb(n_rhs, 0);
  TRY(residues(P, n_rhs, as<int>(P->mr_rt), as<int>(P->mr_rm), as<double>(P->mr_xf), as<double>(P->mr_wre),
               as<double>(P->mr_wim), as<double>(P->mr_dwre), as<int>(P->mr_it), as<double>(P->mr_res), fb.data()));
  if (w_re) CK(cudaMemcpy(w_re, P->mr_wre.p, sizeof(double) * n_rhs, cudaMemcpyDeviceToHost));
  if (w_im) CK(cudaMemcpy(w_im, P->mr_wim.p, sizeof(double) * n_rhs, cudaMemcpyDeviceToHost));
  if (dw_re) CK(cudaMemcpy(dw_re, P->mr_dwre.p, sizeof(double) * n_rhs, cudaMemcpyDeviceToHost));
  if (iters) CK(cudaMemcpy(iters, P->mr_it.p, sizeof(int) * n_rhs, cudaMemcpyDeviceToHost));
  if (resnorm) CK(cudaMemcpy(resnorm, P->mr_res.p, sizeof(double) * n_rhs, cudaMemcpyDeviceToHost));
  if (used_fallback) std::memcpy(used_fallback, fb.data(), sizeof(int) * n_rhs);
  return GW_OK;
}

}  // extern "C"

namespace {

// QP loop (Sec. 3.4) for the targets with run[t] != 0, started at om0[t]: every running state's Sigma(omega) per
// evaluation (one batched residue solve for all of them), then one step of the linearised update or of the step
// tree.  Final states go to hs (states not run keep status 1 and om0); any_fb[t] is set when an evaluation of a
// running state used the dense fallback.
gw_status qp_loop(gw_plan* P, int lin, const std::vector<double>& om0, const std::vector<unsigned char>& run,
                  std::vector<QPState>& hs, std::vector<int>& any_fb) {
  const int n_t = P->n_t;
  TRY(ensure(P, P->qp_st, sizeof(QPState) * n_t));
  hs.assign(n_t, QPState{});
  for (int t = 0; t < n_t; ++t) {
    hs[t].omega = om0[t];
    hs[t].Z = 1.0;
    hs[t].status = run[t] ? 0 : 1;
  }
  CK(cudaMemcpyAsync(P->qp_st.p, hs.data(), sizeof(QPState) * n_t, cudaMemcpyHostToDevice, P->stream));
  std::vector<double> om(n_t);
  std::vector<unsigned char> act(n_t);
  const int maxit = lin ? 1 : P->cfg.qp_maxit;
  for (int it = 0; it < maxit; ++it) {
    CK(cudaMemcpyAsync(hs.data(), P->qp_st.p, sizeof(QPState) * n_t, cudaMemcpyDeviceToHost, P->stream));
    CK(cudaStreamSynchronize(P->stream));
    int n_act = 0;
    for (int t = 0; t < n_t; ++t) {
      om[t] = hs[t].omega;
      act[t] = hs[t].status == 0 ? 1 : 0;
      n_act += act[t];
    }
    if (n_act == 0) break;
    int nf = 0;
    TRY(sigma_eval(P, om, act, &nf));
    if (nf > 0)
      for (int t = 0; t < n_t; ++t)
        if (act[t]) any_fb[t] = 1;   // conservative: flag the active states of an evaluation that fell back
    LAUNCH(gw::launch_qp_step(as<QPState>(P->qp_st), as<double>(P->sg_R), as<double>(P->sg_dR),
                              as<double>(P->sg_I), as<double>(P->sg_dI), P->d_en, P->d_shift, P->cfg.qp_tol,
                              P->cfg.qp_maxit, n_t, lin, P->stream));
  }
  CK(cudaMemcpyAsync(hs.data(), P->qp_st.p, sizeof(QPState) * n_t, cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  for (int t = 0; t < n_t; ++t)
    if (!run[t]) hs[t].omega = om0[t];
  return GW_OK;
}

// Graphical search (Sec. 3.4): f(w) = e_n + shift + Sigma_c(w) - w on qp_window_points evenly spaced points of
// [c_t - qp_window, c_t + qp_window] for every target with run[t], all points of all targets in one batched
// evaluation.  root[t] = the sign change of f with f decreasing (a root of the QP equation, not a pole of Sigma)
// closest to c_t, by linear interpolation; found[t] = 0 if the window holds none.
gw_status graphical_scan(gw_plan* P, const std::vector<double>& c, const std::vector<unsigned char>& run,
                         std::vector<double>& root, std::vector<unsigned char>& found, std::vector<int>& any_fb) {
  const int n_t = P->n_t, np = std::max(2, P->cfg.qp_window_points);
  const double hw = P->cfg.qp_window;
  std::vector<int> tmap;
  std::vector<double> om;
  for (int t = 0; t < n_t; ++t)
    if (run[t])
      for (int j = 0; j < np; ++j) {
        tmap.push_back(t);
        om.push_back(c[t] + hw * (-1.0 + 2.0 * j / (np - 1)));
      }
  root = c;
  found.assign(n_t, 0);
  if (om.empty()) return GW_OK;
  std::vector<unsigned char> act(om.size(), 1);
  int nf = 0;
  TRY(sigma_eval(P, om, act, &nf, &tmap));
  std::vector<double> R(om.size()), I(om.size());
  CK(cudaMemcpyAsync(R.data(), P->sg_R.p, sizeof(double) * om.size(), cudaMemcpyDeviceToHost, P->stream));
  CK(cudaMemcpyAsync(I.data(), P->sg_I.p, sizeof(double) * om.size(), cudaMemcpyDeviceToHost, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  for (size_t k = 0; k < om.size(); ++k) {
    const int t = tmap[k];
    if (nf > 0) any_fb[t] = 1;
    if (k + 1 >= om.size() || tmap[k + 1] != t) continue;
    const double f0 = P->h_en[t] + P->h_shift[t] + R[k] - I[k] - om[k];
    const double f1 = P->h_en[t] + P->h_shift[t] + R[k + 1] - I[k + 1] - om[k + 1];
    if ((f0 > 0.0 && f1 <= 0.0) || (f0 == 0.0 && f1 < 0.0)) {
      const double r = om[k] + (om[k + 1] - om[k]) * f0 / (f0 - f1);
      if (!found[t] || std::fabs(r - c[t]) < std::fabs(root[t] - c[t])) root[t] = r;
      found[t] = 1;
    }
  }
  return GW_OK;
}

// QP energies of the targets with run[t] from the starting points / window centres start[t]: linearised, step
// tree, or graphical search followed by the step tree from the root it found.
gw_status qp_solve_set(gw_plan* P, gw_qp_mode mode, const std::vector<double>& start,
                       const std::vector<unsigned char>& run, std::vector<QPState>& hs, std::vector<int>& any_fb,
                       std::vector<unsigned char>& no_root) {
  const int n_t = P->n_t;
  no_root.assign(n_t, 0);
  if (mode != GW_QP_GRAPHICAL) return qp_loop(P, mode == GW_QP_LINEARISED, start, run, hs, any_fb);
  std::vector<double> root;
  std::vector<unsigned char> found;
  TRY(graphical_scan(P, start, run, root, found, any_fb));
  std::vector<unsigned char> run2(n_t, 0);
  for (int t = 0; t < n_t; ++t) {
    run2[t] = run[t] && found[t];
    no_root[t] = run[t] && !found[t];
  }
  return qp_loop(P, 0, root, run2, hs, any_fb);
}

// QP equation of every target (Sec. 3.4), with the cluster layer when qp_cluster_gap > 0 (not in the linearised
// mode): targets whose KS energies are within qp_cluster_gap of a neighbour in energy form a cluster; the first
// member of each cluster (lowest KS energy) is solved first, then every other member starts from its KS energy
// shifted by that member's QP correction (the step tree's start, or the centre of the graphical window).
// omega0 (host [n_targets]) replaces the KS energies as starting points, or NULL.
gw_status qp_solve_impl(gw_plan* P, gw_qp_mode mode, const double* omega0, double* e_qp, double* z_factor,
                        int* state_status) {
  cudaEvent_t a, b;
  CK(cudaEventCreate(&a));
  CK(cudaEventCreate(&b));
  CK(cudaEventRecord(a, P->stream));
  TRY(ensure_screening(P));
  const int n_t = P->n_t;
  std::vector<double> start(n_t);
  for (int t = 0; t < n_t; ++t) start[t] = omega0 ? omega0[t] : P->h_en[t];
  std::vector<QPState> hs;
  std::vector<int> any_fb(n_t, 0);
  std::vector<unsigned char> no_root;
  const bool cluster = P->cfg.qp_cluster_gap > 0.0 && mode != GW_QP_LINEARISED;
  if (!cluster) {
    std::vector<unsigned char> run(n_t, 1);
    TRY(qp_solve_set(P, mode, start, run, hs, any_fb, no_root));
  } else {
    std::vector<int> order(n_t);
    for (int t = 0; t < n_t; ++t) order[t] = t;
    std::sort(order.begin(), order.end(), [&](int x, int y) { return P->h_en[x] < P->h_en[y]; });
    std::vector<int> rep(n_t);
    std::vector<unsigned char> first(n_t, 0), rest(n_t, 0);
    for (int k = 0; k < n_t; ++k) {
      const int t = order[k];
      if (k == 0 || P->h_en[t] - P->h_en[order[k - 1]] > P->cfg.qp_cluster_gap) {
        rep[t] = t;
        first[t] = 1;
      } else {
        rep[t] = rep[order[k - 1]];
        rest[t] = 1;
      }
    }
    std::vector<QPState> h1;
    std::vector<unsigned char> nr1;
    TRY(qp_solve_set(P, mode, start, first, h1, any_fb, nr1));
    std::vector<double> start2(start);
    for (int t = 0; t < n_t; ++t)
      if (rest[t] && h1[rep[t]].status == 1 && !nr1[rep[t]])
        start2[t] = start[t] + (h1[rep[t]].omega - P->h_en[rep[t]]);
    TRY(qp_solve_set(P, mode, start2, rest, hs, any_fb, no_root));
    for (int t = 0; t < n_t; ++t)
      if (first[t]) {
        hs[t] = h1[t];
        no_root[t] = nr1[t];
      }
  }
  CK(cudaEventRecord(b, P->stream));
  CK(cudaStreamSynchronize(P->stream));
  P->stats.ms_qp = now_ms(P, a, b);
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  bool all_ok = true;
  for (int t = 0; t < n_t; ++t) {
    const bool conv = hs[t].status == 1 && !no_root[t];
    if (e_qp) e_qp[t] = hs[t].omega;
    if (z_factor) z_factor[t] = no_root[t] ? NAN : hs[t].Z;
    if (!conv) all_ok = false;
    if (state_status) state_status[t] = conv ? (any_fb[t] ? 2 : 0) : 1;
  }
  return all_ok ? GW_OK : GW_ERR_NOT_CONVERGED;
}

// Energies of the next eigenvalue cycle, per spin: targets take their QP energies, every other occupied state moves
// by the correction of the highest occupied target of its spin, every other virtual state by that of the lowest
// virtual target of its spin.
std::vector<double> scissor(const gw_plan* P, int spin, const std::vector<double>& e_qp) {
  const int n_occ = P->occ_s[spin];
  const std::vector<double>& ks = P->h_eps_s[spin];
  std::vector<double> out(ks);
  double e_o = -INFINITY, d_o = 0.0, e_v = INFINITY, d_v = 0.0;
  for (int t = 0; t < P->n_t; ++t) {
    if (P->h_spin[t] != spin) continue;
    const int n = P->h_targets[t];
    const double e = ks[n], d = e_qp[t] - e;
    if (n < n_occ && (e > e_o || (e == e_o && d > d_o))) { e_o = e; d_o = d; }
    if (n >= n_occ && (e < e_v || (e == e_v && d < d_v))) { e_v = e; d_v = d; }
  }
  for (int m = 0; m < P->n_bas; ++m) out[m] += m < n_occ ? d_o : d_v;
  for (int t = 0; t < P->n_t; ++t)
    if (P->h_spin[t] == spin) out[P->h_targets[t]] = e_qp[t];
  return out;
}

}  // namespace

extern "C" {

gw_status gw_qp_solve(gw_plan_t P, gw_qp_mode mode, double* e_qp, double* z_factor, int* state_status) {
  if (!P) return GW_ERR_ARG;
  if (mode != GW_QP_LINEARISED && mode != GW_QP_STEPTREE && mode != GW_QP_GRAPHICAL)
    return fail(P, GW_ERR_ARG, "unknown QP mode %d", (int)mode);
  return qp_solve_impl(P, mode, nullptr, e_qp, z_factor, state_status);
}

gw_status gw_evgw(gw_plan_t P, int update_w, gw_qp_mode mode, int max_iter, double tol, double* e_qp,
                  double* z_factor, int* state_status, int* iterations) {
  if (!P) return GW_ERR_ARG;
  if (mode != GW_QP_LINEARISED && mode != GW_QP_STEPTREE && mode != GW_QP_GRAPHICAL)
    return fail(P, GW_ERR_ARG, "unknown QP mode %d", (int)mode);
  if (max_iter <= 0 || !(tol > 0.0)) return fail(P, GW_ERR_ARG, "max_iter must be positive and tol > 0");
  const int n_t = P->n_t;
  std::vector<double> prev(n_t), cur(n_t), z(n_t);
  std::vector<int> st(n_t);
  for (int t = 0; t < n_t; ++t) prev[t] = P->h_en[t];
  std::vector<double> eps_cur[2] = {P->h_eps_s[0], P->h_eps_s[1]};
  gw_status last = GW_OK;
  bool conv = false;
  int it = 0;
  for (it = 1; it <= max_iter; ++it) {
    for (int sp = 0; sp < P->n_spin; ++sp) TRY(set_g_energies(P, sp, eps_cur[sp].data()));
    if (update_w && it > 1) {            // evGW: W from the current energies (cycle 1 is G0W0)
      TRY(set_pair_energies(P, eps_cur[0].data(), eps_cur[1].data()));
      P->screening_done = false;
    }
    last = qp_solve_impl(P, mode, prev.data(), cur.data(), z.data(), st.data());
    if (last != GW_OK && last != GW_ERR_NOT_CONVERGED) break;
    double delta = 0.0;
    for (int t = 0; t < n_t; ++t) delta = std::max(delta, std::fabs(cur[t] - prev[t]));
    prev = cur;
    for (int sp = 0; sp < P->n_spin; ++sp) eps_cur[sp] = scissor(P, sp, cur);
    if (delta < tol) { conv = true; break; }
  }
  // the plan goes back to G0W0: G and W from the KS energies (W is rebuilt on the next call that needs it)
  gw_status rs = GW_OK;
  for (int sp = 0; sp < P->n_spin && rs == GW_OK; ++sp) rs = set_g_energies(P, sp, P->h_eps_s[sp].data());
  if (rs == GW_OK && update_w) {
    rs = set_pair_energies(P, P->h_eps_s[0].data(), P->h_eps_s[1].data());
    P->screening_done = false;
  }
  if (last != GW_OK && last != GW_ERR_NOT_CONVERGED) return last;
  if (rs != GW_OK) return rs;
  for (int t = 0; t < n_t; ++t) {
    if (e_qp) e_qp[t] = cur[t];
    if (z_factor) z_factor[t] = z[t];
    if (state_status) state_status[t] = st[t];
  }
  if (iterations) *iterations = std::min(it, max_iter);
  if (!conv) return fail(P, GW_ERR_NOT_CONVERGED, "eigenvalue cycles did not converge to %g Ha in %d", tol, max_iter);
  return last;
}

gw_status gw_shard_columns(int n_freq, int rank, int world, int* p0, int* p1) {
  if (n_freq <= 0 || world <= 0 || rank < 0 || rank >= world || !p0 || !p1) return GW_ERR_ARG;
  const long n = (long)n_freq + 1;
  *p0 = (int)(n * rank / world);
  *p1 = (int)(n * (rank + 1) / world);
  return GW_OK;
}

gw_status gw_set_shard(gw_plan_t P, int rank, int world, gw_allreduce_fn allreduce_sum, void* ctx) {
  if (!P) return GW_ERR_ARG;
  if (world < 1 || rank < 0 || rank >= world || (world > 1 && !allreduce_sum))
    return fail(P, GW_ERR_ARG, "bad shard (rank %d of %d)", rank, world);
  P->sh_rank = rank;
  P->sh_world = world;
  P->sh_reduce = world > 1 ? allreduce_sum : nullptr;
  P->sh_ctx = ctx;
  P->screening_done = false;
  return GW_OK;
}

gw_status gw_plan_footprint(const gw_config* c, int n_t, unsigned flags, unsigned long long* bytes) {
  if (!c || !bytes || c->n_occ <= 0 || c->n_virt <= 0 || c->n_aux <= 0 || c->n_freq <= 0 || n_t <= 0)
    return GW_ERR_ARG;
  // Mirrors the allocations of plan_create_impl and of every ensure() class below, each at its cap.
  typedef unsigned long long u64;
  const bool mixed = c->precision == GW_PREC_MIXED;
  const u64 n = c->n_aux, n_ov = (u64)c->n_occ * c->n_virt, n_bas = (u64)c->n_occ + c->n_virt;
  const u64 n_g1 = (u64)c->n_freq + 1, ts = mixed ? 4 : 8;
  const u64 ws = (u64)(c->workspace_mb > 0 ? c->workspace_mb : 8192) << 20;
  const u64 ldo = (u64)gw::tc_ld((int)std::min<u64>(n_ov, 2147483647ull)), ldn = (u64)gw::tc_ld(c->n_aux);
  const u64 rows = (u64)n_t * n_bas, nBn = rows * n;
  auto capped = [ws](u64 item, u64 want) { return std::max(item, std::min(ws / std::max<u64>(item, 1) * item, want)); };
  u64 b = 8 * (n_bas + 2 * n_g1 + 3 * (u64)n_t) + 8 * rows * n_g1;         // energies, grid, shifts, W table
  if (!(flags & GW_BORROW_DEVICE_PTRS)) b += 8 * (n * n_ov + nBn);           // B_ia, B_nm
  const u64 ldf = (u64)gw::pf_ldw((int)std::min<u64>(n_ov, 2147483647ull));
  if (mixed) {
    b += 4 * (n * ldf + nBn);                                                // FP32 copies
    b += 6 * (n * ldo + rows * ldn + n_ov * ldn);                             // three BF16 parts of B, B_nm, B^T
    b += 12 * n_ov;                                                          // sorted D and its pair index
    b += 4 * n * (u64)gw::tc_pi_panel_cols((int)std::min<u64>(n_ov, 2147483647ull));   // K-panel hi/lo of B
  }
  b += 8 * n_ov;                                                             // pair energies D_ia
  // imaginary-axis stage: frequency matrices, info/index lists
  b += capped(n * n * ts, n * n * ts * n_g1) + 24 * n_g1;
  if (mixed) {
    // weight table of one Pi launch: a screening chunk or two entries per fallback matrix
    const u64 nb = std::max<u64>(n_g1, 2 * std::max<u64>(1, ws / (2 * n * n * ts)));
    b += 4 * nb * ldf + 16 * nb;
    b += std::min(ws, 8 * nb * n * n * 4);                                     // split-K partials (small problems)
    const u64 per_ns = n * ldn * 24 + n * n * 8;                             // Newton-Schulz split/FP32 iterates
    b += capped(per_ns, per_ns * n_g1) + 6 * n * ldn + 4 * n_g1;             // + the split eps(0)^-1 - 1
    b += 8 * n * n_g1 + 16 * n_g1;                                           // spectrum-estimate vectors
    b += 8 * n_g1 * std::min<u64>(n_g1, 256);                                // matrix of the grid nodes
  } else {
    // digit products: B and its weighted copies, or the inverse factors, their digits and those of B_nm's rows
    const u64 cap = std::min<u64>(ws, (u64)1 << 30), nb = std::max<u64>(n_g1, 2 * std::max<u64>(1, ws / (2 * n * n * ts)));
    const u64 slab = (u64)oz_slab((size_t)cap, c->n_aux, (int)std::min<u64>(n_ov, 2147483647ull));
    const u64 one = 2 * (u64)gw::oz_elems(c->n_aux, (int)slab), per = 2 * (u64)gw::oz_elems(c->n_aux, c->n_aux);
    const u64 eg = std::min(nb, std::max<u64>(1, cap / (2 * one)));
    const u64 sub = std::min(n_g1, std::max<u64>(1, cap / (per + 8 * n * n))), tile = 8 * (u64)gw::oz_sumsq_tiles(c->n_aux) * sub;
    const u64 rc = std::min<u64>(rows, std::max<u64>(128, cap / (per / n)));
    b += std::max(one * eg, rc * (per / n)) + std::max(one * eg, per * sub) + 8 * n * n * sub;
    b += std::min(tile * rows, std::max(cap, tile * 128));                   // the tiles' sums
    if (c->n_aux <= kSmall64) b += 8 * (u64)gw::trsm_w_scratch_elems<double>(c->n_aux, gw::trsm_w_default_ctas());
    b += 12 * n_ov * eg + 8 * std::max(2 * n * eg, rows + n * sub) + 12 * nb;
  }
  // residue batch (at most one right-hand side per target and state at a time)
  u64 batch = c->max_rhs_batch > 0 ? (u64)c->max_rhs_batch
                                   : std::max<u64>(1, std::min<u64>((ws / 2) / (2 * n_ov * ts), 2048));
  batch = std::min(batch, std::max<u64>(1, rows));
  b += batch * (4 * n * ts + 2 * n_ov * ts + 10 * n * 8 + 64);               // V, S, U, Lanczos vectors, state
  if (!mixed && deriv_digits_fit((size_t)ws, c->n_aux, (long)n_ov))            // digits of B^T and V
    b += 16 * (n_ov * ldn + 2 * batch * ldn) + 8 * (n_ov + 2 * batch);
  if (mixed) {
    b += batch * (16 * n + 8 * ldn + 8 * ldo);                               // FP64 solutions, split V and U
    if (c->op_parts >= 3) b += batch * (4 * ldn + 4 * ldo);
    b += batch * 8 * (ldf - n_ov) + 4 * (u64)152 * 128 * 128;                // U rows' padding, partial products
  }
  b += 48 * std::max<u64>(1, rows) + 8 * 6 * (u64)n_t + 64;                  // residue lists, Sigma scratch
  // dense fallback batch
  const u64 mat2 = 2 * n * n * ts;
  const u64 fb = std::max<u64>(1, ws / mat2);
  b += capped(mat2, mat2 * fb) + fb * (2 * n * ts + 8 * n + 8);
  if (mixed) {
    b += fb * (16 * n + 16 * n + 12 * ldn + 12 * ldo + 40);                  // FP64 solutions, V/S, split parts
    b += fb * (32 * n + 16 * n_ov) + 4 * n * n_ov;                           // FP64-residual vectors, df lo part of B
    b += (u64)gw::kDfPartTiles * 64 * 64 * 8;                                // its K ranges' sums
  }
  b += 2 * (u64)lu_work_elems(c->n_aux, (long)std::min<u64>(fb, 1u << 30), !mixed, (size_t)ws);   // blocked-LU operands
  b += fb * (4 * (u64)gw::zlu_index_ints(1) + ts * (u64)gw::zlu_linv_elems(1) + (mixed ? 0 : 8 * (u64)gw::zlu_scale_elems(c->n_aux, 1)));
  *bytes = b + slab_bound(b);
  return GW_OK;
}

gw_status gw_grid(int N, double x0, double* xi, double* wt) {
  if (N <= 0 || !(x0 > 0.0) || !xi || !wt) return GW_ERR_ARG;
  // P_N(t) and P_N'(t) by the three-term recurrence
  auto legendre = [N](double t, double* dp) {
    double p0 = 1.0, p1 = t;
    for (int l = 2; l <= N; ++l) {
      double p2 = ((2.0 * l - 1.0) * t * p1 - (l - 1.0) * p0) / l;
      p0 = p1;
      p1 = p2;
    }
    *dp = N * (t * p1 - p0) / (t * t - 1.0);
    return p1;
  };
  for (int k = 0; k < N; ++k) {
    double t = -std::cos(M_PI * (k + 0.75) / (N + 0.5));   // Newton from the asymptotic node estimate
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p = legendre(t, &dp);
      double dt = p / dp;
      t -= dt;
      if (std::fabs(dt) < 1e-16) break;
    }
    legendre(t, &dp);
    double wgl = 2.0 / ((1.0 - t * t) * dp * dp);
    xi[k] = x0 * (1.0 + t) / (1.0 - t);
    wt[k] = 2.0 * x0 * wgl / ((1.0 - t) * (1.0 - t));
  }
  return GW_OK;
}

gw_status gw_w_table(gw_plan_t P, double* out) {
  if (!P || !out) return P ? fail(P, GW_ERR_ARG, "out is NULL") : GW_ERR_ARG;
  TRY(ensure_screening(P));
  CK(cudaMemcpy(out, P->d_W, sizeof(double) * (size_t)P->n_t * P->n_bas * (P->n_g + 1), cudaMemcpyDeviceToHost));
  return GW_OK;
}

gw_status gw_get_stats(gw_plan_t P, gw_stats* out) {
  if (!P || !out) return GW_ERR_ARG;
  *out = P->stats;
  return GW_OK;
}

void gw_plan_destroy(gw_plan_t P) { free_plan(P); }

const char* gw_last_error(gw_plan_t P) {
  if (!P) return g_create_error.c_str();
  return P->err.c_str();
}

}  // extern "C"
