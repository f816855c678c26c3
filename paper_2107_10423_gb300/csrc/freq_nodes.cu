// Nodes of the imaginary-axis stage.  Every entry of W is a sum over the RPA poles,
//   W_nm(i xi) = -sum_s 2 w_nms^2 Omega_s / (Omega_s^2 + xi^2),   Omega_s >= D_min  (Omega^2 are the eigenvalues of
// D^1/2 (D + 4 B^T B) D^1/2 >= D^2; Sec. 2.2), so as functions on the grid all of them lie in the span of the rows
//   f_Omega(xi_g) = Omega^2 / (Omega^2 + xi_g^2),  Omega in [D_min, inf),
// whose numerical rank is small (37 of 129 at 2e-9 for the 128-point grid and D_min = 0.43; the rank grows with
// log(1/tolerance) log(xi_max/D_min)).  The stage is computed at that many grid points (the nodes) and the other
// columns follow from a fixed matrix.  The nodes are a row-pivoted Gram-Schmidt selection of the sampled family, which
// keeps the matrix small (row 2-norms of 1 to 3 over 32 to 200 points and gaps of 0.01 to 50 Ha): the columns' own
// rounding (about 5e-7 in mixed precision) is not amplified beyond that, and the interpolation's own error, at most 2e-8
// of W(0) there (of themselves for the difference columns, 2e-9), stays below it.
#include "gw_internal.cuh"

#include <algorithm>
#include <cmath>

namespace gw {

namespace {

constexpr double kSamplesPerE = 10;  // sampled poles per factor e, geometric in [D_min, 30 max(xi_max, D_min)]
constexpr double kTol = 2e-9;        // largest residual of the sampled family (each row scaled to maximum 1)
constexpr int kMaxRank = 128;        // beyond this many nodes the stage runs at every grid point

// Row-pivoted Gram-Schmidt of F [nr][m] (row-major, overwritten by its residual): the pivots (in order) until every
// residual element is below tol, and L [nr][kMaxRank] with F ~ L Q.  first >= 0 is taken as the first pivot; stops at
// kMaxRank.  0.5 ms on one core for 106 rows and 37 nodes (a cross approximation of the same family took 0.35 ms and
// found nodes with up to 100 times the error on long grids).
std::vector<int> pivoted_rows(std::vector<double>& F, int nr, int m, double tol, int first, std::vector<double>& L) {
  std::vector<int> piv;
  std::vector<double> q(m), n2(nr);
  std::vector<unsigned char> live(nr, 1);
  L.assign((size_t)nr * kMaxRank, 0.0);
  for (int i = 0; i < nr; ++i) {
    double s = 0.0;
    for (int k = 0; k < m; ++k) s += F[(size_t)i * m + k] * F[(size_t)i * m + k];
    n2[i] = s;
  }
  while ((int)piv.size() < std::min(nr, kMaxRank)) {
    int j = -1;
    if (piv.empty() && first >= 0) {
      j = first;
    } else {
      for (int i = 0; i < nr; ++i)
        if (live[i] && (j < 0 || n2[i] > n2[j])) j = i;
      // the 2-norm bounds the largest element
      if (j < 0 || !(n2[j] > tol * tol)) break;
      double big = 0.0;
      for (int k = 0; k < m; ++k) big = std::max(big, std::fabs(F[(size_t)j * m + k]));
      if (big < tol && n2[j] < m * tol * tol) break;
    }
    const int r = (int)piv.size();
    const double norm = std::sqrt(n2[j]), inv = 1.0 / norm;
    for (int k = 0; k < m; ++k) q[k] = F[(size_t)j * m + k] * inv;
    piv.push_back(j);
    live[j] = 0;
    L[(size_t)j * kMaxRank + r] = norm;
    for (int i = 0; i < nr; ++i) {
      if (!live[i]) continue;
      double* f = &F[(size_t)i * m];
      double p0 = 0.0, p1 = 0.0, p2 = 0.0, p3 = 0.0;
      for (int k = 0; k < m; k += 4) {               // m is a multiple of 4
        p0 += f[k] * q[k];
        p1 += f[k + 1] * q[k + 1];
        p2 += f[k + 2] * q[k + 2];
        p3 += f[k + 3] * q[k + 3];
      }
      const double p = (p0 + p1) + (p2 + p3);
      L[(size_t)i * kMaxRank + r] = p;
      double s0 = 0.0, s1 = 0.0;
      for (int k = 0; k < m; k += 2) {
        f[k] -= p * q[k];
        f[k + 1] -= p * q[k + 1];
        s0 += f[k] * f[k];
        s1 += f[k + 1] * f[k + 1];
      }
      n2[i] = s0 + s1;
    }
  }
  return piv;
}

// Coefficients of every row in the pivot rows: c_i L_S = L_i (L_S lower triangular in pivot order).
std::vector<double> row_coefficients(const std::vector<double>& L, int nr, const std::vector<int>& piv) {
  const int r = (int)piv.size();
  std::vector<double> C((size_t)nr * r, 0.0);
  for (int i = 0; i < nr; ++i) {
    double* c = &C[(size_t)i * r];
    for (int k = r - 1; k >= 0; --k) {
      double v = L[(size_t)i * kMaxRank + k];
      for (int t = k + 1; t < r; ++t) v -= c[t] * L[(size_t)piv[t] * kMaxRank + k];
      c[k] = v / L[(size_t)piv[k] * kMaxRank + k];
    }
  }
  for (int k = 0; k < r; ++k) {       // a node's own row is the unit row
    double* c = &C[(size_t)piv[k] * r];
    std::fill(c, c + r, 0.0);
    c[k] = 1.0;
  }
  return C;
}

// Columns of W from its node columns, one warp-sized group of rows at a time: W[r][g] = sum_p C[p][g] val_p, val the
// row's values at the node positions as the stage left them in W's own columns.  4.5e3 FP64 FMAs a row: at 14448 rows
// (42 targets of a (H2O)_8) 0.15 ms, bound by the FP64 pipe (two FMAs a clock and SM).
constexpr int XR = 8;                 // rows per CTA
__global__ void __launch_bounds__(256) w_expand_kernel(double* __restrict__ W, long R, int n_g, int n_pos,
                                                       const int* __restrict__ col, const double* __restrict__ C) {
  extern __shared__ double val[];     // [XR][n_pos]
  const int ld = n_g + 1;
  for (long r0 = (long)blockIdx.x * XR; r0 < R; r0 += (long)gridDim.x * XR) {
    const int nr = (int)(R - r0 < XR ? R - r0 : XR);
    for (int i = threadIdx.x; i < nr * n_pos; i += blockDim.x)
      val[i] = W[(r0 + i / n_pos) * ld + col[i % n_pos]];
    __syncthreads();
    for (int i = threadIdx.x; i < nr * n_g; i += blockDim.x) {
      const int rr = i / n_g, g = i - rr * n_g;
      const double* v = val + rr * n_pos;
      double s = 0.0;
      for (int p = 0; p < n_pos; ++p) s = fma(C[(long)p * n_g + g], v[p], s);
      W[(r0 + rr) * ld + g] = s;
    }
    __syncthreads();
  }
}

}  // namespace

bool freq_nodes(const std::vector<double>& xi, int n_diff, double D_min, FreqNodes& out) {
  const int n_g = (int)xi.size();
  if (n_g < 24 || !(D_min > 0.0) || !std::isfinite(D_min)) return false;
  for (int g = 0; g < n_g; ++g)
    if (!(xi[g] > 0.0) || !std::isfinite(xi[g]) || (g > 0 && !(xi[g] > xi[g - 1]))) return false;
  const double lo = D_min, hi = 30.0 * std::max(xi[n_g - 1], D_min);
  const int m = 4 * std::max(16, (int)(0.25 * kSamplesPerE * std::log(hi / lo)));
  std::vector<double> O2(m);
  for (int s = 0; s < m; ++s) {
    const double o = lo * std::pow(hi / lo, s / (double)(m - 1));
    O2[s] = o * o;
  }
  auto fill = [&](const std::vector<double>& x, std::vector<double>& F) {
    F.resize(x.size() * m);
    for (size_t i = 0; i < x.size(); ++i) {
      const double x2 = x[i] * x[i], sc = (O2[m - 1] + x2) / O2[m - 1];   // the row's maximum is at the largest pole
      for (int s = 0; s < m; ++s) F[i * m + s] = sc * O2[s] / (O2[s] + x2);
    }
  };
  std::vector<double> F, L;
  // difference-form columns: (W_g - W_0) / xi_g^2 is a sum of 1/(Omega^2 + xi_g^2)
  std::vector<double> xd(xi.begin(), xi.begin() + n_diff);
  std::vector<int> pd;
  std::vector<double> Cd;
  if (n_diff > 0) {
    fill(xd, F);
    pd = pivoted_rows(F, n_diff, m, kTol, -1, L);
    Cd = row_coefficients(L, n_diff, pd);
  }
  // the static point and the other columns
  std::vector<double> xg(1, 0.0);
  xg.insert(xg.end(), xi.begin() + n_diff, xi.end());
  const int ng1 = (int)xg.size();
  fill(xg, F);
  const std::vector<int> pg = pivoted_rows(F, ng1, m, kTol, 0, L);
  const std::vector<double> Cg = row_coefficients(L, ng1, pg);
  const int rd = (int)pd.size(), rg = (int)pg.size(), n_pos = rd + rg;
  if (rd == kMaxRank || rg == kMaxRank || 4 * n_pos > 3 * (n_g + 1)) return false;
  // positions: the static point, then the nodes ascending (difference columns first)
  std::vector<int> od(pd), og(pg.begin() + 1, pg.end());
  std::sort(od.begin(), od.end());
  std::sort(og.begin(), og.end());
  out.col.assign(1, n_g);
  for (int g : od) out.col.push_back(g);
  for (int g : og) out.col.push_back(n_diff + g - 1);
  out.n_diff = rd;
  out.C.assign((size_t)n_pos * n_g, 0.0);
  for (int g = 0; g < n_diff; ++g) {
    out.C[g] = 1.0;                                     // + W_0
    for (int k = 0; k < rd; ++k) {
      const int pos = 1 + (int)(std::lower_bound(od.begin(), od.end(), pd[k]) - od.begin());
      // rows were scaled by (1 + xi^2/Omega_max^2)
      const double sc = (1.0 + xd[pd[k]] * xd[pd[k]] / O2[m - 1]) / (1.0 + xd[g] * xd[g] / O2[m - 1]);
      const double ratio = xd[g] / xd[pd[k]];
      out.C[(size_t)pos * n_g + g] = Cd[(size_t)g * rd + k] * sc * ratio * ratio;
    }
  }
  for (int i = 1; i < ng1; ++i) {
    const int g = n_diff + i - 1;
    for (int k = 0; k < rg; ++k) {
      const int pos = k == 0 ? 0
                             : 1 + rd + (int)(std::lower_bound(og.begin(), og.end(), pg[k]) - og.begin());
      const double sc = (1.0 + xg[pg[k]] * xg[pg[k]] / O2[m - 1]) / (1.0 + xg[i] * xg[i] / O2[m - 1]);
      out.C[(size_t)pos * n_g + g] = Cg[(size_t)i * rg + k] * sc;
    }
  }
  return true;
}

cudaError_t launch_w_expand(double* W, long R, int n_g, int n_pos, const int* col, const double* C, cudaStream_t s) {
  if (R <= 0) return cudaSuccess;
  const long blocks = (R + XR - 1) / XR;
  w_expand_kernel<<<(unsigned)std::min<long>(blocks, 1 << 20), 256, sizeof(double) * XR * n_pos, s>>>(W, R, n_g, n_pos,
                                                                                                     col, C);
  return cudaGetLastError();
}

}  // namespace gw
