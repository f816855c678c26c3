"""Reductions in the epilogues of the mixed-precision tensor-core products, in both tile widths (128 and 256 columns; the
wide one from 120 tiles on), driven through libgw.so with operands whose products are known exactly."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2107_10423_gb300")

pytestmark = pytest.mark.gpu

HEAD = r"""
#include "gw_internal.cuh"
#include "pi_tc.cuh"
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#define CK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) { std::printf("%s: %s\n", #x, cudaGetErrorString(e_)); \
  std::exit(1); } } while (0)
template <typename T> T* up(const std::vector<T>& v) {
  T* p;
  CK(cudaMalloc(&p, v.size() * sizeof(T)));
  CK(cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
  return p;
}
template <typename T> T* zeros(size_t n) {
  T* p;
  CK(cudaMalloc(&p, n * sizeof(T)));
  CK(cudaMemset(p, 0, n * sizeof(T)));
  return p;
}
template <typename T> std::vector<T> down(const T* p, size_t n) {
  std::vector<T> v(n);
  CK(cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost));
  return v;
}
// three BF16 parts of [rows][cols]
struct Split {
  __nv_bfloat16* p[3];
  Split(const std::vector<float>& x, int rows, int cols) {
    float* d = up(x);
    for (auto& q : p) q = zeros<__nv_bfloat16>((size_t)rows * gw::tc_ld(cols));
    CK(gw::tc_split_rows(d, rows, cols, cols, p[0], p[1], 0, p[2]));
  }
  gw::TcOperand op() const { return gw::TcOperand{{p[0], p[1], p[2]}}; }
};
"""

# W[r] = sum_m b[r][m] v[m][r] with v = the rows of B (the left operand is the identity): 22-bit integers, whose products
# and sums FP64 holds exactly (at most 2^44 a term, 256 terms); the sums cancel to about 2^48, so 48 bits do not do.
WRED = HEAD + r"""
int run(int n, int R) {
  std::mt19937_64 g(n + R);
  auto ints = [&] { return (float)((long)(g() % (1ull << 23)) - (1l << 22)); };
  std::vector<float> I((size_t)n * n, 0.f), B((size_t)R * n), b((size_t)R * n);
  for (int i = 0; i < n; ++i) I[(size_t)i * n + i] = 1.f;
  for (auto& v : B) v = ints();
  for (auto& v : b) v = ints();
  Split a(I, n, n), s(B, R, n);
  gw::TcEpi e{};
  e.kind = gw::TC_EPI_WRED;
  e.W = zeros<double>(R);
  e.wld = 1;
  e.gidx = zeros<int>(1);
  e.bvec = up(b);
  e.ldb = n;
  int* err = zeros<int>(1);
  CK(gw::tc_gemm_ex(a.op(), 1, s.op(), 0, 3, n, R, n, e, err, 0));
  CK(cudaDeviceSynchronize());
  const auto W = down(e.W, R);
  if (down(err, 1)[0] != 0) return std::printf("wait\n"), 1;
  for (int r = 0; r < R; ++r) {
    long want = 0;
    for (int m = 0; m < n; ++m) want += (long)B[(size_t)r * n + m] * (long)b[(size_t)r * n + m];
    if (W[r] != (double)want) return std::printf("n %d R %d row %d: %.17g, want %ld\n", n, R, r, W[r], want), 1;
  }
  return 0;
}
int main() {
  if (run(16, 40) || run(200, 129) || run(256, 60 * 256) || run(129, 60 * 256 - 3)) return 1;
  std::printf("ok\n");
  return 0;
}
"""


# Weights c(x) of one right-hand side a pair of rows, with B^T u = 1 and B^T v = 0: rows 2j, 2j + 1 become Re c, Im c.
# x - D runs down to 1e-13 of x at an eta below that: a1 within an ulp (2^-23), its square twice that, eta^2, the sum, two
# divisions and a sum half an ulp each: 2^-20 in all; the parts hold 24 bits.
CPAIR = HEAD + r"""
int run(int nr, int N, int K, double eta) {
  std::mt19937_64 g(nr + N);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  const int M = 2 * nr;
  std::vector<double> x(nr), D(N);
  for (auto& v : x) v = 0.3 + 0.4 * u(g);
  for (int k = 0; k < N; ++k) D[k] = k % 2 ? x[(k / 2) % nr] * (1.0 + (k % 4 == 1 ? 1 : -1) * std::pow(10.0, -13.0 * u(g)))
                                           : 20.0 * u(g) + 0.01;
  std::vector<float> A((size_t)M * K, 0.f), B((size_t)N * K, 0.f);
  for (int j = 0; j < nr; ++j) A[(size_t)2 * j * K] = 1.f;
  for (int k = 0; k < N; ++k) B[(size_t)k * K] = 1.f;
  Split a(A, M, K), b(B, N, K);
  const int ld = gw::tc_ld(N);
  gw::TcEpi e{};
  e.kind = gw::TC_EPI_CPAIR;
  e.Dk = up(D);
  e.x = up(x);
  e.eta = (float)eta;
  e.ohi = zeros<__nv_bfloat16>((size_t)M * ld);
  e.olo = zeros<__nv_bfloat16>((size_t)M * ld);
  e.olo2 = zeros<__nv_bfloat16>((size_t)M * ld);
  e.ldh = ld;
  int* err = zeros<int>(1);
  CK(gw::tc_gemm_ex(a.op(), 1, b.op(), 0, 2, M, N, K, e, err, 0));
  CK(cudaDeviceSynchronize());
  const auto h = down(e.ohi, (size_t)M * ld), l = down(e.olo, (size_t)M * ld), t = down(e.olo2, (size_t)M * ld);
  if (down(err, 1)[0] != 0) return std::printf("wait\n"), 1;
  const double e1 = (double)(float)eta;
  double worst = 0.0;
  for (int j = 0; j < nr; ++j)
    for (int k = 0; k < N; ++k) {
      const double a1 = x[j] - D[k], a2 = -x[j] - D[k], d1 = a1 * a1 + e1 * e1, d2 = a2 * a2 + e1 * e1;
      const double want[2] = {2.0 * (a1 / d1 + a2 / d2), -2.0 * e1 * (1.0 / d1 + 1.0 / d2)};
      const double size[2] = {2.0 * (std::fabs(a1) / d1 + std::fabs(a2) / d2), -want[1]};
      for (int c = 0; c < 2; ++c) {
        const size_t o = (size_t)(2 * j + c) * ld + k;
        const double v = (double)__bfloat162float(h[o]) + (double)__bfloat162float(l[o]) + (double)__bfloat162float(t[o]);
        worst = std::max(worst, std::fabs(v - want[c]) / size[c]);
      }
    }
  if (!(worst < std::ldexp(1.0, -20))) return std::printf("nr %d N %d: %.3g\n", nr, N, worst), 1;
  return 0;
}
int main() {
  if (run(5, 300, 16, 1e-14) || run(64, 1000, 40, 1e-9) || run(128, 60 * 256 - 5, 16, 1e-14) ||
      run(70, 60 * 256, 24, 1e-3)) return 1;
  std::printf("ok\n");
  return 0;
}
"""


def _run(tmp_path, src):
    nvcc = os.environ.get("NVCC") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc")
                                      else shutil.which("nvcc"))
    if not nvcc:
        pytest.skip("nvcc not found")
    (tmp_path / "t.cu").write_text(src)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(PKG, "csrc"), str(tmp_path / "t.cu"),
                        "-o", str(tmp_path / "t"), "-L" + PKG, "-lgw", "-Xlinker", "-rpath=" + PKG],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


def test_w_reduction_keeps_fp64_bits(gwlib, tmp_path):
    _run(tmp_path, WRED)


def test_pole_weights_keep_the_bits_of_the_difference(gwlib, tmp_path):
    _run(tmp_path, CPAIR)
