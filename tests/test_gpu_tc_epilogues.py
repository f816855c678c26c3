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
