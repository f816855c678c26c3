"""Launches of one kernel from several threads at different sizes, as the job server's plans make them: the dynamic
shared-memory limit of a kernel is shared by the process's threads, and a smaller plan's call must not take a larger one's
away between its set-up and its launch."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2107_10423_gb300")

pytestmark = pytest.mark.gpu

SRC = r"""
#include "gw_internal.cuh"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
std::atomic<int> failed{0};
// `count` solves with unit factors of n rows (identity: y stays as it is) on a stream of its own
template <typename T> void work(int n, int count) {
  cudaStream_t s;
  T *A, *y;
  int* perm;
  std::vector<T> h(2 * (size_t)n * n, T(0)), v(2 * n, T(3));
  std::vector<int> id(n);
  for (int i = 0; i < n; ++i) { h[(size_t)i * n + i] = T(1); id[i] = i; }
  bool ok = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess &&
            cudaMalloc(&A, h.size() * sizeof(T)) == cudaSuccess && cudaMalloc(&y, 2 * n * sizeof(T)) == cudaSuccess &&
            cudaMalloc(&perm, n * sizeof(int)) == cudaSuccess &&
            cudaMemcpy(A, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice) == cudaSuccess &&
            cudaMemcpy(y, v.data(), 2 * n * sizeof(T), cudaMemcpyHostToDevice) == cudaSuccess &&
            cudaMemcpy(perm, id.data(), n * sizeof(int), cudaMemcpyHostToDevice) == cudaSuccess;
  if (!ok) { failed += 1 << 20; return; }
  for (int i = 0; i < count; ++i) {
    const cudaError_t e = gw::launch_zlu_solve<T>(A, A + (size_t)n * n, 2L * n * n, n, 1, perm, y, y + n, 2L * n, s);
    if (e != cudaSuccess && failed++ == 0) std::printf("n %d: %s\n", n, cudaGetErrorString(e));
  }
  if (cudaStreamSynchronize(s) != cudaSuccess ||
      cudaMemcpy(h.data(), y, 2 * n * sizeof(T), cudaMemcpyDeviceToHost) != cudaSuccess)
    failed += 1 << 20;
  for (int i = 0; i < 2 * n; ++i)
    if (h[i] != T(3)) { failed += 1 << 10; break; }
}
int main() {
  std::vector<std::thread> t;
  // 68 and 73 KiB of shared memory in FP64, 34 and 50 in FP32
  for (int k = 0; k < 4; ++k) t.emplace_back(work<double>, k % 2 ? 16 : 300, 12000);
  for (int k = 0; k < 2; ++k) t.emplace_back(work<float>, k % 2 ? 16 : 2000, 1500);
  for (auto& th : t) th.join();
  std::printf("%d\n", failed.load());
  return failed.load() != 0;
}
"""


def test_shared_memory_limit_of_concurrent_launches(gwlib, tmp_path):
    nvcc = os.environ.get("NVCC") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc")
                                      else shutil.which("nvcc"))
    if not nvcc:
        pytest.skip("nvcc not found")
    (tmp_path / "t.cu").write_text(SRC)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                        "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(PKG, "csrc"), str(tmp_path / "t.cu"),
                        "-o", str(tmp_path / "t"), "-L" + PKG, "-lgw", "-Xlinker", "-rpath=" + PKG, "-Xcompiler", "-pthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout + r.stderr
