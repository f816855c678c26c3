"""PerDevice (set-up of kernel attributes): once on every device, again where it failed, from any thread."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2107_10423_gb300")

SRC = r"""
#include "gw_internal.cuh"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  gw::PerDevice p;
  int runs[130] = {};
  for (int pass = 0; pass < 3; ++pass)
    for (int d = 0; d < 128; ++d)
      if (p.run(d, [&] { ++runs[d]; return cudaSuccess; }) != cudaSuccess) return 1;
  for (int d = 0; d < 128; ++d)
    if (runs[d] != 1) return std::printf("device %d: %d runs\n", d, runs[d]), 1;
  for (int d : {-1, 128})                       // devices beyond the table: every time
    for (int i = 0; i < 2; ++i)
      if (p.run(d, [&] { ++runs[129]; return cudaSuccess; }) != cudaSuccess) return 1;
  if (runs[129] != 4) return 1;
  gw::PerDevice f;                              // a failure is handed on and tried again
  int n = 0;
  auto fail_once = [&] { return n++ == 0 ? cudaErrorInvalidValue : cudaSuccess; };
  if (f.run(5, fail_once) != cudaErrorInvalidValue || f.run(5, fail_once) != cudaSuccess || n != 2 ||
      f.run(5, fail_once) != cudaSuccess || n != 2) return 1;
  gw::PerDevice q;                              // no thread goes on before a set-up of its device has finished
  std::atomic<int> done{0}, early{0};
  std::vector<std::thread> t;
  for (int k = 0; k < 8; ++k)
    t.emplace_back([&] {
      q.run(0, [&] { std::this_thread::sleep_for(std::chrono::milliseconds(20)); ++done; return cudaSuccess; });
      if (done.load() == 0) ++early;
    });
  for (auto& th : t) th.join();
  if (early.load()) return 1;
  std::printf("ok\n");
  return 0;
}
"""


def test_per_device(gwlib, tmp_path):
    nvcc = os.environ.get("NVCC") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc")
                                      else shutil.which("nvcc"))
    if not nvcc:
        pytest.skip("nvcc not found")
    (tmp_path / "t.cu").write_text(SRC)
    r = subprocess.run([nvcc, "-std=c++17", "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(PKG, "csrc"),
                        str(tmp_path / "t.cu"), "-o", str(tmp_path / "t"), "-Xcompiler", "-pthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
