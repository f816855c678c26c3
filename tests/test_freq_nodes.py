"""Nodes of the imaginary-axis stage (mixed precision): the matrix that gives every grid column of W from the node
columns (host code in libgw.so), and the table built with it against the oracle's dense solves."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2107_10423_gb300")

# Every pole Omega >= D contributes 1/(Omega^2 + xi^2) to each column and -xi^2/(Omega^2 (Omega^2 + xi^2)) to each
# difference from the static one: both families are reproduced at every grid point.  The sampled family is fitted to
# 2e-9; 10 samples per factor e leave poles between them within 50 times that, relative to W(0) for the columns and
# relative to themselves for the differences.
SRC = r"""
#include "gw.h"
#include "gw_internal.cuh"
#include <cmath>
#include <cstdio>
#include <cstdlib>
int main() {
  for (int N : {32, 64, 128, 200}) for (double D : {0.02, 0.2, 0.43, 2.0, 50.0}) {
    std::vector<double> xi(N), wt(N);
    if (gw_grid(N, 0.5, xi.data(), wt.data()) != GW_OK) return 1;
    int nd = 0;
    while (nd < N && xi[nd] < 0.1 * D) ++nd;
    gw::FreqNodes F;
    if (!gw::freq_nodes(xi, nd, D, F)) continue;
    const int np = (int)F.col.size();
    if (F.col[0] != N || (int)F.C.size() != np * N) { std::printf("layout\n"); return 1; }
    for (int p = 1; p < np; ++p)
      if (F.col[p] < 0 || F.col[p] >= N || (p > 1 && F.col[p] <= F.col[p - 1]) || (p <= F.n_diff) != (F.col[p] < nd)) {
        std::printf("N %d D %g: position %d\n", N, D, p);
        return 1;
      }
    for (int q = 0; q < 400; ++q) {
      const double O = D * std::pow(1e5 / D, q / 399.0), O2 = O * O;
      std::vector<double> v(np);
      v[0] = 1.0;
      for (int p = 1; p < np; ++p) {
        const double x2 = xi[F.col[p]] * xi[F.col[p]];
        v[p] = p <= F.n_diff ? -x2 / (O2 + x2) : O2 / (O2 + x2);
      }
      for (int g = 0; g < N; ++g) {
        const double x2 = xi[g] * xi[g];
        double s = 0.0;
        for (int p = g < nd ? 1 : 0; p < np; ++p) s += F.C[(size_t)p * N + g] * v[p];
        const double want = g < nd ? -x2 / (O2 + x2) : O2 / (O2 + x2);
        const double tol = 1e-7 * (g < nd ? x2 / (O2 + x2) : 1.0);
        if (!(std::fabs(s - want) <= tol) || (g < nd && F.C[g] != 1.0)) {
          std::printf("N %d D %g pole %g grid point %d: %.3e, want %.3e\n", N, D, O, g, s, want);
          return 1;
        }
      }
    }
  }
  std::vector<double> xi(64), wt(64);
  gw_grid(64, 0.5, xi.data(), wt.data());
  gw::FreqNodes F;
  std::vector<double> bad(xi);
  std::swap(bad[3], bad[40]);
  if (gw::freq_nodes(bad, 0, 0.5, F) || gw::freq_nodes(xi, 0, 0.0, F) || gw::freq_nodes(xi, 0, NAN, F)) return 1;
  bad = xi;
  bad[0] = 0.0;
  if (gw::freq_nodes(bad, 0, 0.5, F)) return 1;
  std::printf("ok\n");
  return 0;
}
"""


def test_nodes_reproduce_every_pole(gwlib, tmp_path):
    nvcc = os.environ.get("NVCC") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc")
                                      else shutil.which("nvcc"))
    if not nvcc:
        pytest.skip("nvcc not found")
    src = tmp_path / "nodes.cu"
    src.write_text(SRC)
    exe = tmp_path / "nodes"
    cmd = [nvcc, "-std=c++17", "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(PKG, "csrc"), str(src),
           "-o", str(exe), "-L" + PKG, "-lgw", "-Xlinker", "-rpath=" + PKG]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr


# just above one 128-row tile, a ragged size with a long grid, a small gap (wide spectrum: more nodes), a large gap
# (most columns in the difference form), and a grid too short for nodes; workspace_mb = 1 runs at every grid point
@pytest.mark.gpu
@pytest.mark.parametrize("n_aux,n_virt,n_freq,gap", [(129, 40, 128, 0.5), (203, 57, 200, 0.5), (150, 31, 128, 0.02),
                                                     (150, 31, 128, 3.0), (130, 31, 20, 0.5)])
def test_w_table_at_nodes(gwlib, n_aux, n_virt, n_freq, gap):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([[-20.5], np.linspace(-1.3, -0.45, 5), np.linspace(-0.45 + gap, 4.0, n_virt)])
    s = synth.System("nodes", eps, 6, n_aux, 0.6 / np.sqrt(n_aux), 11, np.array([5, 6]))
    B, Bn = s.b_ia(), s.b_nm()
    xi, wt = O.mgl_grid(n_freq, 0.5)
    ref = np.stack([np.stack([O.w_corr(O.pi_imag(s.eps, s.n_occ, B, x), Bn[t].T) for x in np.append(xi, 0.0)], 1)
                    for t in range(len(s.targets))])
    for ws in (0, 1):
        with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, precision=gw.GW_PREC_MIXED, xi=xi, wt=wt, workspace_mb=ws) as p:
            W = p.w_table()
        # Pi from BF16 hi/lo products, about 16 bits an operand and random over the pairs (2^-17 sqrt(2) / sqrt(pairs)
        # of the sum, < 1e-6), and an FP32 inverse (2^-24 sqrt(n_aux) times the condition number, < 1e-5 in all); the
        # nodes add 1e-7 at most
        assert np.abs(W - ref).max() < 1e-5 * np.abs(ref).max()
