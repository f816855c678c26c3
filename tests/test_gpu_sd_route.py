"""Spectral decomposition: the direct route runs where it should (the sweeps would launch 4 (N_ov - 1) kernels each) and the
sweeps where it finds no basis (equal levels of pairs that couple to nothing: their twisted vectors coincide), both give the
oracle's values, and a plan keeps the poles and weights only, not the matrices of the
diagonalisation."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n_occ,n_virt,n_aux,levels", [(1, 8, 5, "distinct"), (5, 250, 130, "distinct"),
                                                       (13, 100, 30, "distinct"), (4, 32, 9, "degenerate"),
                                                       (4, 32, 9, "decoupled"), (11, 120, 40, "decoupled")])
def test_route_and_memory(gwlib, prec, n_occ, n_virt, n_aux, levels):
    from paper_2107_10423_gb300 import gw
    occ = np.linspace(-1.4, -0.45, n_occ) if n_occ > 1 else np.array([-0.5])
    virt = np.geomspace(0.05, 4.0, n_virt)
    if levels != "distinct":
        virt = np.repeat(virt[::4], 4)
    s = synth.System("sd", np.concatenate([occ, virt]), n_occ, n_aux, 0.3 / np.sqrt(n_aux), 77, np.array([n_occ - 1, n_occ]))
    B, Bn = s.b_ia(), s.b_nm()
    if levels == "decoupled":
        B.reshape(n_aux, n_occ, n_virt)[:, :, -8:] = 0.0
    N = n_occ * n_virt
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets,
                 precision=gw.GW_PREC_FP64 if prec == "fp64" else gw.GW_PREC_MIXED) as p:
        before = p.stats()
        first = p.sigma_sd(np.array([-0.2, -0.15]))
        st = p.stats()
        again = p.sigma_sd(np.array([-0.2, -0.15]))
        after = p.stats()
    launches = st["n_kernel_launches"] - before["n_kernel_launches"]
    assert launches >= 4 * (N - 1) if levels == "decoupled" else launches < 100, launches
    if N < 500:
        Om, V = O.casida(s.eps, s.n_occ, B)
        for t, om in enumerate((-0.2, -0.15)):
            ref = O.sigma_c_sd(s.eps, s.n_occ, Bn[t], Om, V, om, 1e-3)
            assert abs(first[0][t] - ref[0]) < 1e-10 * max(1.0, abs(ref[0]))
            assert abs(first[1][t] - ref[1]) < 1e-9 * max(1.0, abs(ref[1]))
    assert after["n_kernel_launches"] - st["n_kernel_launches"] < 8           # the second evaluation reuses the poles
    assert np.array_equal(first[0], again[0]) and np.array_equal(first[1], again[1])
    # poles and weights, and slabs of 32 MiB for what is small
    kept = 8 * N * (1 + 2 * s.n_bas)
    assert st["bytes_device"] - before["bytes_device"] <= kept + 3 * (32 << 20), (st["bytes_device"], kept)
