"""Dense residue solves at the sizes of the LU's other forms: 8, 16 and 32 rows a thread (panels of 4, 2 or 1 columns) and
panels in global memory (n above 8192 in FP64, above 16384 in mixed precision).  Pi has rank n_ov = 36 here, so the
reference is a 36 x 36 solve in the pair space (Woodbury)."""
import time

import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_aux,n_rhs", [("fp64", 2100, 3), ("fp64", 4110, 2), ("fp64", 8203, 2), ("mixed", 2100, 3),
                                              ("mixed", 4110, 2), ("mixed", 8203, 2), ("mixed", 16397, 1)])
def test_dense_residues_of_large_matrices(gwlib, prec, n_aux, n_rhs):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([np.linspace(-1.4, -0.45, 3), np.linspace(0.05, 4.0, 12)])
    s = synth.System("lu", eps, 3, n_aux, 0.6 / np.sqrt(n_aux), n_aux, np.array([2]))
    B, Bn = s.b_ia(), s.b_nm()
    D = O.pair_energies(s.eps, s.n_occ)
    r = np.random.default_rng(n_aux)
    m = r.integers(0, s.n_bas, n_rhs)
    x = np.array([v for v in r.uniform(-2.0, 2.0, 400) if np.abs(np.abs(v) - D).min() > 0.02][:n_rhs])
    eta = 1e-3
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, eta=eta, minres_tol=1e-14, minres_maxit=1, minres_fallback_tol=1e-13,
                 precision=gw.GW_PREC_FP64 if prec == "fp64" else gw.GW_PREC_MIXED) as p:
        t0 = time.perf_counter()
        out = p.residues(np.zeros(n_rhs, dtype=np.int32), m, x)
        took = time.perf_counter() - t0
    print(prec, n_aux, "%.2f s" % took)
    assert out["used_fallback"].all()
    assert took < 60.0                       # the trailing updates of one SM alone would take minutes at the largest sizes
    for j in range(n_rhs):
        a1, a2 = x[j] - D + 1j * eta, -x[j] - D + 1j * eta
        c, dc = 2 * (1 / a1 + 1 / a2), 2 * (-1 / a1 ** 2 + 1 / a2 ** 2)
        q = B.T @ Bn[0, m[j]]
        z = np.linalg.solve(np.diag(1 / c) - B.T @ B, q.astype(complex))      # y = b + B z solves (1 - B c B^T) y = b
        w, t = q @ z, q + (B.T @ B) @ z
        dw = (dc * t * t).sum()
        # condition numbers below 1e3 at 0.02 from the poles: FP64 LU (a few n 2^-53) within 1e-9; mixed with the
        # double-float refinement residual within the 2e-6 of the dense-path tests, its FP32 derivative within 1e-4
        tol, dtol = (1e-9, 1e-8) if prec == "fp64" else (2e-6, 1e-4)
        assert abs(out["w_re"][j] - w.real) < tol * max(1, abs(w)), (j, out["w_re"][j], w)
        assert abs(out["w_im"][j] - w.imag) < tol * max(1, abs(w)), (j, out["w_im"][j], w)
        assert abs(out["dw_re"][j] - dw.real) < dtol * max(1, abs(dw)), (j, out["dw_re"][j], dw)
