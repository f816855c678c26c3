"""Dense residue solves (blocked complex LU, panels of 64 columns held in registers) at the edges of its panels and of
its rows per thread (512 threads), FP64 and mixed, against the oracle's dense complex solve."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_aux,n_rhs", [("fp64", 1, 2), ("fp64", 63, 3), ("fp64", 64, 3), ("fp64", 65, 3),
                                              ("fp64", 129, 40), ("fp64", 513, 3), ("fp64", 1030, 2),
                                              ("mixed", 64, 3), ("mixed", 65, 3), ("mixed", 129, 40), ("mixed", 513, 3),
                                              ("mixed", 1030, 2)])
def test_dense_residues(gwlib, prec, n_aux, n_rhs):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([np.linspace(-1.4, -0.45, 5), np.linspace(0.05, 4.0, 40)])
    s = synth.System("lu", eps, 5, n_aux, 0.6 / np.sqrt(n_aux), n_aux, np.array([4]))
    B, Bn = s.b_ia(), s.b_nm()
    r = np.random.default_rng(n_aux)
    m, x = r.integers(0, s.n_bas, n_rhs), r.uniform(-2.0, 2.0, n_rhs)
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, minres_tol=1e-14, minres_maxit=1, minres_fallback_tol=1e-13,
                 precision=gw.GW_PREC_FP64 if prec == "fp64" else gw.GW_PREC_MIXED) as p:
        out = p.residues(np.zeros(n_rhs, dtype=np.int32), m, x)
    dense = out["used_fallback"] == 1
    assert dense.sum() >= (n_rhs if n_aux > 1 else 0)
    for j in np.nonzero(dense)[0]:
        w, _ = O.w_corr_and_deriv(O.pi_complex(s.eps, s.n_occ, B, x[j], 1e-3),
                                  O.dpi_complex(s.eps, s.n_occ, B, x[j], 1e-3), Bn[0, m[j]])
        # resonances at eta = 1e-3 make 1 - Pi(x) as ill-conditioned as about 1e5: FP64 LU (backward error of a few
        # n 2^-53) within 1e-8; mixed with a double-float refinement residual within the 2e-6 of the dense-path test
        tol = 1e-8 if prec == "fp64" else 2e-6
        assert abs(out["w_re"][j] - w.real) < tol * max(1, abs(w)), (j, out["w_re"][j], w)
        assert abs(out["w_im"][j] - w.imag) < tol * max(1, abs(w)), (j, out["w_im"][j], w)
