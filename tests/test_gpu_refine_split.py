"""K ranges of the double-float refinement residual (at least 512 pairs each): one range just below the first split, a
ragged last range, and several ranges with more than one tile of rows, against the oracle's dense complex solve."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux,n_virt,n_rhs", [(64, 204, 3), (64, 205, 3), (65, 240, 3), (130, 701, 40)])
def test_refinement_ranges(gwlib, n_aux, n_virt, n_rhs):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([np.linspace(-1.4, -0.45, 5), np.linspace(0.05, 4.0, n_virt)])
    s = synth.System("ranges", eps, 5, n_aux, 0.6 / np.sqrt(n_aux), n_virt, np.array([4]))
    B, Bn = s.b_ia(), s.b_nm()
    r = np.random.default_rng(n_virt)
    m, x = r.integers(0, s.n_bas, n_rhs), r.uniform(-2.0, 2.0, n_rhs)
    # refine_tol 0: every solve takes the double-float step
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, minres_tol=1e-14, minres_maxit=1, minres_fallback_tol=1e-13,
                 precision=gw.GW_PREC_MIXED, refine_tol=0.0) as p:
        out = p.residues(np.zeros(n_rhs, dtype=np.int32), m, x)
        assert p.stats()["n_refine_fp64"] == n_rhs
    for j in range(n_rhs):
        w, _ = O.w_corr_and_deriv(O.pi_complex(s.eps, s.n_occ, B, x[j], 1e-3),
                                  O.dpi_complex(s.eps, s.n_occ, B, x[j], 1e-3), Bn[0, m[j]])
        # as the dense-path test: the 48-bit residual leaves the FP32 factors' contraction, within 2e-6
        assert abs(out["w_re"][j] - w.real) < 2e-6 * max(1, abs(w)), (j, out["w_re"][j], w)
        assert abs(out["w_im"][j] - w.imag) < 2e-6 * max(1, abs(w)), (j, out["w_im"][j], w)
