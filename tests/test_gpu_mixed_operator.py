"""The mixed residue operator's forms by batch size (FP32 kernels for up to four right-hand sides; tensor-core products
above, the second split over K where its output tiles are few) against the oracle, at odd sizes: 190 to 3255 pairs."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rhs,batch", [(1, 0), (2, 0), (3, 0), (4, 0), (5, 0), (21, 0), (11, 4), (13, 5)])
@pytest.mark.parametrize("n_aux,n_occ,n_virt", [(30, 5, 38), (129, 7, 61), (257, 15, 217)])
def test_mixed_residues(gwlib, n_aux, n_occ, n_virt, n_rhs, batch):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([np.linspace(-2.0, -0.45, n_occ), np.linspace(0.05, 6.0, n_virt)])
    s = synth.System("op", eps, n_occ, n_aux, 0.6 / np.sqrt(n_aux), n_aux, np.array([n_occ - 1]))
    B, Bn = s.b_ia(), s.b_nm()
    r = np.random.default_rng(n_rhs)
    m, x = r.integers(0, s.n_bas, n_rhs), r.uniform(-0.35, 0.35, n_rhs)     # inside the gap: MINRES converges
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, precision=gw.GW_PREC_MIXED, minres_tol=1e-7, minres_maxit=300,
                 minres_fallback_tol=1e-5, max_rhs_batch=batch) as p:
        out = p.residues(np.zeros(n_rhs, dtype=np.int32), m, x)
    assert not out["used_fallback"].any()
    for j in range(n_rhs):
        w, _ = O.w_corr_and_deriv(O.pi_complex(s.eps, s.n_occ, B, x[j], 1e-3),
                                  O.dpi_complex(s.eps, s.n_occ, B, x[j], 1e-3), Bn[0, m[j]])
        # operator error times the condition number of 1 - Pi(x) in the gap (below 50): BF16 pairs 2^-16, FP32 1e-6
        tol = 50 * (1e-6 if (batch or n_rhs) <= 4 and n_rhs <= 4 else 2.0 ** -16)
        assert abs(out["w_re"][j] - w.real) < tol * max(1, abs(w))
        assert abs(out["w_im"][j] - w.imag) < tol * max(1, abs(w))
