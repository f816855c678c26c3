"""Direct diagonalisation of the Casida matrix (tridiagonalisation, twisted vectors, refinement on digit products) at the
edges of its ranges (the smallest N_ov, warps and row blocks of 8, digit tiles of 128 and 256, rows in shared memory up to
about 1800, wide bisection up to 2800) and at exactly degenerate levels, where the Jacobi sweeps take over, against the
oracle's LAPACK route."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_occ,n_virt,n_aux,degenerate", [
    (1, 7, 5, False), (1, 8, 5, False), (3, 11, 20, False), (4, 32, 9, False), (3, 43, 140, False), (4, 64, 60, False),
    (1, 257, 33, False), (5, 250, 130, False), (12, 160, 40, False), (13, 224, 30, False), (4, 32, 9, True),
    (5, 40, 300, True)])
def test_sd_direct(gwlib, n_occ, n_virt, n_aux, degenerate):
    from paper_2107_10423_gb300 import gw
    occ = np.linspace(-1.4, -0.45, n_occ) if n_occ > 1 else np.array([-0.5])
    virt = np.geomspace(0.05, 4.0, n_virt)
    if degenerate:
        virt = np.repeat(virt[::4], 4)
    s = synth.System("sd", np.concatenate([occ, virt]), n_occ, n_aux, 0.3 / np.sqrt(n_aux), 77, np.array([n_occ - 1, n_occ]))
    B, Bn = s.b_ia(), s.b_nm()
    Om, V = O.casida(s.eps, s.n_occ, B)
    # between the levels: occupied Sigma poles lie below the HOMO, virtual ones above the LUMO
    om = np.array([-0.2, -0.15])
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, precision=gw.GW_PREC_FP64) as p:
        sc, dsc = p.sigma_sd(om)
    for t in range(2):
        # off the poles the sums are well conditioned: eigenvalues to 1e-14 of the norm, vectors orthonormal to 1e-13
        ref = O.sigma_c_sd(s.eps, s.n_occ, Bn[t], Om, V, om[t], 1e-3)
        assert abs(sc[t] - ref[0]) < 1e-10 * max(1.0, abs(ref[0])), (t, sc[t], ref[0])
        assert abs(dsc[t] - ref[1]) < 1e-9 * max(1.0, abs(ref[1])), (t, dsc[t], ref[1])
