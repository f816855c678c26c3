"""FP64 products on digits where rows hold elements of very different size: polarizabilities of rows whose largest elements
meet small ones (computed again on the FP64 pipe), and dense residues at a resonance of a weakly coupled pair with a very
small broadening, where one weight is many orders above the others and half of the rows do not see it."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


def _system(n_aux, n_occ, n_virt):
    eps = np.concatenate([np.linspace(-20.5, -0.45, n_occ), np.linspace(0.05, 9.0, n_virt)])
    return synth.System("ranges", eps, n_occ, n_aux, 0.6 / np.sqrt(n_aux), n_aux + n_virt, np.array([n_occ - 1]))


# one column of its own per row, 1e3 to 1e12 above the others; rows beyond one 64-row tile; disjoint halves (sums of
# |terms| far below the rows' largest elements) and K slabs (1 MiB of work space)
@pytest.mark.parametrize("n_aux,n_occ,n_virt,factor,ws", [(40, 10, 40, 1e3, 0), (130, 10, 40, 1e5, 0),
                                                          (130, 10, 40, 1e7, 1), (70, 5, 80, 1e12, 0)])
@pytest.mark.parametrize("halves", [False, True])
def test_polarizability_rows_of_wide_range(gwlib, n_aux, n_occ, n_virt, factor, ws, halves):
    from paper_2107_10423_gb300 import gw
    s = _system(n_aux, n_occ, n_virt)
    B, Bn = s.b_ia(), s.b_nm()
    r = np.random.default_rng(n_aux)
    if halves:                              # even rows large in the first half of the columns, odd rows in the second
        B[::2, : s.n_ov // 2] *= factor
        B[1::2, s.n_ov // 2:] *= factor
    else:
        B[np.arange(n_aux), r.integers(0, s.n_ov, n_aux)] *= factor
    xi = np.array([0.0, 0.7, 30.0])
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, workspace_mb=ws) as p:
        Pi = p.polarizability(xi)
    D = O.pair_energies(s.eps, s.n_occ)
    for g, x in enumerate(xi):
        w = -4.0 * D / (D * D + x * x)
        # the reference's own error: K products and sums in FP64, each within 2^-53 of the absolute terms so far
        bound = (s.n_ov + 2) * 2.0 ** -53 * ((np.abs(B) * np.abs(w)) @ np.abs(B).T) + 1e-300
        assert np.all(np.abs(Pi[g] - (B * w) @ B.T) <= bound), np.max(np.abs(Pi[g] - (B * w) @ B.T) / bound)
        assert np.array_equal(Pi[g], Pi[g].T)


@pytest.mark.parametrize("eta", [1e-3, 1e-12, 1e-16])
def test_dense_residue_at_a_resonance(gwlib, eta):
    from paper_2107_10423_gb300 import gw
    n_aux = 130
    s = _system(n_aux, 3, 43)
    B, Bn = s.b_ia(), s.b_nm()
    D = O.pair_energies(s.eps, s.n_occ)
    k0 = 57
    B[:, k0] *= np.sqrt(eta)               # the pair's term 2/eta b b^T is as large as the others'
    B[::2, k0] = 0.0
    m, x = np.array([0, 7, 40]), np.full(3, D[k0])
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, eta=eta, minres_tol=1e-14, minres_maxit=1,
                 minres_fallback_tol=1e-13) as p:
        out = p.residues(np.zeros(3, dtype=np.int32), m, x)
    assert out["used_fallback"].all()
    pi = O.pi_complex(s.eps, s.n_occ, B, D[k0], eta)
    # FP64 LU: a backward error of a few n 2^-53 of the matrix, times its condition number and |b|^2
    cond = np.linalg.cond(np.eye(n_aux) - pi)
    for j in range(3):
        b = Bn[0, m[j]]
        w = b @ np.linalg.solve(np.eye(n_aux) - pi, b.astype(complex)) - b @ b
        tol = 4 * n_aux * 2.0 ** -53 * cond * (b @ b)
        assert abs(out["w_re"][j] - w.real) < tol and abs(out["w_im"][j] - w.imag) < tol, (j, out["w_re"][j], w, tol)


@pytest.mark.parametrize("ws", [0, 1])
def test_polarizability_of_non_finite_rows(gwlib, ws):
    from paper_2107_10423_gb300 import gw
    s = _system(200, 13, 79)
    B, Bn = s.b_ia(), s.b_nm()
    B[3, 17], B[70, 1000], B[71, 1000], B[150, 5] = np.inf, -np.inf, np.inf, np.nan
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, workspace_mb=ws) as p:
        Pi = p.polarizability(np.array([0.0, 1.3]))
    D = O.pair_energies(s.eps, s.n_occ)
    for g, x in enumerate((0.0, 1.3)):
        w = -4.0 * D / (D * D + x * x)
        # every product of an infinite element is infinite (no zeros here), its sign that of the other factors
        with np.errstate(invalid="ignore"):
            want = np.array([[np.sum(B[p] * w * B[q]) for q in range(200)] for p in range(200)])
        assert np.array_equal(np.isnan(Pi[g]), np.isnan(want))
        inf = np.isinf(want)
        assert np.array_equal(Pi[g][inf], want[inf])
        ok = np.isfinite(want)
        assert ok.sum() == 196 ** 2 and np.allclose(Pi[g][ok], want[ok], rtol=0, atol=1e-12)
