"""FP64 products on the tensor cores by integer digits (oz_gemm.cu): the polarizability and the W table of FP64 plans
at the edges of the kernel's tiles (128 x 64 outputs, 128 of K), in K slabs (a 1 MiB work space), and with zero and
non-finite rows."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


def _system(n_aux, n_occ, n_virt):
    eps = np.concatenate([np.linspace(-20.5, -0.45, n_occ), np.linspace(0.05, 9.0, n_virt)])
    return synth.System("digits", eps, n_occ, n_aux, 0.6 / np.sqrt(n_aux), n_aux + n_virt, np.array([n_occ - 1]))


@pytest.mark.parametrize("n_aux,n_occ,n_virt,ws", [(1, 1, 1, 0), (63, 3, 11, 0), (64, 4, 32, 0), (65, 3, 43, 0),
                                                   (128, 8, 16, 0), (129, 11, 13, 0), (200, 13, 79, 1),
                                                   (257, 5, 205, 1)])
def test_polarizability_fp64(gwlib, n_aux, n_occ, n_virt, ws):
    from paper_2107_10423_gb300 import gw
    s = _system(n_aux, n_occ, n_virt)
    B, Bn = s.b_ia(), s.b_nm()
    B[:, ::7] *= 1e5                      # wide range along the rows
    if n_aux > 2:
        B[2] = 0.0
    xi = np.array([0.0, 0.3, 7.0])
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, workspace_mb=ws) as p:
        Pi = p.polarizability(xi)
    D = O.pair_energies(s.eps, s.n_occ)
    for g, x in enumerate(xi):
        w = -4.0 * D / (D * D + x * x)
        # the reference's own error: K products and sums in FP64, each within 2^-53 of the absolute terms so far
        bound = (s.n_ov + 2) * 2.0 ** -53 * ((np.abs(B) * np.abs(w)) @ np.abs(B).T) + 1e-300
        assert np.all(np.abs(Pi[g] - (B * w) @ B.T) <= bound)
        assert np.array_equal(Pi[g], Pi[g].T)


@pytest.mark.parametrize("n_aux,n_virt,ws", [(65, 20, 0), (127, 33, 0), (193, 40, 1)])
def test_w_table_fp64(gwlib, n_aux, n_virt, ws):
    from paper_2107_10423_gb300 import gw
    s = _system(n_aux, 4, n_virt)
    B, Bn = s.b_ia(), s.b_nm()
    xi, wt = O.mgl_grid(6, 0.5)
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, xi=xi, wt=wt, workspace_mb=ws) as p:
        W = p.w_table()
    ref = np.stack([O.w_corr(O.pi_imag(s.eps, s.n_occ, B, x), Bn[0].T) for x in np.append(xi, 0.0)], 1)[None]
    # |L^-1 b|^2 - |b|^2 in FP64: a few n 2^-53 of |b|^2 = 0.36 times the condition number (below 100)
    assert np.abs(W - ref).max() < n_aux * 2.0 ** -53 * 0.36 * 100


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_input_is_a_numeric_error(gwlib, bad):
    from paper_2107_10423_gb300 import gw
    s = _system(70, 4, 20)
    B, Bn = s.b_ia(), s.b_nm()
    B[31, 17] = bad
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets) as p:
        with pytest.raises(gw.GWError) as e:
            p.screening()
    assert e.value.status == gw.GW_ERR_NUMERIC


# one right-hand side, an odd few (SIMT rows), the first digit batch (16 rows: 8 right-hand sides) and a ragged larger
# one, sizes on both sides of the 2^23 multiply-add line; max_rhs_batch splits the list into batches of unequal size
@pytest.mark.parametrize("n_rhs,n_aux,n_virt,batch", [(1, 65, 20, 0), (3, 130, 33, 0), (8, 390, 150, 0),
                                                      (37, 257, 95, 0), (70, 257, 95, 33), (9, 84, 19, 4)])
def test_residues_fp64(gwlib, n_rhs, n_aux, n_virt, batch):
    from paper_2107_10423_gb300 import gw
    s = _system(n_aux, 9, n_virt)
    B, Bn = s.b_ia(), s.b_nm()
    r = np.random.default_rng(n_rhs)
    m, x = r.integers(0, s.n_bas, n_rhs), r.uniform(-0.4, 0.4, n_rhs)     # inside the gap: MINRES converges
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, minres_tol=1e-13, minres_maxit=200, minres_fallback_tol=1e-10,
                 max_rhs_batch=batch) as p:
        out = p.residues(np.zeros(n_rhs, dtype=np.int32), m, x)
    assert not out["used_fallback"].any()
    for j in range(n_rhs):
        w, dw = O.w_corr_and_deriv(O.pi_complex(s.eps, s.n_occ, B, x[j], 1e-3),
                                   O.dpi_complex(s.eps, s.n_occ, B, x[j], 1e-3), Bn[0, m[j]])
        # relative residual 1e-13 times the condition number of 1 - Pi(x) in the gap (below 100) on W and dW
        assert abs(out["w_re"][j] - w.real) < 1e-10 * max(1, abs(w))
        assert abs(out["w_im"][j] - w.imag) < 1e-10 * max(1, abs(w))
        assert abs(out["dw_re"][j] - dw.real) < 1e-9 * max(1, abs(dw))
