"""gw_plan_footprint bounds the device bytes of a plan whatever is called on it: small work spaces (many buffers of a few
MiB), both precisions, residue lists that grow, the dense fallback and Sigma evaluations."""
import numpy as np
import pytest

from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_aux,n_occ,n_virt,n_t,ws,n_freq", [
    ("fp64", 1117, 39, 195, 9, 53, 42), ("fp64", 248, 18, 12, 4, 1, 105), ("fp64", 370, 10, 196, 8, 8, 104),
    ("mixed", 126, 5, 38, 2, 1, 128), ("mixed", 332, 49, 214, 2, 92, 61), ("mixed", 929, 40, 161, 9, 9, 87)])
def test_footprint_bounds_every_call(gwlib, prec, n_aux, n_occ, n_virt, n_t, ws, n_freq):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([np.linspace(-1.4, -0.45, n_occ), np.linspace(0.05, 4.0, n_virt)])
    s = synth.System("bound", eps, n_occ, n_aux, 0.6 / np.sqrt(n_aux), 5, np.arange(n_t))
    B, Bn = s.b_ia(), s.b_nm()
    kw = dict(precision=gw.GW_PREC_FP64 if prec == "fp64" else gw.GW_PREC_MIXED, workspace_mb=ws, n_freq=n_freq)
    bound = gw.footprint(s.n_occ, s.n_virt, s.n_aux, n_t, **kw)
    r = np.random.default_rng(n_aux)
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, **kw) as p:
        p.screening()
        for k in (1, 2, 5, 11, 30, 77, 200):
            k = min(k, n_t * s.n_bas)
            p.residues(r.integers(0, n_t, k), r.integers(0, s.n_bas, k), r.uniform(-3.0, 3.0, k))
        p.sigma_cd(s.eps[s.targets] - 0.03)
        st = p.stats()
    assert st["n_fallback"] > 0
    assert st["bytes_device_peak"] <= bound, (st["bytes_device_peak"], bound)
