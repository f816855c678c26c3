"""The W table of mixed plans at the nodes of the grid in several chunks, as large jobs run it: three, four and about ten of
some 37 to 45 matrices at a time, with difference-form nodes on both sides of a chunk's end, against the oracle's dense
solves."""
import numpy as np
import pytest

from oracle import gw_oracle as O
from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_aux,n_freq,gap,ws,chunk", [(203, 128, 0.5, 4, 3), (203, 128, 3.0, 4, 3), (203, 128, 0.02, 6, 4),
                                                       (203, 200, 3.0, 14, 10), (150, 128, 1.0, 7, 10)])
def test_w_table_at_nodes_in_chunks(gwlib, n_aux, n_freq, gap, ws, chunk):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([[-20.5], np.linspace(-1.3, -0.45, 5), np.linspace(-0.45 + gap, 4.0, 47)])
    s = synth.System("nodes", eps, 6, n_aux, 0.6 / np.sqrt(n_aux), 11, np.array([5, 6]))
    B, Bn = s.b_ia(), s.b_nm()
    xi, wt = O.mgl_grid(n_freq, 0.5)
    ref = np.stack([np.stack([O.w_corr(O.pi_imag(s.eps, s.n_occ, B, x), Bn[t].T) for x in np.append(xi, 0.0)], 1)
                    for t in range(len(s.targets))])
    with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, precision=gw.GW_PREC_MIXED, xi=xi, wt=wt, workspace_mb=ws) as p:
        W = p.w_table()
        launches = p.stats()["launches_kernel"][0]      # a Pi launch a chunk, and one for its difference columns
    # several chunks of the nodes: more than one launch, far fewer than the grid's points in chunks of this size
    assert 3 <= launches <= 2 * (60 // chunk + 1), launches
    # as for the nodes in one chunk: BF16 hi/lo products (< 1e-6), an FP32 inverse (< 1e-5 in all), nodes 1e-7
    assert np.abs(W - ref).max() < 1e-5 * np.abs(ref).max()
