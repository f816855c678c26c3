"""The W table of FP64 plans on digit products repeats itself bit for bit: the tiles' sums of squares are added in a fixed
order (roots of the QP search move with that order near poles of Sigma)."""
import numpy as np
import pytest

from paper_2107_10423_gb300 import synth

pytestmark = pytest.mark.gpu


# five and nine column tiles of 32 (the last ragged), and rows and matrices in blocks (1 MiB of work space)
@pytest.mark.parametrize("n_aux,ws", [(129, 0), (257, 0), (257, 1)])
def test_fp64_table_repeats(gwlib, n_aux, ws):
    from paper_2107_10423_gb300 import gw
    eps = np.concatenate([np.linspace(-20.5, -0.45, 5), np.linspace(0.05, 9.0, 61)])
    s = synth.System("repeat", eps, 5, n_aux, 0.6 / np.sqrt(n_aux), 3, np.array([2, 3, 4, 5]))
    B, Bn = s.b_ia(), s.b_nm()
    tables = []
    for _ in range(4):
        with gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, workspace_mb=ws) as p:
            tables.append(p.w_table())
    for t in tables[1:]:
        assert np.array_equal(t, tables[0])
