"""A job that fails in mixed precision is solved again in FP64, and its result and the run's summary say so and why."""
import numpy as np
import pytest

from paper_2107_10423_gb300 import serve, synth


@pytest.mark.parametrize("fails", [(), ("mixed",), ("mixed", "fp64")])
def test_retry_is_reported(monkeypatch, fails):
    from paper_2107_10423_gb300 import gw

    class Plan:
        def __init__(self, *a, precision=None, **kw):
            self.name = "mixed" if precision == gw.GW_PREC_MIXED else "fp64"

        def __enter__(self):
            return self

        def __exit__(self, *a):
            pass

        def screening(self):
            if self.name in fails:
                raise gw.GWError(gw.GW_ERR_CUDA, f"launch failed in {self.name}")

        def qp_solve(self, mode):
            return np.zeros(1), np.ones(1), np.zeros(1, dtype=int)

    monkeypatch.setattr(gw, "Plan", Plan)
    s = synth.water_cluster(1, 1, targets="homo_lumo")
    job = serve.Job(7, 0.0, s, np.zeros((1, 1)), np.zeros((1, 1, 1)))
    job.result = r = serve.run_job(job)
    summary = serve.summarize([job], makespan=1.0)
    if not fails:
        assert r["precision"] == "mixed" and "mixed_error" not in r and summary["mixed_errors"] == {}
        return
    assert "launch failed in mixed" in r["mixed_error"]
    assert list(summary["mixed_errors"]) == [7]
    if len(fails) == 2:
        assert "launch failed in fp64" in r["error"] and summary["completed"] == 0
    else:
        assert r["precision"] == "fp64" and "error" not in r and summary["fp64_fallbacks"] == 1
