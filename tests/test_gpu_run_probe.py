"""The timing probe through an adaptive run: every accepted step leaves its marks."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import rough_fault
from tests.gpu_helpers import gpu_for, rel

pytestmark = pytest.mark.gpu


# with the probe the second half steps sweep their sums: a regrouping in FP64 (tolerance of the run against its
# half steps), the same sums in FP32
@pytest.mark.parametrize("precision,tol", [(0, 1e-11), (1, 0.0)])
def test_probe_reads_a_run_without_dt_min_steps(precision, tol):
    w = rough_fault(1024, 10.0, 1e-3, seed=9, lam_min=80.0)
    a, b = gpu_for(w, precision=precision), gpu_for(w, precision=precision)
    a.probe_enable(1)
    for g in (a, b):
        taken, _, _, rc = g.run(1e9, 1e-6, m0=4, max_steps=3)
        assert rc == 0 and min(taken) > 1
    step, sweep = a.probe_read(0)
    assert 0.0 < sweep < step
    # steps of dt_min, in a run and by themselves
    for g in (a, b):
        taken, _, _, rc = g.run(1e9, 1e-6, m0=1, max_steps=2)
        assert rc == 0 and taken[0] == 1
        g.step()
    step, sweep = a.probe_read(0)
    assert 0.0 < sweep < step
    x, y = a.get_state(), b.get_state()
    for k in ("delta", "V", "theta", "tau_el", "sigma_el"):
        assert rel(x[k], y[k]) <= tol, k
    a.close()
    b.close()
