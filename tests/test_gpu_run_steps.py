"""The adaptive run against single steps: the state of a run is that of its
accepted half steps taken one by one, at sizes of every pass form."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import rough_fault
from tests.gpu_helpers import gpu_for, rel

pytestmark = pytest.mark.gpu


# FP32: the run sweeps every sum as a single step does, so the states agree
# bitwise; FP64: its second half steps take their sums from the whole step's
# (another grouping), a few 1e-15 a step
@pytest.mark.parametrize("N,precision,tol", [(256, 0, 1e-11), (2048, 1, 0.0), (16384, 0, 1e-11), (32768, 1, 0.0)])
def test_run_equals_its_half_steps(N, precision, tol):
    w = rough_fault(N, 10.0, 1e-3, seed=9, lam_min=80.0)
    a, b = gpu_for(w, precision=precision), gpu_for(w, precision=precision)
    rejected = 0
    for eps0, steps in ((1e-7, 9), (1e-12, 3), (1e-6, 6)):   # the second call rejects its way down to dt_min
        taken, m_next, t, rc = a.run(1e9, eps0, m0=64 if eps0 == 1e-12 else 1, max_steps=steps)
        assert rc == 0 and len(taken) == steps
        rejected += eps0 == 1e-12 and max(taken) < 64
        for m in taken:
            for _ in range(1 if m == 1 else 2):
                b.step(max(m // 2, 1) * b.dt_min)
    assert rejected
    x, y = a.get_state(), b.get_state()
    assert abs(x["t"] - y["t"]) <= 1e-12 * y["t"]
    for k in ("delta", "V", "theta", "tau_el", "sigma_el"):
        assert rel(x[k], y[k]) <= tol, (k, rel(x[k], y[k]))
    for u, v in zip(a.get_history(), b.get_history()):
        assert np.abs(u - v).max() <= tol * np.abs(v).max()
    a.close()
    b.close()
