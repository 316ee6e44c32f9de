"""The adaptive run where the whole step of an attempt is rejected by its status
word (no friction solution, opening) while its half steps go on beside it, at
sizes of every pass form: nothing of the attempt remains, and the state is that
of the accepted half steps taken one by one."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import seamount_rupture
from tests.gpu_helpers import gpu_for, rel

pytestmark = pytest.mark.gpu


# FP32: every sum as a single step forms it, bitwise; FP64: the second half
# step's sums are regrouped, some 10 eps of tractions up to 1e8 Pa, which moves
# ln V by 2e-13 (a sigma = 5e5 Pa), and with it the ring's newest slots
@pytest.mark.parametrize("N,precision,tol", [(256, 0, 1e-10), (2048, 1, 0.0), (16384, 0, 1e-10), (32768, 1, 0.0)])
def test_flagged_whole_step_leaves_nothing_behind(N, precision, tol):
    w = seamount_rupture(N=N, amp=200.0)
    a, b = gpu_for(w, precision=precision), gpu_for(w, precision=precision)
    m0 = 1 << 16
    assert b.try_step(m0 * b.dt_min) in (-4, -5)          # the first whole step fails; b stays at its start
    # no error bound: every rejection on the way down is one of the status word, the last of them (unless the
    # second half step fails too) with a first half step that is sound by itself
    taken, _, t, rc = a.run(1e9, 1e30, m0=m0, max_steps=1)
    assert rc == 0 and len(taken) == 1 and taken[0] < m0
    assert a.status()[0] == 0
    for m in taken:
        for _ in range(1 if m == 1 else 2):
            b.step(max(m // 2, 1) * b.dt_min)
    x, y = a.get_state(), b.get_state()
    assert abs(x["t"] - y["t"]) <= 1e-12 * y["t"] and abs(t - y["t"]) <= 1e-12 * y["t"]
    for k in ("delta", "V", "theta", "tau_el", "sigma_el"):
        assert rel(x[k], y[k]) <= tol, (k, rel(x[k], y[k]))
    for u, v in zip(a.get_history(), b.get_history()):
        assert np.abs(u - v).max() <= tol * np.abs(v).max()
    a.close()
    b.close()
