"""The three-launch FP32 spectral pass (N > 16384) in an ensemble, at both of
its shapes (N1 = 2 N2 and N1 = N2); test_gpu_large.py compares it with the
oracle at the same sizes."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import seamount_rupture
from tests.gpu_helpers import gpu_for, rel

pytestmark = pytest.mark.gpu


def _workload(N, k):
    w = seamount_rupture(N=N)
    i = np.arange(N)
    w.V_init = 1e-9 * np.exp(np.cos(2 * np.pi * i / N + k) + 0.5 * np.sin(400 * np.pi * i / N))
    return w


# the same kernels on the same inputs: rounding of the launch order only
def test_ensemble_members_step_as_alone():
    from paper_2107_03550_gb300.sbiem import Batch
    ws = [_workload(N, k) for N, k in ((32768, 0.1), (65536, 0.2), (32768, 0.3))]
    solo = [gpu_for(w, precision=1, eta_w=0.0) for w in ws]
    mem = [gpu_for(w, precision=1, eta_w=0.0) for w in ws]
    b = Batch(mem)
    b.enqueue(3)
    assert not b.status()[0].any()
    for x, y in zip(solo, mem):
        x.enqueue(3)
        u, v = x.get_state(), y.get_state()
        for k in ("delta", "V", "theta", "tau_el", "sigma_el"):
            assert rel(v[k], u[k]) <= 1e-6, k
    b.close()
