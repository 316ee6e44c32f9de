"""The FP64 spectral pass on a CTA cluster (N <= 8192) at every size it serves
and the first above it, against the oracle; a failed step leaves what it wrote
before alone."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import seamount_rupture
from tests.gpu_helpers import compare, gpu_for, oracle_for

pytestmark = pytest.mark.gpu


# the FP64 path's acceptance bound; the quasi-dynamic limit keeps the oracle
# quick at every N and exercises the transforms and the assembly alone, steps
# of 3 dt_min the coefficients outside the power-of-two table
@pytest.mark.parametrize("N", [16, 32, 64, 128, 256, 512, 1024, 2048, 4096, 8192, 16384])
def test_pass_matches_oracle_at_every_size(N):
    w = seamount_rupture(N=N)
    # a slip rate that varies at every N (the workload's patch lies outside the
    # shortest faults, whose shear traction would be rounding alone)
    i = np.arange(N)
    w.V_init = 1e-9 * np.exp(np.cos(2 * np.pi * i / N) + 0.5 * np.sin(6 * np.pi * i / N + 1.0))
    o, g = oracle_for(w, eta_w=0.0), gpu_for(w, eta_w=0.0)
    for m in (1, 3, 2):
        assert o.step(m) == 0
        g.step(m * g.dt_min)
    for k, e in compare(o, g).items():
        assert e < 1e-10, (k, e)
    g.close()


def test_failed_step_keeps_the_tractions_of_the_step_that_failed():
    w = seamount_rupture(N=256, amp=400.0)
    g = gpu_for(w)
    flags = 0
    for _ in range(400):
        g.enqueue(20)
        flags, _ = g.status()
        if flags:
            break
    assert flags, "the steep seamount opens"
    a = g.get_state()
    g.enqueue(5)              # every later step is a no-op
    b = g.get_state()
    for k in ("delta", "V", "theta", "tau_el", "sigma_el"):
        assert np.array_equal(a[k], b[k]), k
    g.close()
