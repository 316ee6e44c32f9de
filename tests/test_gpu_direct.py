"""The direct form of the history sweep (FP64 handles, FP32 handles above
N = 16384, ensembles) against the bulk-async form of the same handle, which a
copy-wait limit of the caller's selects: uneven windows, two cutting planes,
steps past the short windows, ring heads anywhere, streamed and table weights."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import large_fault, random_history, seamount_rupture
from tests.gpu_helpers import gpu_for, rel

pytestmark = pytest.mark.gpu


# FP64 sums of up to 4 N products in another order: 4 N eps = 6e-11 at the
# worst, of terms that mostly cancel; FP32 form: as the oracle parity tests
# (weights and products rounded to FP32 once)
@pytest.mark.parametrize("N,precision,kw,tol", [
    (16, 0, {}, 1e-12), (256, 0, dict(kc_L=151.3, kcN_L=93.7), 1e-12), (2048, 0, dict(kc_L=233.0), 1e-12),
    (32768, 1, {}, 2e-6), (32768, 1, dict(kc_L=120.5, kcN_L=201.0), 2e-6), (32768, 1, dict(quadrature=1), 2e-6)])
def test_direct_sums_match_the_bulk_async_form(N, precision, kw, tol):
    w = large_fault(N=N, dx=4.0) if N > 16384 else seamount_rupture(N=N)
    g = gpu_for(w, precision=precision, **kw)
    R = np.maximum(g.windows() - 1, 0)
    HT, HN, _ = random_history(R, 41, 1e-3)
    g.set_history(HT, HN)
    for k, m in enumerate((1, 3, 255, 256, int(R.max()), int(R.max()) + 1, 1 << 30)):
        if k == 2:
            g.step()              # every ring head moves off zero (the rings wrap)
            assert g.status()[0] == 0
        direct = g.history_sums(m)
        g.set_wait_limit(1 << 22 | 1)
        bulk = g.history_sums(m)
        g.set_wait_limit()
        for a, b in zip(direct, bulk):
            assert rel(a, b) <= tol, (m, rel(a, b))
    g.close()


def test_sweep_mark_without_history():
    # the quasi-dynamic limit has nothing to sweep: the mark between sweep and
    # finish is recorded all the same
    import torch
    g = gpu_for(seamount_rupture(N=256), eta_w=0.0)
    st = torch.cuda.current_stream()
    g.set_stream(st)
    a, b, c = (torch.cuda.Event(enable_timing=True) for _ in range(3))
    b.record()
    torch.cuda.synchronize()
    a.record()
    g.history_enqueue(1, sweep_done=b)
    c.record()
    torch.cuda.synchronize()
    assert a.elapsed_time(b) >= 0.0 and b.elapsed_time(c) >= 0.0
    g.close()
