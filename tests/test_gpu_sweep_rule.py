"""One rule says which form the history sweep takes, and the reports follow it:
a caller's copy-wait limit brings the bulk-async form with its own grid, table
error and streamed weights, and the default limit takes it back."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import large_fault, seamount_rupture
from tests.gpu_helpers import gpu_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision", [(256, 0), (32768, 1)])
def test_reports_follow_the_wait_limit(N, precision):
    g = gpu_for(large_fault(N=N, dx=4.0) if N > 16384 else seamount_rupture(N=N), precision=precision)
    slots = g.history_size()
    direct, bytes_direct = g.get_sweep(), g.footprint()[0]
    assert direct["shape"] == 3 and direct["ctas_per_sm"] == 1 and direct["lag_ctas_per_sm"] == 1
    # FP64 streams every weight (32 + 16 B a slot), FP32 none (16 B a slot)
    assert bytes_direct == (48 * slots if precision == 0 else 16 * slots)
    g.set_wait_limit((1 << 22) + 1)
    bulk, bytes_bulk = g.get_sweep(), g.footprint()[0]
    assert bulk["ctas_per_sm"] > 1                         # 512-thread CTAs of the direct form: one an SM
    if precision == 0:
        assert bytes_bulk == 48 * slots and bulk["table_err"] == -1.0
    else:
        # modes with ds = c_s k dt_min up to 1/64 evaluate their weights on chip, the others stream them
        R = np.maximum(g.windows() - 1, 0)
        ds = 2 * np.pi * np.arange(R.size) / N * 0.25
        assert bytes_bulk == 16 * slots + 8 * int(R[ds > 1 / 64].sum()) > bytes_direct
        assert 0 < bulk["table_err"] != direct["table_err"]
    g.step()
    g.set_wait_limit()
    assert g.get_sweep() == direct and g.footprint()[0] == bytes_direct
    g.step()
    g.close()
