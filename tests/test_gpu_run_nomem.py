"""The adaptive run where its buffers cannot be had: the call is refused, what
it allocated is given back, steps go on, and a later call runs."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import rough_fault
from tests.gpu_helpers import gpu_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_run_refused_for_memory_can_be_tried_again(precision):
    import torch
    from paper_2107_03550_gb300.sbiem import SbiemError
    held, left = {}, [None]

    def alloc(n):
        if left[0] is not None:
            if left[0] == 0:
                return 0
            left[0] -= 1
        t = torch.empty(n, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    w = rough_fault(1024, 10.0, 1e-3, seed=9, lam_min=80.0)
    a, b = gpu_for(w, precision=precision), gpu_for(w, precision=precision, allocator=(alloc, held.pop))
    before, size = dict(held), b.footprint()[1]
    for k in (0, 2, 4, 7, 12, 16):                # refused at the snapshot, at the staging
        left[0] = k
        with pytest.raises(SbiemError) as e:
            b.run(1e9, 1e-7, m0=4, max_steps=3)
        assert e.value.code == -2
        # the snapshot (four blocks) may stay once it is whole
        kept = 4 if k >= 4 else 0
        assert len(held) == len(before) + kept, (k, len(held) - len(before))
    size_snap = b.footprint()[1]
    assert size < size_snap
    left[0] = 16
    with pytest.raises(SbiemError):
        b.run(1e9, 1e-7, m0=4, max_steps=3)
    assert b.footprint()[1] == size_snap
    left[0] = None
    for g in (a, b):
        g.step()
        taken, _, _, rc = g.run(1e9, 1e-7, m0=4, max_steps=6)
        assert rc == 0 and len(taken) == 6
    x, y = a.get_state(), b.get_state()
    for k in x:
        assert np.array_equal(x[k], y[k]), k
    a.close()
    b.close()
    assert not held
