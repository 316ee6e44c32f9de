"""A caller's allocator of any alignment: the library aligns its arrays itself
(the FP64 sweep reads a ring slot by one 32-byte load)."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import random_history, seamount_rupture
from tests.gpu_helpers import gpu_for

pytestmark = pytest.mark.gpu


# the same kernels on the same values: bitwise
@pytest.mark.parametrize("off", [0, 16, 48])
@pytest.mark.parametrize("precision", [0, 1])
def test_results_do_not_depend_on_the_allocators_alignment(precision, off):
    import torch
    held, sizes = {}, []

    def alloc(n):
        t = torch.empty(n + off, dtype=torch.uint8, device="cuda")
        held[t.data_ptr() + off] = t
        sizes.append(n)
        return t.data_ptr() + off

    def free(ptr):
        held.pop(ptr)

    w = seamount_rupture(N=256)
    a, b = gpu_for(w, precision=precision), gpu_for(w, precision=precision, allocator=(alloc, free))
    assert len(held) == len(sizes) - (off > 0)             # one misaligned block, given back
    HT, HN, _ = random_history(np.maximum(a.windows() - 1, 0), 5, 1e-6)
    for g in (a, b):
        g.set_history(HT, HN)
        g.enqueue(3)
        assert g.status()[0] == 0
    for x, y in zip(a.history_sums(1), b.history_sums(1)):
        assert np.array_equal(x, y)
    u, v = a.get_state(), b.get_state()
    for k in u:
        assert np.array_equal(u[k], v[k]), k
    a.close()
    b.close()
    assert not held
