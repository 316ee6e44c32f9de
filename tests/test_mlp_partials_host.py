"""The number of partial gradients of the learned guess, and with it the order
of their sum, follows from the rows alone: no device is asked for it."""
import ctypes

import pytest

from paper_2107_03550_gb300 import sbiem


@pytest.fixture(scope="module")
def train_ctas():
    try:
        lib = sbiem.load_library()
    except ImportError:
        import __graft_entry__
        __graft_entry__.build()
        lib = sbiem.load_library()
    fn = getattr(lib, "_ZN5sbiem10train_ctasEl")          # int sbiem::train_ctas(int64_t)
    fn.restype, fn.argtypes = ctypes.c_int, [ctypes.c_int64]
    return fn


@pytest.mark.parametrize("rows,ctas", [(1, 1), (64, 1), (65, 2), (64 * 303 + 1, 304), (64 * 304 + 1, 304),
                                       (1 << 24, 304)])
def test_partial_gradients_follow_from_the_rows(train_ctas, rows, ctas):
    assert train_ctas(rows) == ctas
