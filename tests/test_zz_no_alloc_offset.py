"""The allocation-free convolution into outputs aligned as their type (double)
asks and no more: with and without history, the sums of aligned outputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("slots", [0, 1, 2049])
def test_outputs_of_eight_byte_alignment(precision, slots):
    import torch

    from paper_2107_03550_gb300.sbiem import history_sums_noalloc
    nmodes = 1025
    rng = np.random.default_rng(slots)
    R = np.full(nmodes, slots)
    R[::3] = 0
    M = np.where(R > 0, R + 1, 0)
    ft = torch.float64 if precision == 0 else torch.float32
    off = lambda v: np.concatenate([[0], np.cumsum(v)[:-1]])
    d = lambda v, t: torch.tensor(v, dtype=t, device="cuda").contiguous()
    args = [d(rng.standard_normal((max(int(R.sum()), 1), 4)), ft), d(rng.standard_normal((max(int(M.sum()), 1), 2)), ft),
            d(off(R), torch.int64), d(off(M), torch.int64), d(R, torch.int32), d(M, torch.int32),
            torch.zeros(nmodes, dtype=torch.int32, device="cuda")]
    got = []
    for shift in (0, 1):
        out = [torch.full((2 * nmodes + 2,), 7.0, dtype=torch.float64, device="cuda") for _ in range(2)]
        assert out[0].data_ptr() % 16 == 0
        torch.cuda.synchronize()
        history_sums_noalloc(nmodes, precision, 1, *(a.data_ptr() for a in args), *(o.data_ptr() + 8 * shift for o in out))
        torch.cuda.synchronize()
        for o in out:
            # nothing beside the outputs is written
            assert torch.all(o[:shift] == 7.0) and torch.all(o[2 * nmodes + shift:] == 7.0)
        got.append([o[shift:shift + 2 * nmodes].cpu().numpy().reshape(-1, 2) for o in out])
    for x, y in zip(*got):
        assert np.array_equal(x, y)                       # the same sums in the same order
        assert np.all(x[R == 0] == 0.0)
