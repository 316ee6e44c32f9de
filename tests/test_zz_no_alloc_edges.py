"""Chunk table of the allocation-free convolution at the edges of its blocks
of 1024 modes, and the refusal of a history past the table."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _call(torch, R, precision, m, seed=5):
    from paper_2107_03550_gb300.sbiem import history_sums_noalloc
    rng = np.random.default_rng(seed)
    R = np.asarray(R, dtype=np.int64)
    M = np.where(R > 0, R + 1, 0)
    ft = torch.float64 if precision == 0 else torch.float32
    off = lambda v: np.concatenate([[0], np.cumsum(v)[:-1]])
    head = np.where(R > 0, rng.integers(0, np.maximum(R, 1)), 0)
    ring = rng.standard_normal((max(int(R.sum()), 1), 4))
    wts = rng.standard_normal((max(int(M.sum()), 1), 2))
    d = lambda v, t: torch.tensor(v, dtype=t, device="cuda").contiguous()
    b = dict(ring=d(ring, ft), weights=d(wts, ft), ring_off=d(off(R), torch.int64), w_off=d(off(M), torch.int64),
             R=d(R, torch.int32), M=d(M, torch.int32), head=d(head, torch.int32),
             AT=torch.full((R.size, 2), 7.0, dtype=torch.float64, device="cuda"),
             AN=torch.full((R.size, 2), 7.0, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    try:
        history_sums_noalloc(R.size, precision, m, *(b[k].data_ptr() for k in (
            "ring", "weights", "ring_off", "w_off", "R", "M", "head", "AT", "AN")))
    finally:
        torch.cuda.synchronize()
        out = np.concatenate([b["AT"].cpu().numpy(), b["AN"].cpu().numpy()], axis=1)
        _call.out = out
    ring, wts = b["ring"].cpu().numpy().astype(np.float64), b["weights"].cpu().numpy().astype(np.float64)
    ro, wo = off(R), off(M)
    ref = np.zeros((R.size, 4))
    size = np.zeros(R.size)
    for n in np.flatnonzero(R + 1 > m):
        i = np.arange(R[n] + 1 - m)
        s = ring[ro[n] + (head[n] + i) % R[n]]
        w = wts[wo[n] + m + i]
        ref[n] = (s * w[:, [0, 0, 1, 1]]).sum(axis=0)
        size[n] = (np.abs(s) * np.abs(w[:, [0, 0, 1, 1]])).sum(axis=0).max()
    return out, ref, size


# |error| <= products x eps x sum of their magnitudes, per mode (at most 4100
# products here; blocked FP32 sums stay far below it)
@pytest.mark.parametrize("precision,eps", [(0, 1.2e-16), (1, 6.0e-8)])
@pytest.mark.parametrize("nmodes", [1, 2, 1023, 1024, 1025, 4097])
def test_sums_at_block_edges(nmodes, precision, eps):
    import torch
    rng = np.random.default_rng(nmodes)
    R = rng.choice([0, 1, 2, 31, 255, 2047, 2048, 2049, 4100], size=nmodes, p=[.2, .1, .1, .2, .3, .03, .03, .02, .02])
    R[-1] = 2049
    for m in (1, 2, 300):
        out, ref, size = _call(torch, R, precision, m)
        assert np.all(np.abs(out - ref).max(axis=1) <= 4100 * eps * size), m


def test_history_past_the_chunk_table_is_refused_untouched():
    import torch

    from paper_2107_03550_gb300.sbiem import SbiemError
    # 65537 one-slot modes are too many modes; 32769 modes of 2049 slots have 65538 chunks
    with pytest.raises(SbiemError) as ei:
        _call(torch, np.full(32769, 2049), 1, 1)
    assert ei.value.code == -1
    assert np.all(_call.out == 7.0)
    out, ref, _ = _call(torch, np.full(3, 5), 1, 1)   # and the next call works
    assert np.allclose(out, ref, atol=1e-5)
