"""The weights the direct sweep evaluates on chip, read out one lag per mode (a
ring with a single slot of 1 sums to its weight), against 64 bits: no further
off than weights stored in FP32, which round once."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import large_fault
from tests.gpu_helpers import gpu_for

pytestmark = pytest.mark.gpu


def _read_out(g, seed):
    """Per mode (with history) a random lag's weights (shear, normal), their s and FP64 values."""
    from paper_2107_03550_gb300.sbiem import kernel_values
    p = g.params
    R = np.maximum(g.windows() - 1, 0)
    off = np.concatenate([[0], np.cumsum(R)[:-1]])
    n = np.flatnonzero(R)
    i = np.random.default_rng(seed).integers(0, R[n])
    H = np.zeros(int(R.sum()), dtype=np.complex128)
    H[off[n] + i] = 1.0
    g.set_history(H, H)
    m = 1
    ds = p.cs * (2 * np.pi * n / (p.N * p.dx)) * g.dt_min
    ref = np.stack(kernel_values((i + m + 0.5) * ds, p.cs / p.cp)) * g.dt_min
    got = np.stack([x[n].real for x in g.history_sums(m)])
    return ds, got, ref


# a stored weight's error is its rounding, uniform in +-1/2 ulp; the table's adds the rounding of the polynomial's
# varying part (up to 0.06 of the weight's scale, five operations) and 1e-8 of the table: in quadrature below 2 % of
# the rms (16384 modes x 4 draws: the sample's own scatter is below 1 %), and at most a fifth of an ulp at max|C|
def test_table_weights_round_as_stored_ones():
    g = gpu_for(large_fault(N=32768, dx=4.0), precision=1)
    assert g.get_sweep()["gen_ds_max"] > 0
    got, ref = [], []
    for seed in range(4):
        _, w, r = _read_out(g, seed)
        got.append(w)
        ref.append(r)
    got, ref = np.concatenate(got, 1), np.concatenate(ref, 1)
    stored = ref.astype(np.float32)
    for w, r, st in zip(got, ref, stored):
        assert np.sqrt(np.mean((w - r) ** 2)) <= 1.05 * np.sqrt(np.mean((st - r) ** 2))
    scale = np.abs(ref).max()
    assert np.abs(got - ref).max() <= np.abs(stored - ref).max() + 0.2 * 2.0 ** -24 * scale
    g.close()


# the table's error grows like (c_p/c_s)^5: where it would show, the sweep keeps the bulk-async form, whose modes with
# ds = c_s k dt_min above 1/64 read stored weights (the library's FP64 route is good to 1e-13)
@pytest.mark.parametrize("ratio,table", [(1.2, True), (2.0, True), (3.0, False), (5.0, False)])
def test_table_serves_only_where_it_is_as_good(ratio, table):
    w = large_fault(N=32768, dx=4.0)
    g = gpu_for(w, precision=1, cp=ratio * w.cs)
    sw = g.get_sweep()
    assert sw["gen_ds_max"] > 0 and (sw["ctas_per_sm"] == 1) == table
    if table:
        assert 0 < sw["table_err"] <= 1e-8
    ds, got, ref = _read_out(g, 7)
    high = ds > 1 / 64
    for x, r in zip(got[:, high], ref[:, high]):
        stored = np.sqrt(np.mean((r.astype(np.float32) - r) ** 2))
        # 16000 draws of a rounding error; the table: 2 % on top and up to 1e-8 of max|C| for c_p = 2 c_s
        assert np.sqrt(np.mean((x - r) ** 2)) <= (1.01 * stored if not table else
                                                  1.05 * stored + 1e-8 * np.abs(ref).max())
    g.close()


def test_ensemble_shares_the_table_only_where_it_serves():
    from paper_2107_03550_gb300.sbiem import Batch
    from paper_2107_03550_gb300.workloads import seamount_rupture
    for ratio, direct in ((1.7320508, True), (5.0, False)):
        w = seamount_rupture(N=1024)
        mem = [gpu_for(w, precision=1, cp=ratio * w.cs) for _ in range(2)]
        solo = gpu_for(w, precision=1, cp=ratio * w.cs)
        b = Batch(mem)
        sw = b.get_sweep()
        assert sw["shape"] == 3 and sw["gen_ds_max"] > 0 and (sw["ctas_per_sm"] == 1) == direct
        b.enqueue(3)
        solo.enqueue(3)
        assert not b.status()[0].any() and solo.status()[0] == 0
        u, v = mem[1].get_state(), solo.get_state()
        # three steps on an empty history: FP32 sums grouped in another way
        for k in ("delta", "V", "theta"):
            assert np.abs(u[k] - v[k]).max() <= 1e-5 * np.abs(v[k]).max(), k
        b.close()
