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
