"""The three-launch FP32 spectral pass (N > 16384), a template instance of its
own at every size, against the oracle: two steps without history on a slip rate
and a curvature that excite every mode alike."""
import numpy as np
import pytest

from paper_2107_03550_gb300.workloads import seamount_rupture
from tests.gpu_helpers import gpu_for, oracle_for

pytestmark = pytest.mark.gpu


# An FP32 transform's rounding is white over the modes, at most lg N roundings of the input's rms in each: the shear
# traction multiplies what the forward one adds to the slip by S k, k <= pi/dx (rms over the modes k_max / sqrt 3),
# the normal traction by S; the inverse adds its own to both, on the scale of tau + i sigma.  Eight times the rms of
# both covers the largest of 2^20 elements (5.3 sigma); the tractions themselves are some 1e4 times that.
@pytest.mark.parametrize("lgN", [15, 16, 17, 18, 19, 20])
def test_tractions_match_the_oracle(lgN):
    N = 1 << lgN
    w = seamount_rupture(N=N)
    rng = np.random.default_rng(lgN)
    w.V_init = 1e-9 * np.exp(0.5 * rng.standard_normal(N))
    w.kappa = 0.05 * rng.standard_normal(N)
    o, g = oracle_for(w, eta_w=0.0), gpu_for(w, precision=1, eta_w=0.0)
    for _ in range(2):
        assert o.step() == 0
        g.step()
    s = g.get_state()
    t, eps = 2 * w.dt_min, 2.0 ** -24
    S = w.mu * (1 - (w.cs / w.cp) ** 2)
    rms = lambda x: float(np.sqrt(np.mean(np.abs(x) ** 2)))
    forward = lgN * eps * rms(w.V_init * (1 + 1j * w.kappa)) * S * t
    inverse = lgN * eps * rms(o.last["tau_el"] + 1j * o.last["sig_el"])
    for k, ref, f in (("tau_el", o.last["tau_el"], np.pi / w.dx / np.sqrt(3.0)), ("sigma_el", o.last["sig_el"], 1.0)):
        bound = 8 * (forward * f + inverse)
        assert bound < 1e-3 * rms(ref)
        assert np.abs(s[k] - ref).max() <= bound, (k, np.abs(s[k] - ref).max(), bound)
    g.close()
