"""Gradient of the learned guess at the edges of its 64-row tiles and of its
CTAs' tile loops, against the FP64 oracle."""
import numpy as np
import pytest

from oracle.mlp import N_PARAMS, loss_and_grad

pytestmark = pytest.mark.gpu


# targets far from the outputs (residuals near 10 against outputs of order 1),
# so that even a single row's loss and gradient carry the relative error of an
# FP32 forward pass, a few 1e-6 after sums of 64 products: 1e-5 on the loss,
# 1e-4 of the largest entry on the gradient (as at 1000 rows)
@pytest.mark.parametrize("rows", [1, 63, 64, 65, 128 * 152 + 1, 60000])
def test_gradient_matches_oracle_at_tile_edges(rows):
    from paper_2107_03550_gb300.sbiem import mlp_grad
    rng = np.random.default_rng(900 + rows)
    theta = rng.normal(0, 0.2, N_PARAMS).astype(np.float32)
    X = rng.normal(0, 1, (rows, 5)).astype(np.float32)
    t = rng.normal(10, 1, rows).astype(np.float32)
    loss, g = mlp_grad(theta, X, t)
    loss_o, g_o = loss_and_grad(theta.astype(np.float64), X.astype(np.float64), t.astype(np.float64))
    assert abs(loss - loss_o) <= 1e-5 * loss_o
    assert np.abs(g - g_o).max() <= 1e-4 * np.abs(g_o).max()
