"""Gradient of the network where a weight has overflowed (needs a GPU)."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_1206_1199_gb300 import _lib as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 100, 127, 128, 129, 1000])
def test_gradient_with_an_infinite_first_layer_weight(n):
    # an infinite weight saturates its hidden unit for every row; the last block's
    # places past the last row have no part in the sums, so these stay finite
    L.load()
    from paper_1206_1199_gb300 import mlp
    w = mlp.init_weights(4)
    w[3] = np.inf  # unit 0, input 3
    net = mlp.ThetaNet(w)
    rng = np.random.default_rng(9)
    x = rng.normal(size=(n, 6)).astype(np.float32)
    t = np.sin(x[:, 0]).astype(np.float32)
    g, loss = net.grad(x, t)
    wb = omlp.bf16_round(net.weights())
    xs = (x.astype(np.float64) - net.mean) / net.std
    gr = omlp.grad(wb, xs, t)
    assert np.isfinite(gr).all()
    assert np.abs(g - gr).max() <= 1e-4 * np.abs(gr).max()
    assert abs(loss - omlp.loss(wb, xs, t)) <= 1e-4 * omlp.loss(wb, xs, t)
