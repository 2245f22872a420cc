"""The learned angle's choice at the edges of its early end (needs a GPU):
grids of odd and even length, of one angle, not increasing, weights and
statistics outside the range in which the search may end early, against a plain
evaluation of every angle."""
import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import mlp

pytestmark = pytest.mark.gpu


def every_angle(net, feats, count, grid, target, theta0, fallback):
    """The rule with every prediction taken by the library's forward kernel."""
    g, k = len(feats), len(grid)
    rows = np.concatenate([np.repeat(feats, k, 0), np.tile(np.asarray(grid, np.float32), g)[:, None]], 1)
    with np.errstate(all="ignore"):
        y = net.predict(rows).reshape(g, k)
    th, tg = net.learned_theta(feats, count, grid, target, theta0, fallback)
    gv = np.asarray(grid, np.float32)
    with np.errstate(invalid="ignore"):
        ok = y <= tg[:, None]
    want = np.maximum(np.where(ok, gv[None], gv[0]).max(1), gv[0])
    want[np.isnan(tg) | ~np.isfinite(y).all(1)] = fallback
    return th, want


@pytest.mark.parametrize("grid", [(0.7,), (0.5, 0.9), tuple(0.3 + 0.1 * k for k in range(13)), (0.9, 0.4, 1.2, 0.4)])
@pytest.mark.parametrize("n", [1, 7, 8, 9, 500, 9501, 38001])
@pytest.mark.parametrize("case", ["plain", "large_weight", "large_input", "nan_weight"])
def test_choice_equals_the_evaluation_of_every_angle(grid, n, case):
    L.load()
    rng = np.random.Generator(np.random.PCG64(n))
    w = mlp.init_weights(3)
    w[-1] = -3.0
    if case == "large_weight":
        w[5] = 3e38  # the angle's weight of the first hidden unit: its sum overflows
    elif case == "nan_weight":
        w[40] = np.nan
    net = mlp.ThetaNet(w, calib=1.0)
    feats = rng.standard_normal((n, 5)).astype(np.float32)
    if case == "large_input":
        feats[::3, 2] = 1e30
    count = rng.integers(1, 65, n).astype(np.int32)
    th, want = every_angle(net, feats, count, grid, 1e-3, 0.9, 0.55)
    np.testing.assert_array_equal(th, want)
