"""The direct sum where its two-float form meets the limits of its scales (needs a
GPU), against a sum in extended precision."""
import numpy as np
import pytest

from paper_1206_1199_gb300 import ic, system as S
from test_gpu_direct import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("largest", [1e-37, 8e37, 8.6e37, 1e38, 1.8e38, 3e38])
def test_direct_sum_with_the_largest_masses(largest):
    # 2^126 is 8.507e37, 2^127 1.701e38; the tolerance of the sums at other scales:
    # 2^-46 + 2^-53 sqrt(n) of the sum of the terms' magnitudes
    n, eps = 65536, 1e-3
    pos, mass = ic.plummer(n, 73)
    mass = (mass.astype(np.float64) * (largest / float(mass.max()))).astype(np.float32)
    sub = ic.subsample(n, 5, 6)
    acc, pot = S.direct_sum(pos, mass, eps, sub)
    ra, rp, mag = reference(pos, mass, eps, sub)
    tol = 2.0 ** -46 + 2.0 ** -53 * np.sqrt(n)
    assert np.all(np.abs(acc - ra).max(1) <= tol * mag[:, 0])
    assert np.all(np.abs(pot - rp) <= tol * mag[:, 1])
