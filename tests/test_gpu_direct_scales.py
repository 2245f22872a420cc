"""The direct sum where its two-float form meets the limits of its scales (needs a
GPU), against a sum in extended precision."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1206_1199_gb300 import _lib as L
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


@pytest.mark.parametrize("n", [65535, 65536])
def test_direct_sum_of_sources_at_an_odd_start(n):
    # sources that start on an 8-byte boundary only: the same bytes
    L.load()
    pos, mass = ic.plummer(n, 74)
    sub = ic.subsample(n, 40, 6)
    want = S.direct_sum(pos, mass, 1e-3, sub)
    src = S._particle_sources(pos, mass, "cuda")
    moved = torch.empty(src.numel() + 8, dtype=torch.uint8, device="cuda")[8:]
    moved.copy_(src)
    t = torch.from_numpy(np.ascontiguousarray(sub, np.int64)).to("cuda")
    scratch = torch.empty(4 * int(L.load().otoo_direct_chunks(n, 40)) * 40, dtype=torch.float64, device="cuda")
    acc = torch.empty((40, 3), dtype=torch.float64, device="cuda")
    pot = torch.empty(40, dtype=torch.float64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    L.call("otoo_direct", moved.data_ptr(), n, t.data_ptr(), 40, 1e-3 ** 2, acc.data_ptr(), pot.data_ptr(),
           scratch.data_ptr(), status.data_ptr(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    np.testing.assert_array_equal(acc.cpu().numpy(), want[0])
    np.testing.assert_array_equal(pot.cpu().numpy(), want[1])
