"""The FP64 direct sum on both sides of its size rule and at the limits of the
two-float form (needs a GPU), against a sum in extended precision."""
import ctypes

import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


def reference(pos, mass, eps, targets):
    """Accelerations, potentials and the sums of the terms' magnitudes in
    extended precision (long double)."""
    ld = np.longdouble
    p, m, e2 = pos.astype(ld), mass.astype(ld), ld(float(eps) ** 2)
    acc, pot, mag = [], [], []
    for i in targets:
        d = [p[:, k] - p[i, k] for k in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2] + e2
        q = 1 / np.sqrt(r2)
        w = m * q
        w[i] = 0
        g = w * q * q
        acc.append([np.sum(g * d[k]) for k in range(3)])
        pot.append(-np.sum(w))
        mag.append((np.sum(g * np.sqrt(r2 - e2)), np.sum(w)))
    return np.array(acc, ld), np.array(pot, ld), np.array(mag, ld)


@pytest.mark.parametrize("n,n_tgt", [(65535, 1), (65536, 1), (65536, 257), (65537, 256), (70001, 129)])
@pytest.mark.parametrize("scale", ["unit", "offset", "large", "small", "tiny_eps"])
def test_direct_sum_at_the_two_float_rule(n, n_tgt, scale):
    # pairs of relative error 2^-47 (two-float) or a few 2^-53 (FP64) and the
    # rounding of sums of n terms in FP64 runs of at most a chunk: within
    # 2^-46 + 2^-53 sqrt(n) of the sum of the terms' magnitudes
    pos, mass = ic.plummer(n, 71)
    eps = 1e-3
    if scale == "offset":
        pos = pos + np.array([3e4, -2e4, 1e4])
    elif scale == "large":
        pos, mass, eps = pos * 1e13, (mass.astype(np.float64) * 2e30).astype(np.float32), eps * 1e13
    elif scale == "small":
        pos, mass, eps = pos * 1e-13, (mass.astype(np.float64) * 1e-25).astype(np.float32), eps * 1e-13
    elif scale == "tiny_eps":
        eps = 1e-9
    sub = ic.subsample(n, n_tgt, 5)
    acc, pot = S.direct_sum(pos, mass, eps, sub)
    k = np.unique(np.linspace(0, n_tgt - 1, 6).round().astype(int))
    ra, rp, mag = reference(pos, mass, eps, sub[k])
    tol = 2.0 ** -46 + 2.0 ** -53 * np.sqrt(n)
    assert np.all(np.abs(acc[k] - ra).max(1) <= tol * mag[:, 0])
    assert np.all(np.abs(pot[k] - rp) <= tol * mag[:, 1])


def test_direct_sum_reports_bad_targets_and_infinite_positions():
    import torch
    n = 65536
    pos, mass = ic.plummer(n, 72)
    src = S._particle_sources(pos, mass, "cuda")
    t = torch.tensor([5, n, 7, -1], dtype=torch.int64, device="cuda")
    scratch = torch.empty(4 * int(L.load().otoo_direct_chunks(n, 4)) * 4, dtype=torch.float64, device="cuda")
    acc = torch.empty((4, 3), dtype=torch.float64, device="cuda")
    pot = torch.empty(4, dtype=torch.float64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    args = (t.data_ptr(), 4, 1e-6, acc.data_ptr(), pot.data_ptr(), scratch.data_ptr(), status.data_ptr(), st)
    L.call("otoo_direct", src.data_ptr(), n, *args)
    assert int(status.item()) == 2
    good = acc[[0, 2]].clone()
    want, _ = S.direct_sum(pos, mass, 1e-3, [5, 7])
    np.testing.assert_array_equal(good.cpu().numpy(), want)
    # an infinite source position: NaN or infinite sums, no error of its own
    pos[9, 1] = np.inf
    a, p = S.direct_sum(pos, mass, 1e-3, [5, 7])
    assert not np.isfinite(a).all()
