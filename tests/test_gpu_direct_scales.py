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


def in_fp64(pos, mass, eps, targets, chunk):
    """The sums in FP64: pairs one after another within a chunk of the sources,
    then the chunks."""
    mass, e2 = mass.astype(np.float64), float(eps) ** 2
    acc, pot = [], []
    for i in targets:
        d = pos - pos[i]
        q = 1.0 / np.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2] + e2)
        w = mass * q
        w[i] = 0.0
        g = w * q * q
        t = np.stack([g * d[:, 0], g * d[:, 1], g * d[:, 2], -w], 1)
        s = [np.add.accumulate(t[k:k + chunk])[-1] for k in range(0, len(t), chunk)]
        s = np.add.accumulate(np.array(s))[-1]
        acc.append(s[:3])
        pot.append(s[3])
    return np.array(acc), np.array(pot)


def far_out(r):
    def make(n):
        pos, mass = ic.plummer(n, 75)
        pos[n // 3] = np.array([0.6, -0.64, 0.48]) * r
        return pos, mass
    return make


def groups_of(k, sep):
    # every fifth of the system in tight groups of k neighbours
    def make(n):
        pos, mass = ic.plummer(n, 76)
        rng = np.random.default_rng(76)
        for g in range(n // (5 * k)):
            pos[g * k:(g + 1) * k] = pos[g * k] + sep * rng.standard_normal((k, 3))
        return pos, mass
    return make


@pytest.mark.parametrize("make,eps", [(far_out(1e2), 1e-3), (far_out(1e3), 1e-3), (far_out(1e4), 1e-3), (far_out(1e5), 1e-3),
                                      (far_out(1e6), 1e-2), (far_out(1e7), 5e-2), (groups_of(3, 1e-5), 1e-6),
                                      (groups_of(10, 1e-4), 1e-5), (groups_of(100, 1e-3), 1e-4),
                                      (lambda n: ic.hernquist(n, 77), 1e-4), (lambda n: ic.plummer(n, 78), 0.3)],
                         ids=["far1e2", "far1e3", "far1e4", "far1e5", "far1e6", "far1e7", "groups3", "groups10", "groups100",
                              "hernquist", "soft"])
def test_direct_sum_no_less_exact_than_in_fp64(make, eps):
    # a particle far out of a dense core, close groups whose pairs are most of a
    # target's acceleration, a softening of the core's size: the 2-norm of the error
    # over the targets is no larger than that of FP64 pairs summed in FP64
    n, nt = 66000, 600
    pos, mass = make(n)
    t = np.arange(nt) if "groups" in make.__qualname__ else np.sort(ic.subsample(n, nt, 8))
    acc, pot = S.direct_sum(pos, mass, eps, t)
    chunks = int(L.load().otoo_direct_chunks(n, nt))
    chunk = ((n + chunks - 1) // chunks + 127) // 128 * 128
    k = np.arange(0, nt, 20)
    ra, rp, _ = reference(pos, mass, eps, t[k])
    fa, fp = in_fp64(pos, mass, eps, t[k], chunk)

    def err(a, r):
        d = a.astype(np.longdouble) - r
        return float(np.sqrt((d * d).sum() / (r * r).sum()))
    assert err(acc[k], ra) <= err(fa, ra)
    assert err(pot[k], rp) <= err(fp, rp)


@pytest.mark.parametrize("light", [1e-10, 1e-25, 1e-30])
def test_direct_sum_of_light_sources_on_a_heavy_one(light):
    # the heavy particle's own acceleration is the light ones' alone, on both sides
    # of the mass ratio the two-float form takes
    n, eps = 65536, 1e-3
    pos, mass = ic.plummer(n, 79)
    mass = (mass.astype(np.float64) * n * light).astype(np.float32)
    mass[7] = 1.0
    acc, pot = S.direct_sum(pos, mass, eps, [7, 100])
    ra, rp, mag = reference(pos, mass, eps, [7, 100])
    tol = 2.0 ** -46 + 2.0 ** -53 * np.sqrt(n)
    assert np.all(np.abs(acc - ra).max(1) <= tol * mag[:, 0])
    assert np.all(np.abs(pot - rp) <= tol * mag[:, 1])
