"""The FP64 form's quadrupole cells (monopole part in FP64, quadrupole part in
two-float arithmetic) against an evaluation of the same lists in extended
precision (needs a GPU), over units, softenings and targets per thread."""
import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


def reference(lists, n, groups, per_group=4):
    """Accelerations, potentials and sums of the terms' magnitudes of a few
    targets of the given groups, from the lists, in long double."""
    ld = np.longdouble
    src, quad, lst, g = lists.src, lists.quad, lists.list, lists.groups
    idx, acc, pot, mag = [], [], [], []
    for k in groups:
        gr = g[k]
        e = lst[gr["list_off"]:gr["list_off"] + gr["n_cell"] + gr["n_part"]]
        nc = int(gr["n_cell"])
        x = np.stack([src["x"][e], src["y"][e], src["z"][e]], 1).astype(ld)
        m = src["m"][e].astype(ld)
        q = {f: quad[e[:nc] - n][f].astype(ld) for f in ("xx", "yy", "zz", "xy", "xz", "yz", "b2")}
        e2 = ld(gr["eps2"])
        for i in range(int(gr["first"]), int(gr["first"]) + min(int(gr["count"]), per_group)):
            r = x - np.array([src["x"][i], src["y"][i], src["z"][i]], ld)
            iq = 1 / np.sqrt((r * r).sum(1) + e2)
            w = m.copy()
            w[e == i] = 0
            a = (w * iq ** 3)[:, None] * r
            p = -(w * iq)
            rc, qc = r[:nc], iq[:nc]
            n0 = q["xx"] * rc[:, 0] + q["xy"] * rc[:, 1] + q["xz"] * rc[:, 2]
            n1 = q["xy"] * rc[:, 0] + q["yy"] * rc[:, 1] + q["yz"] * rc[:, 2]
            n2 = q["xz"] * rc[:, 0] + q["yz"] * rc[:, 1] + q["zz"] * rc[:, 2]
            nv = np.stack([n0, n1, n2], 1)
            u = (rc * nv).sum(1) - q["b2"] * e2
            aq = (2.5 * u * qc ** 7)[:, None] * rc - (qc ** 5)[:, None] * nv
            pq = -0.5 * u * qc ** 5
            idx.append(i)
            acc.append(a.sum(0) + aq.sum(0))
            pot.append(p.sum() + pq.sum())
            mag.append((np.sqrt((a * a).sum(1)).sum() + np.sqrt((aq * aq).sum(1)).sum(), -p.sum() + np.abs(pq).sum()))
    return np.array(idx), np.array(acc, ld), np.array(pot, ld), np.array(mag, ld)


@pytest.mark.parametrize("iblock", [1, 2, 4])
@pytest.mark.parametrize("scale,mscale,eps", [(1.0, 1.0, 1e-3), (1e12, 1e15, 1e-3), (1e-9, 1e-12, 1e-3), (1.0, 1.0, 1.0),
                                              (1.0, 1.0, 1e-9), (1.0, "spread", 1e-3)])
@pytest.mark.parametrize("theta", [0.5, 1.0])
def test_quadrupole_cells_of_the_fp64_form(iblock, scale, mscale, eps, theta):
    # a monopole pair in FP64 is within 8 roundings of 2^-53, a quadrupole term
    # within 2^-46 of itself and no cell's exceeds an eighth of its monopole
    # here; the sums (FP64 over up to 2000 terms a thread) are within
    # 2^-53 sqrt(2000): together below 2^-47 of the terms' magnitudes
    L.load()
    n = 5000
    pos, mass = ic.hernquist(n, 91)
    if mscale == "spread":  # light cells before heavy ones in a list: other units on the way
        mscale = np.where(pos[:, 0] < 0, 1e-20, 1.0)
    pos, mass = pos * scale, (mass.astype(np.float64) * mscale).astype(np.float32)
    lists = S.Tree(pos, mass, 8).lists(theta, 64, eps * scale, True)
    tune = L.default_tune(64)
    tune.iblock = iblock
    dev = S.DeviceSystem.upload(lists, lists.plan(tune), "cuda", use_perm=False)
    a, p = (t.cpu().numpy() for t in S.force(dev, precision=L.OTOO_FP64))
    with np.errstate(invalid="ignore"):
        idx, ra, rp, mag = reference(lists, n, np.linspace(0, lists.n_groups - 1, 12).astype(int))
    tol = 2.0 ** -47
    # (in the largest units the moments of big cells are past the FP32 range of
    # the stored records: both sides are then not finite)
    fin = np.isfinite(rp)
    assert np.array_equal(fin, np.isfinite(ra).all(1))
    assert np.array_equal(fin, np.isfinite(p[idx])) and np.array_equal(fin, np.isfinite(a[idx]).all(1))
    assert np.all(np.abs(a[idx] - ra).max(1)[fin] <= tol * mag[fin, 0])
    assert np.all(np.abs(p[idx] - rp)[fin] <= tol * mag[fin, 1])
