"""FP64 to FP32 on the integer pipe (needs a GPU): the sources' float pairs and
the cell records bit for bit those of the conversions, over ties, signs, zeros
and magnitudes in and out of FP32's normal range."""
import warnings

import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


def values(n):
    rng = np.random.default_rng(17)
    f = rng.standard_normal(n).astype(np.float32)
    ulp = np.spacing(np.abs(f)).astype(np.float64)
    x = f.astype(np.float64)
    kinds = [x, x + 0.5 * ulp, x - 0.5 * ulp, np.nextafter(x + 0.5 * ulp, np.inf), np.nextafter(x + 0.5 * ulp, -np.inf),
             rng.standard_normal(n), np.ldexp(rng.standard_normal(n), rng.integers(-190, 20, n)),
             np.ldexp(rng.standard_normal(n), rng.integers(-80, -60, n)),
             np.full(n, 0.0), np.full(n, -0.0), np.float64(np.nextafter(np.float32(2), np.float32(0))) + 2.0 ** -25 + 0.0 * x]
    return np.concatenate(kinds)


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 100, 2.0 ** 126, 2.0 ** 127.5, 2.0 ** -60])
def test_float_pairs_of_the_sources(scale):
    L.load()
    v = values(400) * scale
    v = np.random.default_rng(3).permutation(v)
    pos = v[:len(v) // 3 * 3].reshape(-1, 3)
    lists = S.Tree(pos, np.full(len(pos), 1.0 / len(pos), np.float32), 8).lists(0.5, 64, 1e-3 * scale, False)
    dev = S.DeviceSystem.upload(lists, lists.plan(L.default_tune(64)), "cuda")
    S.force(dev)
    got = dev.bufs["split"].cpu().numpy().view(np.float32).reshape(-1, 8)[:len(lists.src)]
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")
        for k, c in enumerate("xyz"):
            x = lists.src[c].astype(np.float64)
            h = x.astype(np.float32)
            lo = (x - h.astype(np.float64)).astype(np.float32)
            np.testing.assert_array_equal(got[:, k].view(np.uint32), h.view(np.uint32))
            np.testing.assert_array_equal(got[:, 4 + k].view(np.uint32), lo.view(np.uint32))
    np.testing.assert_array_equal(got[:, 3], lists.src["m"])


@pytest.mark.parametrize("scale", [1e-43, 1e-37, 1e-19, 1e15, 1e30])
def test_records_out_of_the_normal_range(scale):
    # (the quadrupoles leave FP32's range here: the walk records against their own
    # FP64 fields, the links against the host build's)
    L.load()
    pos, mass = ic.plummer(3000, 63)
    pos = pos * scale
    dev = S.DeviceTree.build(pos, mass, 8, 64, True, "cuda").bufs
    host = S.DeviceTree(S.Tree(pos, mass, 8), 64, True, "cpu").bufs
    d, h = (b["cell"].cpu().numpy().view(np.dtype(L.WCell)) for b in (dev, host))
    links = [sorted(zip(c["begin"], c["end"], c["nchild"])) for c in (d, h)]
    assert links[0] == links[1]
    w = dev["cell64"].cpu().numpy().view(np.dtype(L.WCell64))
    com, lo, gc = (w[k].astype(np.float64) for k in ("com", "lo", "gc"))
    hi = com.astype(np.float32)
    e = com - gc
    s = np.sqrt((e[:, 0] * e[:, 0] + e[:, 1] * e[:, 1]) + e[:, 2] * e[:, 2])
    for got, want in ((d["com_hi"], hi), (d["com_lo"], (com - hi.astype(np.float64)).astype(np.float32)),
                      (d["e"], (com - lo).astype(np.float32)), (d["side"], w["side"].astype(np.float32)),
                      (d["s"], s.astype(np.float32))):
        np.testing.assert_array_equal(np.ascontiguousarray(got).view(np.uint32), want.view(np.uint32))
