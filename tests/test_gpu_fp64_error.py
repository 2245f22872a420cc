"""Error of the FP64 form where cells are near and their quadrupoles matter (needs
a GPU), against the same lists in extended precision."""
import numpy as np
import pytest
import torch

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S
from test_gpu_fp64_form import reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,n,n_crit,theta,eps,iblock",
                         [("king", 5000, 64, 0.9, 4e-3, 2), ("polytrope_pair", 8000, 64, 1.0, 1e-2, 2),
                          ("plummer", 8000, 32, 1.0, 1e-4, 1), ("hernquist", 20000, 32, 0.9, 1e-2, 4),
                          ("plummer", 60000, 64, 0.9, 1e-3, 2), ("plummer", 20000, 128, 0.5, 0.3, 2)])
def test_error_of_the_fp64_form_is_that_of_rounding(model, n, n_crit, theta, eps, iblock):
    # the result's rounding (0.29 x 2^-52 = 0.64e-16 rms), a thread's running sum of one to
    # two hundred pairs (each addition 0.29 x 2^-52 of the sum so far, in a share of a
    # quarter to a half of the total: 0.6e-16 to 1.2e-16 together), a pair's own roundings
    # (2.2 x 2^-53 over many pairs): below 1.4e-16, without room for a part of 2^-47
    L.load()
    pos, mass = ic.make(model, n, 93)
    lists = S.Tree(pos, mass, 8).lists(theta, n_crit, eps, True)
    tune = L.default_tune(n_crit)
    tune.iblock = iblock
    dev = S.DeviceSystem.upload(lists, lists.plan(tune), "cuda", use_perm=False)
    a, p = (t.cpu().numpy() for t in S.force(dev, precision=L.OTOO_FP64))
    idx, ra, rp, _ = reference(lists, n, np.linspace(0, lists.n_groups - 1, 40).astype(int), 5)

    def err(x, r):
        d = x.astype(np.longdouble) - r
        return float(np.sqrt((d * d).sum() / (r * r).sum()))
    assert err(a[idx], ra) <= 1.4e-16
    assert err(p[idx], rp) <= 1.4e-16


@pytest.mark.parametrize("copies,threads", [(1, 256), (300, 128)])  # up to 14 items per SM, and more
@pytest.mark.parametrize("n_crit,iblock", [(100, 1), (250, 2), (400, 4)])
def test_items_of_more_targets_than_threads(n_crit, iblock, copies, threads):
    # an item's targets are taken in passes of the CTA's threads: the same bits as from
    # items of one pass each (every item several times over writes the same values)
    L.load()
    n = 3000
    pos, mass = ic.plummer(n, 94)
    lists = S.Tree(pos, mass, 8).lists(0.7, n_crit, 1e-2, True)
    tune = L.default_tune(64)
    tune.iblock = iblock
    plan = lists.plan(tune)
    g = lists.groups
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def run(first, size, group):
        items = np.zeros(len(group), plan.items.dtype)
        items["g"], items["i0"], items["ni"], items["slot"] = group, first, size, -1
        items["j1"] = (g["n_cell"] + g["n_part"])[group]
        items = np.tile(items, copies)
        assert items["ni"].max() <= 128 * iblock and (len(items) > 14 * sms) == (threads == 128)
        dev = S.DeviceSystem.upload(lists, plan, "cuda")
        dev.bufs["items"] = torch.from_numpy(items.view(np.uint8).reshape(-1).copy()).cuda()
        dev.struct.items, dev.struct.n_items, dev.struct.n_splits = dev.bufs["items"].data_ptr(), len(items), 0
        return [t.cpu().numpy() for t in S.force(dev, precision=L.OTOO_FP64)]
    whole = run(np.zeros(len(g), int), g["count"], np.arange(len(g)))
    parts = [(k, i, min(threads, int(c) - i)) for k, c in enumerate(g["count"]) for i in range(0, int(c), threads)]
    k, i, c = (np.array(x) for x in zip(*parts))
    assert iblock == 1 or threads == 256 and iblock == 2 or len(parts) > len(g)
    for x, y in zip(whole, run(i, c, k)):
        np.testing.assert_array_equal(x, y)
