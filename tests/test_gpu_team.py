"""Small launches give a work item to a CTA, larger ones to a warp: the same
bits either way (needs a GPU).  A system on its own takes the one form, packed
with enough copies of itself to pass the rule's line the other."""
import ctypes

import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block,iblock,tile,packed", [(128, 2, 128, 0), (128, 2, 256, 1), (64, 2, 128, 1),
                                                      (128, 1, 128, 0), (64, 1, 128, 1), (128, 1, 256, 1),
                                                      (256, 1, 128, 0), (256, 2, 128, 0), (128, 2, 64, 0),
                                                      (128, 4, 256, 0), (64, 4, 128, 0)])
@pytest.mark.parametrize("quad", [True, False])
@pytest.mark.parametrize("split", [300, 100000])
def test_small_and_large_launches_give_the_same_bits(block, iblock, tile, packed, quad, split):
    L.load()
    import torch
    items_per_sm = 80
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pos, mass = ic.plummer(6000, 81)
    lists = S.Tree(pos, mass, 8).lists(0.6, 64, 1e-2, quad)
    tune = L.Tune(block=block, iblock=iblock, tile=tile, split=split, ctas_per_sm=0, packed=packed)
    plan = lists.plan(tune)
    one = S.DeviceSystem.upload(lists, plan, "cuda")
    a, p = (t.cpu().numpy() for t in S.force(one))
    assert plan.n_items <= items_per_sm * sms
    copies = int(items_per_sm * sms // plan.n_items) + 2
    many = S.Lists.pack([lists] * copies)
    mplan = many.plan(tune)
    assert mplan.n_items > items_per_sm * sms
    am, pm = (t.cpu().numpy() for t in S.force(S.DeviceSystem.upload(many, mplan, "cuda")))
    off = many.sys_part_off
    for k in (0, copies // 2, copies - 1):
        np.testing.assert_array_equal(am[off[k]:off[k + 1]], a)
        np.testing.assert_array_equal(pm[off[k]:off[k + 1]], p)


@pytest.mark.parametrize("block,iblock,tile,packed", [(128, 2, 128, 0), (128, 2, 256, 1), (128, 4, 128, 0), (64, 1, 128, 1)])
def test_short_items_below_the_line(block, iblock, tile, packed):
    # few enough items for the kernel with both forms, too short for a CTA each
    L.load()
    import torch
    line = 80 * torch.cuda.get_device_properties(0).multi_processor_count
    pos, mass = ic.plummer(70000, 82)
    lists = S.Tree(pos, mass, 8).lists(1.0, 32, 1e-2, True)
    plan = lists.plan(L.Tune(block=block, iblock=iblock, tile=tile, split=8192, ctas_per_sm=0, packed=packed))
    a, p = (t.cpu().numpy() for t in S.force(S.DeviceSystem.upload(lists, plan, "cuda")))
    copies = line // plan.n_items + 2
    many = S.Lists.pack([lists] * copies)
    mplan = many.plan(plan.tune)
    assert plan.n_items <= line < mplan.n_items
    am, pm = (t.cpu().numpy() for t in S.force(S.DeviceSystem.upload(many, mplan, "cuda")))
    off = many.sys_part_off
    for k in (0, copies - 1):
        np.testing.assert_array_equal(am[off[k]:off[k + 1]], a)
        np.testing.assert_array_equal(pm[off[k]:off[k + 1]], p)
