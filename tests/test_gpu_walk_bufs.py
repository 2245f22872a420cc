"""A device walk's counter words and totals as its buffers show them (needs a GPU)."""
import ctypes

import pytest
import torch

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pooled", [False, True])
def test_views_of_the_walk_head(pooled):
    L.load()
    pos, mass = ic.plummer(3000, 95)
    tree = S.DeviceTree.build(pos, mass, 8, 64, True, "cuda")
    pool = S.BufferPool("cuda") if pooled else None
    side = torch.cuda.Stream()
    for stream in (None, None, side):
        dl = tree.walk(0.7, 1e-2, pool=pool, stream=stream)
        c, t = dl.bufs["counter"], dl.bufs["totals"]
        assert c.dtype == torch.int32 and c.numel() == 4 and c.data_ptr() == dl.struct.counter
        assert t.dtype == torch.int64 and t.data_ptr() == dl.struct.totals
        assert int(t[0]) == dl.n_list and int(t[1]) == dl.interactions and int(c[1]) == 0
        plan = dl.plan(L.default_tune(64), stream)
        assert plan.n_items >= dl.n_groups
        L.call("otoo_walk_check_status", ctypes.byref(dl.struct), S._stream(stream, "cuda"))
    with pytest.raises(KeyError):
        dl.bufs["no such buffer"]
