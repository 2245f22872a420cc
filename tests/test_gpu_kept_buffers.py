"""Steps that reuse a pool's buffers (needs a GPU): systems that grow and shrink,
plans that outgrow the kept items and splits, another stream than the current
one -- the same items, splits and forces as with fresh buffers."""
import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_stream", [False, True])
def test_plans_in_kept_buffers(own_stream):
    L.load()
    import torch
    pool = S.BufferPool("cuda")
    stream = torch.cuda.Stream() if own_stream else None
    grown = 0
    for n, split in ((500, 8192), (20000, 8192), (20000, 64), (20000, 64), (300, 64), (300, 32), (6000, 500), (30000, 32)):
        pos, mass = ic.plummer(n, 83)
        dt = S.DeviceTree.build(pos, mass, 8, 64, True, "cuda")
        torch.cuda.synchronize()
        tune = L.default_tune(64)
        tune.split = split
        got = {}
        for name, p, st in (("fresh", None, None), ("kept", pool, stream)):
            before = p.bufs["splits"].numel() if p and "splits" in p.bufs else 0
            dl = dt.walk(0.6, 1e-2, pool=p, stream=st)
            plan = dl.plan(tune, stream=st)
            step = S.DeviceStep(dl, plan)
            a, q = S.force(step, stream=st)
            torch.cuda.synchronize()
            got[name] = (plan.n_items, plan.n_splits, plan.partial_doubles,
                         sorted(tuple(r)[:6] for r in plan.items[["g", "i0", "ni", "j0", "j1", "slot"]].tolist()),
                         plan.splits.tolist(), a.cpu().numpy(), q.cpu().numpy())
            grown += p is not None and p.bufs["splits"].numel() > before
        f, k = got["fresh"], got["kept"]
        assert f[:5] == k[:5]
        # (a one-pass walk lists a group's cells in another order)
        np.testing.assert_allclose(k[5], f[5], rtol=0, atol=2e-5 * np.abs(f[5]).max())
        np.testing.assert_allclose(k[6], f[6], rtol=2e-5)
    assert grown >= 3
