"""Positions and masses the device tree refuses (needs a GPU): the error, and that
it comes back in the time of a build."""
import time

import numpy as np
import pytest
import torch

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mac,extra", [("theta", {}), ("sw", dict(delta=1e-4))])
@pytest.mark.parametrize("what", ["inf", "nan", "mass0", "mass_nan"])
def test_refusal_is_no_slower_than_a_build(mac, extra, what):
    # an infinite coordinate gives every particle the same key: one leaf of all of
    # them, if the cells were made
    n = 1 << 20
    pos, mass = ic.plummer(n, 81)

    def build(p, m):
        p, m = torch.from_numpy(p).cuda(), torch.from_numpy(m).cuda()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        try:
            S.DeviceTree.build(p, m, 8, 64, True, "cuda", mac=mac, **extra)
            code = 0
        except L.OtooError as e:
            code = e.code
        return time.perf_counter() - t0, code
    good = min(build(pos, mass)[0] for _ in range(3))
    p, m = pos.copy(), mass.copy()
    if what in ("inf", "nan"):
        p[n // 2, 1] = np.inf if what == "inf" else np.nan
    else:
        m[n // 2] = 0.0 if what == "mass0" else np.nan
    t, codes = zip(*(build(p, m) for _ in range(3)))
    assert all(c == L.OTOO_EINVAL for c in codes)
    assert min(t) <= 1.5 * good
    assert build(pos, mass)[1] == 0
