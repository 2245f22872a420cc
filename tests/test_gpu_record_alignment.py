"""Cell records into arrays that start on a 16-byte boundary and into one that
does not (needs a GPU): the same bytes."""
import ctypes

import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 50, 9000])
def test_records_at_an_odd_start(n):
    import torch
    L.load()
    pos, mass = ic.king(n, 66)
    ref = S.DeviceTree.build(pos, mass, 8, 64, True, "cuda")
    cap, dev, u8, i32 = max(1024, n), "cuda", torch.uint8, torch.int32
    p, m = torch.from_numpy(pos).to(dev), torch.from_numpy(mass).to(dev)
    b = dict(src=torch.empty((n + cap) * 32, dtype=u8, device=dev), quad=torch.empty(cap * 32, dtype=u8, device=dev),
             cell=torch.empty(cap * 64, dtype=u8, device=dev), cell64=torch.empty(cap * 96 + 8, dtype=u8, device=dev)[8:],
             first=torch.empty(n, dtype=i32, device=dev), count=torch.empty(n, dtype=i32, device=dev),
             perm=torch.empty(n, dtype=torch.int64, device=dev), level=torch.empty(cap, dtype=i32, device=dev),
             status=torch.empty(2, dtype=i32, device=dev))
    t = L.DevTree()
    t.n_part, t.cap_cell, t.leaf_size, t.n_crit, t.use_quad, t.mac = n, cap, 8, 64, 1, S.MAC_KINDS["theta"]
    t.h_sph = None
    t.src, t.quad, t.cell, t.cell64 = (b[k].data_ptr() for k in ("src", "quad", "cell", "cell64"))
    t.group_first, t.group_count, t.perm = b["first"].data_ptr(), b["count"].data_ptr(), b["perm"].data_ptr()
    t.cell_level, t.status = b["level"].data_ptr(), b["status"].data_ptr()
    nbytes = int(L.load().otoo_devtree_scratch_bytes(n, cap))
    scratch = torch.empty(nbytes, dtype=u8, device=dev)
    L.call("otoo_devtree_build", p.data_ptr(), m.data_ptr(), ctypes.byref(t), scratch.data_ptr(), nbytes,
           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    nc = int(t.n_cell)
    assert nc == ref.n_cell
    for k, size in (("src", (n + nc) * 32), ("quad", nc * 32), ("cell", nc * 64), ("cell64", nc * 96)):
        assert torch.equal(b[k][:size], ref.bufs[k][:size]), k
