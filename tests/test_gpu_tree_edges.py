"""The device tree at the edges of its kernels' tiles and leaf-size paths,
against the host build (needs a GPU): bit-exact order, cells and groups,
moments to rounding (check_tree of test_gpu_tree.py)."""
import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic
from test_gpu_tree import check_tree

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    return L.load()


@pytest.mark.parametrize("n", [2, 31, 33, 2047, 2048, 2049, 4097])
@pytest.mark.parametrize("leaf", [1, 8, 64, 65, 127, 300, 5000])
def test_cells_at_tile_and_leaf_edges(n, leaf):
    pos, mass = ic.hernquist(n, 61)
    check_tree(pos, mass, leaf, 16 if leaf < 16 else 64)


@pytest.mark.parametrize("leaf", [1, 8, 64, 100])
def test_cells_of_coincident_and_lattice_particles(leaf):
    # runs of equal keys longer than a tile, next to a lattice whose cell
    # faces coincide with particle positions
    g = np.stack(np.meshgrid(*[np.arange(8) / 8.0] * 3, indexing="ij"), -1).reshape(-1, 3)
    pos = np.concatenate([g, np.full((2500, 3), 0.1), np.full((70, 3), 0.7)])
    check_tree(pos, np.full(len(pos), 1.0 / len(pos), np.float32), leaf, 32)


@pytest.mark.parametrize("n", [4095, 4096, 4097, 8192, 12289, 70001])
@pytest.mark.parametrize("model", ["uniform", "hernquist", "pairs"])
def test_order_across_sort_tiles(n, model):
    # one tile and several, the last one full, nearly empty and ragged; in
    # "pairs" every position occurs many times, so equal keys span the tiles
    # and the order among them is the callers'
    if model == "pairs":
        p, _ = ic.plummer(37, 62)
        pos = p[np.arange(n) % 37]
    else:
        pos, _ = ic.make(model, n, 62)
    check_tree(pos, np.full(n, 1.0 / n, np.float32), 8, 64)


@pytest.mark.parametrize("mac", ["sw", "sph"])
def test_repeated_builds_are_bit_equal(mac):
    # cells of 1, of a few, of more than 64 and of more than 2048 particles
    # (the forms of the radius pass), built many times: the same records
    import torch

    from paper_1206_1199_gb300 import system as S
    pos, mass = ic.hernquist(30000, 53)
    p, m = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    h = torch.from_numpy(ic.sph_radii(pos, mass, 64, "hernquist")).cuda() if mac == "sph" else None
    ref = None
    for _ in range(200):
        dt = S.DeviceTree.build(p, m, 8, 64, True, "cuda", mac, 1e-5 if mac == "sw" else 0.0, 0.0, h_sph=h)
        got = [dt.bufs[k].clone() for k in ("cell", "cell64", "first", "count")]
        if ref is None:
            ref = got
        assert all(torch.equal(a, b) for a, b in zip(ref, got))


@pytest.mark.parametrize("n", [32767, 32769, 262143, 262145])
@pytest.mark.parametrize("leaf,mac", [(8, "theta"), (70, "theta"), (16, "sw")])
def test_leaves_across_block_sizes(n, leaf, mac):
    # the block sizes of the leaf kernel; leaves of 1, of a few and of more than 64 particles
    pos, mass = ic.plummer(n, 64)
    kw = dict(mac="sw", delta=1e-3) if mac == "sw" else {}
    check_tree(pos, mass, leaf, 64 if leaf < 64 else 128, **kw)


@pytest.mark.parametrize("kind", ["lattice", "shell", "pairs"])
@pytest.mark.parametrize("shift", [0.0, 3e4, -1e7])
@pytest.mark.parametrize("leaf", [8, 40, 300])
def test_radii_with_many_candidates(kind, shift, leaf):
    # many particles at a cell's largest distance, or within the FP32 bounds of
    # it (large coordinates): the FP64 radius about the record's own centre of
    # mass (the host's differs from it by the rounding of large coordinates).
    # With a huge delta the record's r_b is that radius: b / 2 + sqrt(b^2 / 4).
    if kind == "lattice":
        g = np.arange(16) / 16.0
        pos = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    elif kind == "shell":
        v = np.random.default_rng(7).standard_normal((5000, 3))
        pos = v / np.linalg.norm(v, axis=1)[:, None]
    else:
        pos = np.repeat(ic.plummer(1500, 65)[0], 3, axis=0)
    pos = pos + shift
    from paper_1206_1199_gb300 import system as S
    d = S.DeviceTree.build(pos, np.full(len(pos), 1.0 / len(pos), np.float32), leaf, 64, True, "cuda", "sw", 1e290).bufs
    w = d["cell"].cpu().numpy().view(np.dtype(L.WCell))
    w64 = d["cell64"].cpu().numpy().view(np.dtype(L.WCell64))
    p = pos[d["perm"].cpu().numpy()]
    b = np.array([np.sqrt(((w64["com"][k] - p[w["begin"][k]:w["end"][k]]) ** 2).sum(1).max()) for k in range(len(w))])
    # (the squared distance's, the square root's and r_b's roundings)
    assert np.all(np.abs(w64["rb"] - b) <= 8 * 2.0 ** -53 * b + 1e-140)
