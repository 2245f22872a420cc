"""The set walk's tests against the host walk (needs a GPU): angles per group
on both sides of the cube rule's limit, angle 0, positions far from the origin,
systems of one to a few groups, leaves with many particles.  Every group must
get the host's entries."""
import numpy as np
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import ic, system as S

pytestmark = pytest.mark.gpu

ANGLES = {"mixed": [0.0, 1e-6, 0.3, 0.5699, 0.57, 0.5774, 0.58, 1.0, 3.0, 1e20], "zero": [0.0], "wide": [0.7, 0.9],
          "one": None}


@pytest.mark.parametrize("n,leaf,shift,scale", [(1, 8, 0.0, 1.0), (70, 8, 0.0, 1.0), (3000, 1, 0.0, 1.0),
                                                (6000, 8, 1e6, 1.0), (6000, 16, -3.0, 1e-9), (6000, 8, 0.0, 1e12)])
@pytest.mark.parametrize("angles", sorted(ANGLES))
def test_sets_against_the_host_walk(n, leaf, shift, scale, angles):
    L.load()
    pos, mass = ic.plummer(n, 61)
    pos = (pos + shift) * scale
    if n == 3000:  # leaves beyond a warp: coincident particles
        pos[100:170] = pos[100]
        pos[500:533] = pos[500]
    t = S.Tree(pos, mass, leaf)
    dt = S.DeviceTree(t, 32, True)
    tpg = ANGLES[angles]
    if tpg is not None:
        tpg = np.random.default_rng(n).choice(np.float32(tpg), dt.n_groups).astype(np.float32)
    theta = 0.5
    hl = t.lists(theta, 32, 0.01 * scale, True, theta_per_group=tpg)
    gh, lh = hl.groups, hl.list
    for gs in (0, 1, 2, 8):
        dl = dt.walk(theta, 0.01 * scale, theta_per_group=tpg, group_set=gs)
        gd, ld = dl.groups, dl.list
        for k in ("first", "count", "n_cell", "n_part", "list_off", "cx", "cy", "cz", "theta"):
            np.testing.assert_array_equal(gd[k], gh[k], err_msg=k)
        assert (dl.n_list, dl.interactions, dl.cell_interactions) == (hl.n_list, hl.interactions, hl.cell_interactions)
        for g in range(len(gh)):
            o, nc = gh["list_off"][g], gh["n_cell"][g]
            e = o + nc + gh["n_part"][g]
            np.testing.assert_array_equal(np.sort(ld[o:o + nc]), np.sort(lh[o:o + nc]))
            np.testing.assert_array_equal(np.sort(ld[o + nc:e]), np.sort(lh[o + nc:e]))
        de = dt.walk(theta, 0.01 * scale, theta_per_group=tpg, group_set=gs, exact=True)
        np.testing.assert_array_equal(de.list, ld)
