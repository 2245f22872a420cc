"""The autotuner's search on the host (no GPU): the step and its time are
stand-ins."""
import pytest

from paper_1206_1199_gb300 import _lib as L
from paper_1206_1199_gb300 import autotune, ic, system as S


@pytest.mark.parametrize("fastest", [(128, 4, 256, 8192), (128, 1, 256, 4096), (64, 4, 128, 2048), (128, 2, 64, 4096),
                                     (128, 2, 256, 16384), (256, 1, 128, 4096)])
def test_search_reaches_every_kernel_and_times_it_once(monkeypatch, fastest):
    # the value of packed names a kernel and changes nothing, so both of its values
    # measure alike but for noise: a time that depends on the knobs, each knob's own
    # share smallest at the fastest, with noise on the second time of a kernel
    L.load()
    pos, mass = ic.plummer(500, 7)
    seen = []

    def time_step(dev, lists, tune, **kw):
        key = (tune.block, tune.iblock, tune.tile, tune.split)
        ms = 1.0 + sum(0.1 * (a != b) for a, b in zip(key, fastest)) - 0.01 * seen.count(key)
        seen.append(key)
        return ms
    monkeypatch.setattr(S.DeviceSystem, "upload", classmethod(lambda cls, lists, plan, device: object()))
    monkeypatch.setattr(autotune, "_time_step", time_step)
    w = dict(leaf_size=8, theta=0.7, eps=1e-2, use_quad=True)
    best, table = autotune.search(pos, mass, w, n_crits=(32, 64), device="cpu", log=lambda s: None)
    t = best["tune"]
    assert (t["block"], t["iblock"], t["tile"], t["split"]) == fastest
    assert (t["block"], t["iblock"], t["tile"], t["packed"]) in autotune.VARIANTS
    rows = [(r["n_crit"], r["block"], r["iblock"], r["tile"], r["split"]) for r in table]
    assert len(rows) == len(set(rows))
