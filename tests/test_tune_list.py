"""The list autotuner's trials, on a stand-in for the library: every skin is
timed at every width of the list walk, in both precisions (the float64 walk
takes a width too), the width a small system's unset walk takes among them."""
import pytest

from paper_1411_3019_gb300 import inputs, md, tune


class _Sim:
    def __init__(self, systems, stream=None):
        self.h = {"skin": systems[0]["params"]["cell_size"] - inputs.WCA_RC, "width": None}

    def set_state(self):
        pass

    def step(self, n):
        pass

    def sync(self):
        pass

    def close(self):
        pass


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_every_width_is_timed(monkeypatch, precision):
    monkeypatch.setattr(md, "Simulation", _Sim)
    monkeypatch.setattr(md, "md_set_neighbor_list", lambda h, skin, cap: None)
    monkeypatch.setattr(md, "md_set_option", lambda h, key, val: h.update(width=val))
    monkeypatch.setattr(md, "md_get_option", lambda h, key: 0)
    monkeypatch.setattr(md, "md_profile_step", lambda h, n: {"pair": {32: 3.0, 16: 2.0, 8: 1.0}[h["width"]], "integrate": h["skin"]})
    systems = [inputs.sphere_system(n=60, R=6.0, precision=precision)]
    out = tune.autotune_list(systems, 64, skins=(0.3, 0.4))
    assert {(t["skin"], t["list_warp"]) for t in out["trials"]} == {(s, w) for s in (0.3, 0.4) for w in (32, 16, 8)}
    assert (out["skin"], out["list_warp"]) == (0.3, 8)
    out = tune.autotune_list(systems, 64, skins=(0.3,), list_warps=(32, 16))
    assert {t["list_warp"] for t in out["trials"]} == {32, 16}
