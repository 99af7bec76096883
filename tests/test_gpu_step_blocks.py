"""GPU: a long md_step call replays blocks of several steps, short calls single
steps: the same bits however the steps are cut, with the list and without,
with options changed in between, and the launch count counts every kernel."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs, md

pytestmark = pytest.mark.gpu


def _run(kind, precision, cuts, skin=0.0, option=None):
    tol = 1e-12 if precision == "fp64" else 1e-10
    systems = ([inputs.sphere_system(n=700, R=12.0, seed=2, dmin=0.9, precision=precision, dt=0.002, tol=tol)]
               if kind == "sphere" else inputs.capsid_systems(nsys=2, ncone=20, precision=precision, tol=tol)
               if kind == "capsid" else inputs.free_on_surface({"kind": "torus", "center": (0.0, 0.0, 0.0),
                                                               "p": (6.0, 2.0, 0, 0)}, 300, precision=precision))
    for s in systems:
        if skin:
            s["params"] = dict(s["params"], cell_size=float(np.max(s["params"]["rcut"])) + skin)
    with md.Simulation(systems) as sim:
        if skin:
            md.md_set_neighbor_list(sim.h, skin, 256)
        sim.set_state()
        per = None
        for k, n in enumerate(cuts):
            if option and k == len(cuts) // 2:
                md.md_set_option(sim.h, *option)
            sim.step(n)
            if n >= 32 and skin:
                per = md.md_last_launch_count(sim.h) / n
        sim.sync()
        st = sim.state()
    return [st["x"], st["v"], st["p_half"], st["step"]], per


@pytest.mark.parametrize("kind,precision,skin", [("sphere", "mixed", 0.3), ("sphere", "fp64", 0.3), ("sphere", "mixed", 0.0),
                                                 ("capsid", "mixed", 0.4), ("free", "mixed", 0.0)])
def test_cuts_change_no_bit(kind, precision, skin):
    a, per = _run(kind, precision, [130, 7, 33])
    b, _ = _run(kind, precision, [1] * 20 + [40, 9, 64, 1, 36])
    assert all(np.array_equal(p, q) for p, q in zip(a, b))
    if skin:
        c, per = _run(kind, precision, [130, 7, 33], skin)
        d, _ = _run(kind, precision, [1] * 20 + [40, 9, 64, 1, 36], skin)
        assert all(np.array_equal(p, q) for p, q in zip(c, d))
        assert per == (4 if kind == "capsid" else 3)


def test_an_option_between_blocks_takes_effect():
    a, _ = _run("sphere", "mixed", [100, 100], 0.3, (md.MD_OPT_FUSED_REBUILD, 0))
    b, _ = _run("sphere", "mixed", [100, 100], 0.3)
    assert all(np.array_equal(p, q) for p, q in zip(a, b))
