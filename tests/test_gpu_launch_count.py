"""GPU: md_last_launch_count of the resident engine counts the kernels of the
list rebuild that ends the call: four for the cell list, then three for the
visiting order, or one for the neighbour list where that is on."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("skin,rebuild", [(0.0, 7), (0.3, 5)])
@pytest.mark.parametrize("profile", [False, True])
def test_resident_launches(skin, rebuild, profile):
    s = I.sphere_system(n=300, R=8.0, seed=2, precision="mixed", tol=1e-10)
    s["params"] = dict(s["params"], cell_size=float(np.max(s["params"]["rcut"])) + 0.3)
    with md.Simulation([s]) as sim:
        if skin:
            md.md_set_neighbor_list(sim.h, skin, 64)
        md.md_set_option(sim.h, md.MD_OPT_ENGINE, 1)
        md.md_set_option(sim.h, md.MD_OPT_RESIDENT_STEPS, 10)
        sim.set_state()
        if profile:
            md.md_profile_step(sim.h, 20)
        else:
            sim.step(20)
        sim.sync()
        assert md.md_last_launch_count(sim.h) == 2 * 2 + rebuild  # two chunks: the engine and the step counter
