"""GPU: a handle without a thermostat draws no normals and holds no memory for
them; it runs as before with and without the list, and its option still reads
and switches."""
import numpy as np
import pytest
import torch

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu

SPHERE = {"kind": "sphere", "center": (0.0, 0.0, 0.0), "p": (900.0, 0.0, 0.0, 0.0)}


@pytest.mark.parametrize("precision,per_particle", [("mixed", 16), ("fp64", 24)])
def test_normals_are_held_with_a_thermostat_only(precision, per_particle):
    n = 1 << 21
    used = []
    torch.cuda.init()
    for kT in (1.0, 0.0, 1.0, 0.0):
        before = torch.cuda.mem_get_info()[0]
        h = md.md_create(SPHERE, I.wca_params(precision=precision, kT=kT), n)
        used.append(before - torch.cuda.mem_get_info()[0])
        md.md_destroy(h)
    # (the driver hands memory out in blocks of 2 MB)
    assert abs((used[2] - used[3]) - per_particle * n) <= 4 << 20


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("skin", [0.0, 0.3])
def test_runs_without_a_thermostat(skin, precision):
    s = I.nve_systems(1, n=300, precision=precision, tol=1e-10)
    for q in s:
        q["params"] = dict(q["params"], cell_size=float(np.max(q["params"]["rcut"])) + 0.3)
    out = []
    for store in (1, 0):
        with md.Simulation(s) as sim:
            if skin:
                md.md_set_neighbor_list(sim.h, skin, 128)
            md.md_set_option(sim.h, md.MD_OPT_STORE_NOISE, store)
            assert md.md_get_option(sim.h, md.MD_OPT_STORE_NOISE) == store
            sim.set_state()
            sim.step(30)
            sim.sync()
            out.append(sim.state())
    assert all(np.array_equal(out[0][k], out[1][k]) for k in ("x", "v", "p_half"))
