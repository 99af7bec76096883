"""GPU: a particle that has moved just beyond skin / 2 since the last build
rebuilds the list, at the edge of float32's resolution, in both precisions (the
Verlet list's promise that every pair within r_c is listed rests on it)."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu

RC, SKIN = 2.5, 0.3


def _free(x, v, precision, half, dt):
    prm = I.wca_params(precision=precision, dt=dt, gamma=0.0, kT=0.0, box_lo=(-half,) * 3, box_hi=(half,) * 3,
                       cell_size=RC + SKIN)
    prm["rcut"][0, 0] = RC
    return [I._system("free", {"kind": "none", "center": (0.0,) * 3, "p": (0.0,) * 4}, prm, x, v)]


def _directions(g, m):
    u = g.normal(size=(m, 3))
    return u / np.linalg.norm(u, axis=1)[:, None]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_a_move_beyond_half_the_skin_rebuilds(precision):
    g = np.random.default_rng(10)
    dt, missed = 0.01, 0
    for _ in range(150):
        x = np.stack([g.uniform(-20, 20, 3), np.full(3, 40.0)])
        v = np.zeros((2, 3))
        v[0] = _directions(g, 1)[0] * ((SKIN / 2 + 2e-8) / dt)
        with md.Simulation(_free(x, v, precision, 48.0, dt)) as sim:
            md.md_set_neighbor_list(sim.h, SKIN, 4)
            sim.set_state()
            before = md.md_get_option(sim.h, md.MD_OPT_NLIST_BUILDS)
            sim.step(1)
            missed += md.md_get_option(sim.h, md.MD_OPT_NLIST_BUILDS) == before
    assert missed == 0
