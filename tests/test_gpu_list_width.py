"""GPU: MD_OPT_LIST_WARP holds as set, on systems small enough that the unset
walk takes fewer particles per warp, and every width, on both sides of the
sizes at which the unset walk changes it, gives the per-lane walk's bits."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


def _forces(n, precision, options, max_neighbors):
    s = I.sphere_system(n=n, R=0.66 * n ** 0.5, seed=3, dmin=0.8, precision=precision, tol=1e-10)
    s["params"] = dict(s["params"], cell_size=float(np.max(s["params"]["rcut"])) + 0.4)
    with md.Simulation([s]) as sim:
        for key, val in options:
            md.md_set_option(sim.h, key, val)
        md.md_set_neighbor_list(sim.h, 0.4, max_neighbors)
        assert md.md_get_option(sim.h, md.MD_OPT_LIST_WARP) == dict(options).get(md.MD_OPT_LIST_WARP, 32)
        sim.set_state()
        return sim.forces()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,max_neighbors", [(5, 64), (1033, 64), (16385, 64), (32769, 64), (32769, 128)])
def test_every_width_gives_the_same_bits(n, max_neighbors, precision):
    want = _forces(n, precision, [(md.MD_OPT_PAIR_QUEUE, 0)], max_neighbors)
    for width in (None, 8, 16, 32):
        got = _forces(n, precision, [] if width is None else [(md.MD_OPT_LIST_WARP, width)], max_neighbors)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), width
