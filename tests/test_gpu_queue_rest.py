"""GPU: the queues of the warp-per-particle kernel and of the float64 list walk
where nearly every chunk fills them, so that a rest is moved to the front after
each evaluation and written over by the next chunk's hits: a dense liquid gives
the row kernel's and the per-lane walk's bits."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


def _forces(systems, options=(), skin=0.0):
    with md.Simulation(systems) as sim:
        for key, val in options:
            md.md_set_option(sim.h, key, val)
        if skin:
            md.md_set_neighbor_list(sim.h, skin, 512)
        sim.set_state()
        return sim.forces()


@pytest.mark.parametrize("rc", [2.5, 3.4])
def test_float64_list_walk_of_a_dense_liquid(rc):
    def systems():
        s = I.lj_lattice(13, rc=rc, seed=5, precision="fp64")
        s[0]["params"] = dict(s[0]["params"], cell_size=rc + 0.1)
        return s
    want = _forces(systems(), [(md.MD_OPT_PAIR_QUEUE, 0)], 0.1)
    for _ in range(5):
        got = _forces(systems(), [(md.MD_OPT_PAIR_QUEUE, 1)], 0.1)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_warp_kernel_of_a_dense_liquid(precision):
    s = I.lj_lattice(14, rc=3.4, seed=6, precision=precision)  # 2,744 particles, small enough for the resident engine
    want = _forces(s * 5)  # 13,720 particles: the row kernel
    for _ in range(5):
        got = _forces(s)
        assert all(np.array_equal(a, b[:s[0]["n"]]) for a, b in zip(got, want))
