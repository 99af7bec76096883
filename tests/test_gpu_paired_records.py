"""GPU: the mixed list of a handle on either side of the size from which a
slot's record and low part share a sector: the queued and the per-lane walk give
the same bits, and switching the list off and on again gives the cell list's
forces and the same list's."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [94, 95])  # 830,584 and 857,375 particles
def test_list_on_and_off(k):
    s = I.lj_lattice(k, rc=1.3, seed=3, precision="mixed")
    s[0]["params"] = dict(s[0]["params"], cell_size=1.6)
    with md.Simulation(s) as sim:
        sim.set_state()
        cells = sim.forces()
        md.md_set_neighbor_list(sim.h, 0.3, 32)
        queued = sim.forces()
        md.md_set_option(sim.h, md.MD_OPT_PAIR_QUEUE, 0)
        lanes = sim.forces()
        md.md_set_neighbor_list(sim.h, 0.0)
        off = sim.forces()
        md.md_set_option(sim.h, md.MD_OPT_PAIR_QUEUE, 1)
        md.md_set_neighbor_list(sim.h, 0.3, 32)
        again = sim.forces()
        sim.step(12)
        sim.sync()
        f, _ = sim.forces()
        x = sim.state()["x"]
        md.md_set_neighbor_list(sim.h, 0.0)
        g, _ = sim.forces()
    for a in (lanes, again):
        assert np.array_equal(a[0], queued[0]) and np.array_equal(a[1], queued[1])
    assert np.array_equal(off[0], cells[0]) and np.array_equal(off[1], cells[1])
    # at most 18 neighbours, terms of at most 500 eps/sigma at 0.96 sigma; two float32 sums of them in different orders
    assert np.abs(queued[0] - cells[0]).max() < 18 * 500 * 2 * 2.0 ** -24
    assert np.isfinite(x).all() and np.abs(f - g).max() < 18 * 500 * 2 * 2.0 ** -24
