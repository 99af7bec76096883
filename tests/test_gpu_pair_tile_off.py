"""GPU: MD_OPT_PAIR_TILE = 0 holds as set. A dense large system takes the tiled
kernel while nothing is set; with 0 set it takes the row kernel: the bits of
the same system batched with a sparse one (whose handle takes the row kernel by
itself) and a trajectory's too."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


def _run(systems, tile):
    with md.Simulation(systems) as sim:
        if tile is not None:
            md.md_set_option(sim.h, md.MD_OPT_PAIR_TILE, tile)
        assert md.md_get_option(sim.h, md.MD_OPT_PAIR_TILE) == (tile or 0)
        sim.set_state()
        f, u = sim.forces()
        sim.step(20)
        sim.sync()
        return f, u, sim.state()["x"]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_zero_is_the_row_kernel(precision):
    dense = I.lj_lattice(24, seed=3, precision=precision)
    # 72^3 cells for 200 particles more: one candidate in 27 cells on average
    sparse = I.sphere_system(n=200, R=40.0, seed=2, precision=precision, tol=1e-10, dt=0.001)
    for key in ("ntypes", "eps", "sigma", "rcut", "mass"):
        sparse["params"][key] = dense[0]["params"][key]
    n = dense[0]["n"]
    row = _run([dense[0], sparse], None)
    off = _run(dense, 0)
    assert all(np.array_equal(a, b[:n]) for a, b in zip(off, row))
    tiled = _run(dense, 8)
    assert all(np.array_equal(a, b) for a, b in zip(_run(dense, None), tiled))
    assert not np.array_equal(tiled[0], off[0])
