"""GPU: the pair kernel a dense large system takes by default (the cell-tiled
one, 8 particles per warp) against the same handle's other kernels."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs, md

pytestmark = pytest.mark.gpu


def _forces(systems, opts):
    with md.Simulation(systems) as sim:
        for key, val in opts.items():
            md.md_set_option(sim.h, key, val)
        sim.set_state()
        return sim.forces()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("k,rc", [(24, 2.5), (25, 2.5), (26, 4.0)])
def test_dense_default(k, rc, precision):
    systems = inputs.lj_lattice(k, rc=rc, seed=3, precision=precision)
    f, u = _forces(systems, {})
    ft, ut = _forces(systems, {md.MD_OPT_PAIR_TILE: 8})
    assert np.array_equal(f, ft) and np.array_equal(u, ut)
    fl, ul = _forces(systems, {md.MD_OPT_PAIR_LANES: 2})
    # another order of up to 210 terms of at most 150 eps/sigma: each addition rounds a partial sum of that size
    # (and two kernels' roundings add): 210 * 150 * 2^-24 * 2 in float32, 2^-53 in float64
    tol = 210 * 150 * 2.0 * (2.0 ** -53 if precision == "fp64" else 2.0 ** -24)
    assert np.abs(f - fl).max() < tol and np.abs(u - ul).max() < tol
