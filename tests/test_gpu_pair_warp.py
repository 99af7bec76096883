"""GPU: the warp-per-particle pair kernel of small systems gives the row
kernel's bits. A handle takes the warp kernel up to 12,288 particles (mixed) or
8,192 (float64) and the row kernel above, and the systems of a batch never
interact, so one system alone (warp) and the same system as the first of
enough copies (row) must give the same forces and energies bit for bit: a
single particle, sizes around the queue's 32, open and hashed grids, a periodic
liquid with a long cutoff, bonds with exclusions and types, walls. (The row and
warp kernels against the oracle: the parity tests, above and below those
sizes.)"""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs, md

pytestmark = pytest.mark.gpu

LIMIT = {"mixed": 12288, "fp64": 8192}


def _system(kind, n, precision):
    if kind == "sphere":
        return inputs.sphere_system(n=n, R=max(2.0, 0.9 * n ** 0.5), seed=3, dmin=0.95, precision=precision, tol=1e-10)
    if kind == "crowded":  # about 40 candidates in the stencil
        return inputs.sphere_system(n=n, R=0.45 * n ** 0.5, seed=3, dmin=0.6, precision=precision, tol=1e-10)
    if kind == "liquid":
        return inputs.lj_lattice(n, seed=4, precision=precision)[0]
    if kind == "smooth":
        return inputs.nve_systems(1, n=n, precision=precision)[0]
    if kind == "beads":
        return inputs.c5_bead_molecules(nmol=n, R=max(4.0, 0.9 * n ** 0.5), seed=5, precision=precision)[0]
    return inputs.c3_bump_crowders(n_surf=n // 5, n_free=n - n // 5, seed=6, precision=precision)[0]


def _forces(systems):
    with md.Simulation(systems) as sim:
        sim.set_state()
        return sim.forces()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind,n", [("sphere", 5), ("sphere", 1000), ("sphere", 8192), ("crowded", 33), ("crowded", 700),
                                    ("liquid", 9), ("liquid", 12), ("smooth", 500), ("beads", 200), ("bump", 6000)])
def test_same_bits_as_the_row_kernel(kind, n, precision):
    s = _system(kind, n, precision)
    assert s["n"] <= LIMIT[precision]
    copies = LIMIT[precision] // s["n"] + 1
    f1, u1 = _forces([s])
    f2, u2 = _forces([s] * copies)
    assert np.array_equal(f1, f2[:s["n"]]) and np.array_equal(u1, u2[:s["n"]])
    assert np.abs(f1).max() > 0.0 or n < 10


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_one_particle(precision):
    f, u = _forces([_system("sphere", 1, precision)])
    assert not f.any() and not u.any()
