"""GPU: the resident engine's kernels by the composed surfaces a handle has (none,
thylakoids, a bump, both) give the global engine's bits, with and without
bonds, walls and exclusions."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


def _thylakoid(n, seed):
    surf = I.thylakoid_surface()
    prm = I.wca_params(precision="mixed", dt=0.001, rattle_tol=1e-10, seed=seed, box_lo=(-33, -15, -15), box_hi=(33, 15, 15),
                       periodic=(0, 0, 1))
    g = I.rng(seed, 2)
    x = I.rsa(lambda k, m: I.sample_thylakoid(surf, m, g, 30.0), [n], 0.95, g, periodic=(0, 0, 1),
              box=((-33, -15, -15), (33, 15, 15)))[0]
    return I._system("thylakoid", surf, prm, x, I.maxwell(n, 1.0, 1.0, g))


def _systems(kind):
    bump = I.c3_bump_crowders(n_surf=150, n_free=400, seed=5, precision="mixed", tol=1e-10)
    sphere = I.sphere_system(n=300, R=8.0, seed=2, dmin=0.95, precision="mixed", tol=1e-10, dt=0.001)
    if kind == "none":
        return [sphere, I.sphere_system(n=200, R=7.0, seed=3, dmin=0.95, precision="mixed", tol=1e-10, dt=0.001)]
    if kind == "thylakoids":
        return [_thylakoid(400, 7), sphere, _thylakoid(300, 8)]
    if kind == "bump":
        return bump
    if kind == "both":
        return [*bump, _thylakoid(400, 9)]
    s = I.c5_bead_molecules(nmol=60, R=6.0, seed=4, precision="mixed", tol=1e-10)[0]  # bonds, exclusions, types
    t = _thylakoid(100, 10)
    for key in ("ntypes", "eps", "sigma", "rcut", "mass"):
        t["params"][key] = s["params"][key]
    return [s, t]


@pytest.mark.parametrize("kind", ["none", "thylakoids", "bump", "both", "bonded"])
def test_same_bits_as_the_global_engine(kind):
    out = []
    for engine in (0, 1):
        with md.Simulation(_systems(kind)) as sim:
            md.md_set_option(sim.h, md.MD_OPT_ENGINE, engine)
            sim.set_state()
            sim.step(30)
            sim.sync()
            st = sim.state()
            out.append([st["x"], st["v"], st["p_half"], *sim.forces()])
    assert all(np.array_equal(a, b) for a, b in zip(*out))
