"""GPU: the mixed path's thylakoid solve against the oracle for every particle:
all finite, all but a few equal to the two solves' tolerances, and those few,
where a particle within rounding of a junction takes the neighbouring piece,
within what the pieces differ by."""
import numpy as np
import pytest

import oracle
from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("image", [0, 1])
def test_every_particle(image):
    n, steps, dt = 6000, 5, 0.01
    surf = I.thylakoid_surface(center=(1.0, -2.0, 0.7))
    prm = I.noninteracting(I.wca_params(precision="mixed", dt=dt, gamma=0.0, rattle_tol=1e-10,
                                        box_lo=(-32, -16, -15.0), box_hi=(34, 14, 15.0), periodic=(0, 0, 1)))
    g = I.rng(16, 4)
    x = I.sample_thylakoid(surf, n, g, 30.0)
    x[:, 2] += 30.0 * image * g.integers(-4, 5, n)
    v = I.maxwell(n, 1.0, 1.0, g)
    ref = oracle.System(surf, prm, n)
    ref.set_state(x, v, np.zeros(n, np.int32), None, np.ones(n, np.uint8))
    ref.step(steps)
    with md.Simulation([I._system("thylakoid", surf, prm, x, v)]) as sim:
        sim.set_state()
        sim.step(steps)
        sim.sync()
        got = sim.state()["x"]
    assert np.isfinite(got).all()
    err = np.abs(got - ref.state()["x"]).max(axis=1)
    # stops within 1e-10 of the surface on both sides, each step's difference carried on by the velocity
    assert (err >= 2e-10 * steps * (steps + 1)).sum() <= n // 1000
    # another piece through the same tangent plane: |v dt|^2 / 2 times a curvature of at most 1 / 1.5, |v| up to 4.5,
    # carried on for the steps left
    assert err.max() < 0.5 * (4.5 * dt) ** 2 / 1.5 * steps
