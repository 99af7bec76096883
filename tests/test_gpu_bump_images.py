"""GPU: particles on a Gaussian bump that cross from one periodic image of it
into the next, in a box so narrow that the bump is high at the crossing. The
surface has a crease there; in both precisions the step ends on the image the
particle has come to, as in the oracle."""
import numpy as np
import pytest

import oracle
from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("center", [(0.0, 0.0, 0.0), (0.7, -1.3, 0.4)])
@pytest.mark.parametrize("image", [0, 3])
def test_crossing_into_the_next_image(precision, center, image):
    A, w, L, n, steps = 5.0, 4.0, 12.0, 2000, 6
    surf = {"kind": "gaussian_bump", "center": center, "p": (A, w, 0.0, 0.0)}
    prm = I.noninteracting(I.wca_params(precision=precision, gamma=0.0, kT=0.0, dt=0.01, rattle_tol=1e-10,
                                        box_lo=(-L / 2, -L / 2, -3.0), box_hi=(L / 2, L / 2, A + 3.0), periodic=(1, 1, 0)))
    g = I.rng(3, 3)
    x = I.sample_surface(surf, n, g, box=((-L / 2, -L / 2, 0.0), (L / 2, L / 2, 0.0)))
    x[:, :2] += image * L
    v = I.maxwell(n, 1.0, 1.0, g)
    sy = I._system("bump", surf, prm, x, v)
    ref = oracle.System(surf, prm, n)
    ref.set_state(x, v, sy["type"], None, sy["constrained"])
    with md.Simulation([sy]) as sim:
        sim.set_state()
        for _ in range(steps):
            sim.step(1)
            ref.step(1)
            assert sim.residual()["max_g_over_gradg"] < 1e-10
        sim.sync()
        got = sim.state()["x"]
    want = ref.state()["x"]
    crossed = (np.round((x - center)[:, :2] / L) != np.round((want - center)[:, :2] / L)).any(1)
    assert crossed.sum() >= 10
    # each side stops within 1e-10 of the surface in every step, along normals of slope at most A / (w sqrt(e)) = 0.76
    # (1 / cos: 1.26); a velocity that differs by 2e-10 / dt carries it on, at most `steps` times
    assert np.abs(got - want).max() < 2 * 1.26 * 1e-10 * steps * (steps + 1)
