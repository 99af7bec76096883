"""GPU: max_newton counts the updates of Algorithm 1's position half. One step
without forces or noise, where the number of float64 Newton updates each
particle needs is known from a numpy iteration of the same residual: a cap of
that many converges, one less reports MD_FLAG_RATTLE_DIVERGED, on the surfaces whose
solve starts in float32 (plane, sphere, ellipsoid, cylinder in float64; the
thylakoid's planes and cylinders on the mixed path), with the exact and the
frozen normal, and for lengths whose coefficients leave float32's range."""
import numpy as np
import pytest

import oracle
from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu

TOL = 1e-12
SURF = {"plane": (0.6, -0.3, 0.9), "sphere": (10.0, 0.0, 0.0), "ellipsoid": (15.0, 12.0, 9.0), "cylinder": (6.0, 2.0, 0.0)}


def _g(kind, p, x):
    if kind == "plane":
        return x @ p, np.broadcast_to(p, x.shape)
    if kind == "ellipsoid":
        w = x / p ** 2
        return (w * x).sum(1) - 1.0, 2.0 * w
    y = x * (np.array([1.0, 1.0, 0.0]) if kind == "cylinder" else 1.0)
    return (y * y).sum(1) - p[0] ** 2, 2.0 * y


def _newton(kind, p, x, v, dt, frozen, updates):
    """|g| / |grad g(x^k)| after 0, 1, ... updates, and the last iterate."""
    _, n0 = _g(kind, p, x)
    nn = (n0 * n0).sum(1)
    y = x + dt * (v - ((n0 * v).sum(1) / nn)[:, None] * n0)
    mu, off = np.zeros(len(x)), []
    for _ in range(updates + 1):
        z = y - mu[:, None] * n0
        g, n1 = _g(kind, p, z)
        off.append(np.abs(g) / np.sqrt(nn))
        mu = mu + g / (nn if frozen else (n1 * n0).sum(1))
    return np.array(off), z


def _points(kind, scale, n=600):
    g = I.rng(11, 3)
    p = np.array(SURF[kind])
    if kind == "plane":
        x = g.uniform(-9, 9, (n, 3))
        x -= ((x @ p) / (p @ p))[:, None] * p
    else:
        x = I.sample_surface({"kind": kind, "center": (0.0, 0.0, 0.0), "p": tuple(p)}, n, g, box=((-9,) * 3, (9,) * 3))
    if kind in ("sphere", "ellipsoid"):
        p = p * scale
    return x * scale, 4.0 * scale * g.standard_normal((n, 3)), p


@pytest.mark.parametrize("kind,frozen,scale", [(k, f, 1.0) for k in SURF for f in (0, 1)] +
                         [("ellipsoid", 0, 2.0 ** -40), ("sphere", 0, 2.0 ** -80)])
def test_cap_counts_float64_updates(kind, frozen, scale):
    dt, tol = 0.002, TOL * scale
    x, v, p = _points(kind, scale)
    off, z = _newton(kind, p, x, v, dt, frozen, 8)
    # particles whose residual is within a factor of the tolerance at some update are left out: rounding decides there
    clear = ((off < 0.5 * tol) | (off > 2.0 * tol)).all(axis=0)
    x, v, off, z = x[clear], v[clear], off[:, clear], z[clear]
    assert len(x) > 300
    surf = {"kind": kind, "center": (0.0, 0.0, 0.0), "p": tuple(SURF[kind]) if kind in ("plane", "cylinder") else tuple(p)}
    for cap in (1, 2, 3):
        prm = I.noninteracting(I.wca_params(precision="fp64", gamma=0.0, kT=0.0, dt=dt, rattle_tol=tol, max_newton=cap,
                                            frozen_normal=frozen, box_lo=(-9.5,) * 3, box_hi=(9.5,) * 3,
                                            periodic=(0, 0, 1) if kind == "cylinder" else (0, 0, 0)))
        with md.Simulation([I._system(kind, surf, prm, x, v)]) as sim:
            sim.set_state()
            sim.step(1)
            flags = md.md_status(sim.h)
            got = sim.state()["x"]
        converges = bool((off[:cap + 1] < tol).any(axis=0).all())
        assert flags == (0 if converges else md.MD_FLAG_RATTLE_DIVERGED), (cap, flags)
        if converges:  # stops within tol of the surface along n0 (times 1.1 for |n1| against |n0|), and some roundings
            assert np.abs(got - z).max() < 1.1 * tol + 1e-14 * np.abs(x).max()


def test_thylakoid_pieces_take_the_callers_updates():
    surf = I.thylakoid_surface()
    g = I.rng(7, 1)
    x = I.sample_thylakoid(surf, 2000, g, 30.0)
    v = 3.0 * g.standard_normal(x.shape)
    prm = I.noninteracting(I.wca_params(precision="mixed", gamma=0.0, kT=0.0, dt=0.01, rattle_tol=TOL, box_lo=(-33, -15, -15),
                                        box_hi=(33, 15, 15), periodic=(0, 0, 1)))
    con = np.ones(len(x), np.uint8)
    ref = oracle.System(surf, prm, len(x))
    ref.set_state(x, v, np.zeros(len(x), np.int32), None, con)
    ref.step(1)
    # a normal displacement of at most (4.5 * 3 * 0.01)^2 / (2 * 1.5) = 6e-3 on curvature 1 / 1.5 leaves 2.5e-5, 4e-10
    # and 1e-19 after one, two and three updates; only a few particles are that fast
    for cap, flagged in ((1, True), (3, False)):
        with md.Simulation([I._system("thylakoid", surf, dict(prm, max_newton=cap), x, v, None, con)]) as sim:
            sim.set_state()
            sim.step(1)
            assert md.md_status(sim.h) == (md.MD_FLAG_RATTLE_DIVERGED if flagged else 0), cap
            got = sim.state()["x"]
    # both stop within 1e-12 of the surface; double-float rounds at 2^-46 of lengths up to 30 (4e-13), a few times
    assert np.abs(got - ref.state()["x"]).max() < 4e-12
