"""GPU: float64 list walk and stored normals. The queued walk (screened in
float32, float64 terms on full warps) gives the per-lane walk's bits for every
warp width, in forces, energies and a trajectory across rebuilds; stored normals
give the redrawn ones' bits with and without the list, in both precisions,
through a restore."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs, md

pytestmark = pytest.mark.gpu


def _systems(kind, precision):
    tol = 1e-12 if precision == "fp64" else 1e-10
    if kind == "sphere":
        return [inputs.sphere_system(n=1033, R=14.0, seed=2, dmin=0.9, precision=precision, dt=0.002, tol=tol)]
    if kind == "beads":
        return inputs.c5_bead_molecules(nmol=150, R=7.0, seed=4, precision=precision, tol=tol)
    if kind == "bump":
        return inputs.c3_bump_crowders(n_surf=600, n_free=1500, seed=5, precision=precision, tol=tol)
    if kind == "batch":
        return inputs.c4_replicas(nrep=5, seed=8, nmin=30, nmax=400, rmin=5.0, rmax=9.0, precision=precision, tol=tol)
    return inputs.nve_systems(1, n=300, precision=precision, tol=tol)


def _run(kind, precision, skin, opts, steps=(25, 15)):
    systems = _systems(kind, precision)
    for s in systems:
        if skin:
            s["params"] = dict(s["params"], cell_size=float(np.max(s["params"]["rcut"])) + skin)
    with md.Simulation(systems) as sim:
        for key, val in opts.items():
            md.md_set_option(sim.h, key, val)
        if skin:
            md.md_set_neighbor_list(sim.h, skin, 128)
        sim.set_state()
        f0 = sim.forces()
        sim.step(steps[0])
        st = sim.state()
        md.md_restore(sim.h, st["x"], st["p_half"], st["step"])
        sim.step(steps[1])
        sim.sync()
        st = sim.state()
        f1 = sim.forces()
    return [f0[0], f0[1], st["x"], st["v"], st["p_half"], f1[0], f1[1]]


@pytest.mark.parametrize("kind", ["sphere", "beads", "bump", "batch", "nve"])
def test_float64_walks_give_the_same_bits(kind):
    ref = _run(kind, "fp64", 0.2, {md.MD_OPT_PAIR_QUEUE: 0})
    for width in (32, 16, 8):
        got = _run(kind, "fp64", 0.2, {md.MD_OPT_PAIR_QUEUE: 1, md.MD_OPT_LIST_WARP: width})
        assert all(np.array_equal(a, b) for a, b in zip(ref, got)), width


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("kind,skin", [("sphere", 0.0), ("sphere", 0.3), ("bump", 0.0), ("batch", 0.0)])
def test_stored_normals_give_the_same_bits(kind, skin, precision):
    a = _run(kind, precision, skin, {md.MD_OPT_STORE_NOISE: 1})
    b = _run(kind, precision, skin, {md.MD_OPT_STORE_NOISE: 0})
    assert all(np.array_equal(p, q) for p, q in zip(a, b))
