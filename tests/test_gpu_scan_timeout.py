"""GPU: steps that go on after a scan of the bucket counters has timed out. The
bucket bounds are then in range but need not ascend; every pair kernel stays in
bounds and ends, the next synchronising call reports MD_ERR_TIMEOUT, and after a
restore the run repeats one that never timed out bit for bit."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


def _systems(kind, precision):
    if kind == "surfaces":
        return I.c2_ellipsoid_torus(n_ell=4000, n_tor=1500, seed=8, precision=precision)
    return I.lj_lattice(52, rc=2.5, seed=3, precision=precision)  # the tiled kernel by default


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("kind,options", [("surfaces", {}), ("surfaces", {md.MD_OPT_PAIR_TILE: 8}),
                                          ("surfaces", {md.MD_OPT_PAIR_TILE: 32}), ("surfaces", {md.MD_OPT_PAIR_LANES: 4}),
                                          ("liquid", {})])
def test_steps_after_a_timed_out_scan(kind, options, precision):
    with md.Simulation(_systems(kind, precision)) as sim:
        for key, val in options.items():
            md.md_set_option(sim.h, key, val)
        sim.set_state()
        assert md.md_cell_list(sim.h)["bucket_start"].shape[0] - 1 > 8192  # more than one scan tile
        sim.step(2)
        start = sim.state()
        sim.step(3)
        sim.sync()
        want = sim.state()
        md.md_restore(sim.h, start["x"], start["p_half"], start["step"])
        md.md_set_option(sim.h, md.MD_OPT_SPIN_LIMIT, 0)
        sim.step(4)  # the second step's pair kernel takes the first one's broken list
        assert md.md_status(sim.h) & md.MD_FLAG_TIMEOUT
        md.md_set_option(sim.h, md.MD_OPT_SPIN_LIMIT, 1 << 22)
        md.md_restore(sim.h, start["x"], start["p_half"], start["step"])
        sim.step(3)
        sim.sync()
        got = sim.state()
    for key in ("x", "v", "p_half"):
        assert np.array_equal(got[key], want[key]), key


@pytest.mark.parametrize("skin", [0.0, 0.3])
def test_first_list_timed_out(skin):
    """A state whose first cell list is cut short is refused with MD_ERR_TIMEOUT; set again, the run is the usual one."""
    systems = _systems("surfaces", "mixed")
    if skin:
        for s in systems:
            s["params"] = dict(s["params"], cell_size=float(np.max(s["params"]["rcut"])) + skin)
    got = []
    for limit in (1 << 22, 0):
        with md.Simulation(systems) as sim:
            if skin:
                md.md_set_neighbor_list(sim.h, skin, 64)
            md.md_set_option(sim.h, md.MD_OPT_SPIN_LIMIT, limit)
            if limit == 0:
                with pytest.raises(md.MdError) as e:
                    sim.set_state()
                assert e.value.code == md.MD_ERR_TIMEOUT
                md.md_set_option(sim.h, md.MD_OPT_SPIN_LIMIT, 1 << 22)
            sim.set_state()
            sim.step(3)
            sim.sync()
            got.append(sim.state()["x"])
    assert np.array_equal(got[0], got[1])


def test_what_is_read_after_a_timeout_has_a_rebuilt_list():
    """md_status reports and clears the timeout as md_sync does; forces read then, and the next md_step, have the cell
    list rebuilt first."""
    got = []
    for limit in (1 << 22, 0):
        with md.Simulation(_systems("surfaces", "mixed")) as sim:
            sim.set_state()
            md.md_set_option(sim.h, md.MD_OPT_SPIN_LIMIT, limit)
            sim.step(1)
            assert md.md_status(sim.h) == (0 if limit else md.MD_FLAG_TIMEOUT)
            md.md_set_option(sim.h, md.MD_OPT_SPIN_LIMIT, 1 << 22)
            f, u = sim.forces()
            sim.step(3)
            sim.sync()
            got.append([f, u, *(sim.state()[k] for k in ("x", "v", "p_half"))])
    assert all(np.array_equal(a, b) for a, b in zip(*got))
