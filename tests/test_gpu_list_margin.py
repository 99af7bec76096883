"""GPU, float64 Verlet list: a pair at the very cutoff of its types. The list
build and the list walk test in float32 on rounded records; what is listed and
what is evaluated is decided in float64: a pair a part in 1e9 outside r_c + skin
takes no entry of a full list, one as far inside does, and pairs just inside a
cutoff much shorter than the cell edge give the per-lane walk's bits."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs, md

pytestmark = pytest.mark.gpu


def _directions(g, m):
    u = g.normal(size=(m, 3))
    return u / np.linalg.norm(u, axis=1)[:, None]


def _sites(g, k, a):
    """k^3 points a apart (each moved by up to 1) in a periodic cube of edge k a about 0."""
    idx = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)
    return (idx + 0.5) * a - 0.5 * k * a + g.uniform(-1, 1, idx.shape)


def _free(x, prm, types=None):
    return [inputs._system("free", {"kind": "none", "center": (0.0,) * 3, "p": (0.0,) * 4}, prm, x,
                           np.zeros_like(x), types)]


@pytest.mark.parametrize("side", [1, -1])
def test_a_full_list_counts_only_pairs_within_the_skin(side):
    g = np.random.default_rng(5)
    at = _sites(g, 4, 10.0)
    u = _directions(g, at.shape[0])
    rs = 1.5 + 0.3
    x = np.concatenate([at, at + u, at - u * (rs * (1 + side * 1e-9))])  # the second within r_c of the first only
    prm = inputs.wca_params(precision="fp64", box_lo=(-20.0,) * 3, box_hi=(20.0,) * 3, periodic=(1, 1, 1),
                            cell_size=2.5)
    prm["rcut"][0, 0] = 1.5
    with md.Simulation(_free(x, prm)) as sim:
        md.md_set_neighbor_list(sim.h, 0.3, 1)
        if side > 0:
            sim.set_state()
            sim.sync()
        else:
            with pytest.raises(md.MdError) as e:
                sim.set_state()
                sim.sync()
            assert e.value.code == md.MD_ERR_NLIST_FULL


def test_pairs_just_inside_a_short_cutoff_are_evaluated():
    g = np.random.default_rng(6)
    k, a, rc = 14, 8.0, 0.3
    at = _sites(g, k, a)
    x = np.concatenate([at, at + _directions(g, at.shape[0]) * (rc * (1 - 1e-9))])
    h = 0.5 * k * a
    prm = inputs.wca_params(ntypes=2, precision="fp64", box_lo=(-h,) * 3, box_hi=(h,) * 3, periodic=(1, 1, 1),
                            cell_size=4.0)
    prm["rcut"][:, :] = 3.0
    prm["rcut"][1, 1], prm["sigma"][1, 1] = rc, 0.25
    got = []
    for queue in (0, 1):
        with md.Simulation(_free(x, prm, np.ones(x.shape[0], np.int32))) as sim:
            md.md_set_option(sim.h, md.MD_OPT_PAIR_QUEUE, queue)
            md.md_set_neighbor_list(sim.h, 0.2, 16)
            sim.set_state()
            got.append(sim.forces())
    assert np.all(np.abs(got[0][0]).max(axis=1) > 0.1)  # every pair counts: the force at the cutoff is not zero
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
