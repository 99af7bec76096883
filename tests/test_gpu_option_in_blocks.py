"""GPU: an option that changes bits, set between blocks of steps, takes effect at
once: the run equals one cut into single steps with the same switch at the same
step, and differs from the run without it."""
import numpy as np
import pytest

from paper_1411_3019_gb300 import inputs as I, md

pytestmark = pytest.mark.gpu


def _run(cuts, precision, switch):
    s = I.sphere_system(n=700, R=12.0, seed=2, dmin=0.9, precision=precision, dt=0.002, tol=1e-10)
    s["params"] = dict(s["params"], cell_size=float(np.max(s["params"]["rcut"])) + 0.3)
    with md.Simulation([s]) as sim:
        sim.set_state()
        for k, n in enumerate(cuts):
            if k == len(cuts) // 2 and switch == "lanes":
                md.md_set_option(sim.h, md.MD_OPT_PAIR_LANES, 2)
            if k == len(cuts) // 2 and switch == "list":
                md.md_set_neighbor_list(sim.h, 0.3, 64)
            sim.step(n)
        sim.sync()
        st = sim.state()
    return [st[k] for k in ("x", "v", "p_half", "step")]


# (in float64 another order of a WCA particle's few terms is lost in the rounding of the momentum)
@pytest.mark.parametrize("switch,precision", [("lanes", "mixed"), ("list", "mixed"), ("list", "fp64")])
def test_a_switch_between_blocks(switch, precision):
    blocks = _run([100, 100], precision, switch)  # eight-step blocks run from step 64 on
    singles = _run([1] * 200, precision, switch)
    assert all(np.array_equal(a, b) for a, b in zip(blocks, singles))
    plain = _run([100, 100], precision, None)
    assert not np.array_equal(blocks[0], plain[0])
