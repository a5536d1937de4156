"""The pair that SW.autotune returns is the tiling it keeps: given to another
context of the same grid it takes the same path to the same state."""
import numpy as np
import pytest

from paper_1711_04471_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def SW():
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.sw import SW
    return SW


@pytest.mark.parametrize("n", [100, 300, 1100])
def test_autotuned_pair_is_the_one_kept(SW, n):
    from paper_1711_04471_gb300.sw import ONE_LAUNCH
    inp = inputs.sw_hump(n=n)
    with SW(inp.params(), inp.H, inp.eta0) as a, SW(inp.params(), inp.H, inp.eta0) as b:
        default = a.chip_plan()
        T, rows = a.autotune(trial_steps=60)
        plan = a.chip_plan()
        assert plan == (default if rows == ONE_LAUNCH else None)
        if plan:
            assert T == plan[2]
        b.set_tiling(T, rows)
        assert b.chip_plan() == plan
        a.step(50)
        b.step(50)
        x, y = a.get_state(), b.get_state()
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(x[f], y[f]), f


def test_one_launch_on_a_grid_that_does_not_fit(SW):
    """The launches run, as with any segment height beyond the grid's."""
    from paper_1711_04471_gb300.sw import ONE_LAUNCH
    inp = inputs.sw_hump(n=1100)
    out = []
    for tiling in ((2, 0), (2, ONE_LAUNCH)):
        with SW(inp.params(), inp.H, inp.eta0) as g:
            g.set_tiling(*tiling)
            assert g.chip_plan() is None
            g.step(9)
            out.append(g.get_state())
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(out[0][f], out[1][f]), f
