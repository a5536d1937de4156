"""The FP64 2DSW path at grids of more rows than a launch has blocks in y, and
at cell sizes that take every form of its division, against the FP64 oracle
bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1711_04471_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def SW64():
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.sw import SW64
    return SW64


@pytest.mark.parametrize("ny", [65535, 65536, 131075])
def test_tall_grids_are_set_up_and_read(SW64, ny):
    rng = np.random.default_rng(ny)
    H = rng.uniform(-1.0, 10.0, (ny, 3))
    eta = np.maximum(rng.uniform(-0.5, 0.5, (ny, 3)), -H)
    p = dict(nx=3, ny=ny, dx=10.0, dy=10.0, dt=0.1)
    with SW64(p, H, eta) as g:
        st = g.get_state()
        vol, wet = g.volume()
    assert np.array_equal(st["eta"], eta)
    assert np.array_equal(st["wet"], (H + eta > 0.05).astype(np.uint8))
    assert st["u"].shape == (ny, 4) and not st["u"].any()
    assert st["v"].shape == (ny + 1, 3) and not st["v"].any()
    assert vol == pytest.approx(100.0 * (H + eta).sum(), rel=1e-13)


@pytest.mark.parametrize("steps", [1, 16])
def test_a_step_that_cannot_be_launched_leaves_the_state(SW64, steps):
    """A step has a block row per grid row, so 70000 rows cannot be launched:
    the call fails, and the state reads as before it."""
    from paper_1711_04471_gb300._native import GBSWError
    rng = np.random.default_rng(1)
    H = rng.uniform(-1.0, 10.0, (70000, 3))
    with SW64(dict(nx=3, ny=70000, dx=10.0, dy=10.0, dt=0.1), H, np.maximum(0.0, -H)) as g:
        before = g.get_state()
        with pytest.raises(GBSWError) as e:
            g.step(steps)
        assert e.value.status == -2
        after = g.get_state()
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(before[f], after[f]), f


# |1 - RN(1/d) d| <= 2^-54 (one correction of the quotient) or more (two), and
# cell sizes past 2^100 either way (plain division)
@pytest.mark.parametrize("dx,dy", [(10.0, 12.5), (7.3, 3.7), (1.9999, 9.7), (1.3 * 2.0 ** -101, 1.7 * 2.0 ** -102),
                                   (1.3 * 2.0 ** 101, 1.7 * 2.0 ** 102), (7.3, 1.7 * 2.0 ** 5)])
def test_every_form_of_the_division_bitwise(SW64, dx, dy):
    base = inputs.sw_wetdry(n=90, seed=17)
    inp = inputs.SWInput(90, 90, dx, dy, 0.02 * min(dx, dy), base.H, base.eta0, hmin=base.hmin)
    o = oracle.SWState(inp.params(), inp.H, inp.eta0).run(150)
    with SW64(inp.params(), inp.H, inp.eta0) as g:
        g.step(150)
        st = g.get_state()
    assert np.abs(st["u"]).max() > 0 and np.isfinite(st["eta"]).all()
    assert np.array_equal(st["eta"], o.eta_i)
    assert np.array_equal(st["u"], o.u_f)
    assert np.array_equal(st["v"], o.v_f)
    assert np.array_equal(st["wet"], o.wet_i)
