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
