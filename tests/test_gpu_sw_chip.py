"""The 2DSW steps of a grid that fits on the chip (csrc/sw_chip.cuh, the
automatic tiling) against the streaming kernel, bit for bit: every count of
cells per thread, one tile and many, ragged tiles, tiles narrower than their
halo, calls shorter and longer than the steps between exchanges, and calls
that follow one another."""
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


def case(nx, ny, seed):
    """A wet/dry rectangle cut from the square workload."""
    base = inputs.sw_wetdry(n=max(nx, ny, 40), seed=seed, sample=64, bisect_iters=16)
    return inputs.SWInput(nx, ny, base.dx, base.dy, base.dt, base.H[:ny, :nx].copy(), base.eta0[:ny, :nx].copy(),
                          hmin=base.hmin)


@pytest.mark.parametrize("nx,ny", [(2, 2), (7, 3), (33, 40), (100, 100), (5, 700), (900, 4), (257, 190), (500, 500),
                                   (640, 411), (801, 777), (1000, 1000), (1100, 1020), (1400, 900)])
def test_chip_steps_bitwise(SW, nx, ny):
    inp = case(nx, ny, seed=nx + ny)
    calls = (1, 2, 3, 4, 5, 31, 0, 64)
    with SW(inp.params(), inp.H, inp.eta0) as g:
        g.set_tiling(1, 0)
        for n in calls:
            g.step(n)
        ref, vref = g.get_state(), g.volume()
    with SW(inp.params(), inp.H, inp.eta0) as g:
        for n in calls:
            g.step(n)
        got, vgot = g.get_state(), g.volume()
        for f in ("eta", "u", "v", "wet"):
            assert np.array_equal(got[f], ref[f]), f
        assert vgot == vref
        g.set_state(eta=inp.eta0.astype(np.float32), u=np.zeros((ny, nx + 1), np.float32),
                    v=np.zeros((ny + 1, nx), np.float32))
        g.step(sum(calls))
        again = g.get_state()
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(again[f], ref[f]), f
