"""Every kernel of the one-launch 2DSW path (csrc/sw_chip.cuh: 1 .. 14 cells per
thread) with every number of steps between exchanges, one column or row of
tiles and many, the last tiles smaller than the first, tiles narrower than
their halo, against the streaming kernel bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# grid: tiles in x, tiles in y, steps between exchanges, cells per thread, on 152 SMs
PLANS = [
    ((2, 3), (1, 1, 1, 1)), ((133, 134), (4, 34, 2, 1)), ((1992, 15), (143, 1, 2, 1)), ((23, 909), (1, 114, 2, 1)),
    ((1079, 7), (50, 3, 3, 1)), ((1910, 5), (107, 1, 3, 1)), ((8, 895), (1, 69, 3, 1)), ((184, 13), (16, 7, 4, 1)),
    ((797, 5), (100, 1, 4, 1)), ((4, 74), (1, 9, 4, 1)), ((59, 1216), (2, 68, 2, 2)), ((41, 1458), (1, 122, 2, 2)),
    ((142, 343), (5, 29, 3, 2)), ((23, 1794), (1, 106, 3, 2)), ((1573, 19), (69, 2, 4, 2)), ((1852, 18), (133, 1, 4, 2)),
    ((19, 1587), (1, 123, 4, 2)), ((1442, 86), (25, 6, 2, 3)), ((63, 1883), (1, 145, 2, 3)), ((372, 284), (15, 10, 3, 3)),
    ((395, 476), (7, 21, 2, 4)), ((89, 1883), (1, 145, 2, 4)), ((678, 211), (15, 10, 3, 4)), ((170, 1548), (3, 50, 2, 5)),
    ((654, 328), (15, 10, 3, 5)), ((1680, 180), (19, 8, 2, 6)), ((594, 455), (15, 10, 3, 6)), ((275, 1320), (3, 49, 2, 7)),
    ((362, 918), (6, 25, 3, 7)), ((1523, 267), (14, 10, 2, 8)), ((213, 1881), (4, 38, 3, 8)), ((979, 500), (8, 19, 2, 9)),
    ((1447, 376), (15, 10, 2, 10)), ((371, 1771), (4, 38, 2, 11)), ((431, 1562), (3, 49, 2, 12)), ((1496, 527), (15, 10, 2, 13)),
    ((1278, 657), (10, 15, 2, 14)),
]


@pytest.fixture(scope="module")
def SW():
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.sw import SW
    return SW


def case(nx, ny):
    """Hills and basins with rough ground, a third of the cells dry, and a wavy surface."""
    rng = np.random.default_rng(nx * 10007 + ny)
    x, y = np.arange(nx), np.arange(ny)[:, None]
    H = 6.0 + 15.0 * np.sin(x / 11.0 + 1.0) * np.cos(y / 13.0) + rng.uniform(-0.3, 0.3, (ny, nx))
    eta = np.maximum(0.4 * np.cos(x / 7.0) * np.cos(y / 5.0), -H)
    return dict(nx=nx, ny=ny, dx=10.0, dy=10.0, dt=0.1), H, eta


def test_every_count_of_cells_is_here():
    assert {p[3] for _, p in PLANS} == set(range(1, 15))


@pytest.mark.parametrize("size,plan", PLANS, ids=["%dx%d" % s for s, _ in PLANS])
def test_chip_plans_bitwise(SW, size, plan):
    import torch
    p, H, eta = case(*size)
    calls = (1, 2, 3, 5, 31, 0, 64)
    out = []
    for launches in (True, False):
        with SW(p, H, eta) as g:
            if launches:
                g.set_tiling(1, 0)
                assert g.chip_plan() is None
            elif torch.cuda.get_device_properties(0).multi_processor_count == 152:
                assert g.chip_plan() == plan
            for n in calls:
                g.step(n)
            out.append((g.get_state(), g.volume()))
    (ref, vref), (got, vgot) = out
    for f in ("eta", "u", "v", "wet"):
        assert np.isfinite(ref[f]).all() and np.array_equal(got[f], ref[f]), f
    assert vgot == vref
