"""The pressure solve in one cooperative launch (csrc/poisson_tile.cuh)
against the half-sweep launches and the FP64 oracle, at the sizes where the
cut of the grid changes.

The grid is periodic in y, so a right-hand side that repeats after ny rows
gives an iterate that repeats after ny rows: doubling ny step by step takes
the same problem through every kind of tile (registers with one, two and
four groups per thread, shared memory with and without the residual) up to
a grid that only the half-sweep launches hold.  The start is zero, so every
path sees the same residual, and the iterates must agree bit for bit.
"""
import numpy as np
import pytest

import oracle
from oracle import les as ol

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def solve():
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300.les import poisson_solve
    return poisson_solve


def test_repeated_grid_gives_repeated_iterates(solve):
    import torch
    nx, nz, n = 256, 96, 12
    b = torch.randn((nz, 20, nx), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    first = None
    while b.shape[1] <= 640:     # 15.7 M cells: more than the shared memory of all SMs holds
        p = torch.zeros_like(b)
        st, it, rho = solve(p, b, 4.0, tol=-1.0, max_iter=n)
        assert (st, it) == (0, n)
        if first is None:
            first = p
        assert torch.equal(p, first.repeat(1, b.shape[1] // 20, 1)), b.shape
        b = torch.cat([b, b], 1)


@pytest.mark.parametrize("nx,ny,nz", [(2, 2, 2), (8, 2, 3), (9, 4, 2), (16, 16, 12), (33, 18, 7), (17, 64, 12),
                                      (72, 48, 40), (400, 20, 30), (1500, 6, 5), (64, 300, 3)])
def test_iterates_match_oracle(solve, nx, ny, nz):
    """7 iterations from a random start: 14 half-sweeps, each within a few
    FP32 roundings (at most 8 of 2^-24) of the FP64 update of values of the
    same size, so within 14 * 8 * 2^-24 = 7e-6 of the FP64 iterate."""
    import torch
    n = 7
    rng = np.random.default_rng(nx * 1000003 + ny * 1009 + nz)
    P = ol.make_params(nx, ny, nz, tol=0.0, max_iter=n)
    bo, po = ol.padded(P), ol.padded(P)
    bf, pf = (rng.standard_normal((nz, ny, nx)).astype(np.float32) for _ in range(2))
    ol.interior(bo)[:] = bf
    ol.interior(po)[:] = pf
    ol.sor(P, bo, po)
    p, b = torch.from_numpy(pf).cuda(), torch.from_numpy(bf).cuda()
    st, it, rho = solve(p, b, 4.0, tol=-1.0, max_iter=n)
    assert (st, it) == (0, n)
    want = ol.interior(po)
    assert np.linalg.norm(p.cpu().numpy() - want) <= 7e-6 * np.linalg.norm(want)
    assert abs(rho - ol.residual(P, bo, po)) <= 1e-4 * rho
