"""Waits between thread blocks that give up (GBSW_FAULT=sync_timeout gives them
no budget): the kernels leave, the next synchronising call reports
GBSW_ERR_TIMEOUT, and work without the injection then runs as before."""
import numpy as np
import pytest

from paper_1711_04471_gb300 import inputs

pytestmark = pytest.mark.gpu

TIMEOUT = -6


@pytest.fixture(scope="module")
def N():
    import paper_1711_04471_gb300 as P
    P.build()
    from paper_1711_04471_gb300 import _native
    return _native


def rhs(nx, ny, nz):
    import torch
    return torch.randn((nz, ny, nx), generator=torch.Generator(device="cuda").manual_seed(nx), device="cuda")


def test_chip_steps_that_give_up_are_reported(N, monkeypatch):
    from paper_1711_04471_gb300.sw import SW
    inp = inputs.sw_hump(n=500)          # 147 tiles
    with SW(inp.params(), inp.H, inp.eta0) as g:
        g.set_tiling(3, 0)
        g.step(100)
        want = g.get_state()
    monkeypatch.setenv("GBSW_FAULT", "sync_timeout")
    for read in ("volume", "get_state"):
        with SW(inp.params(), inp.H, inp.eta0) as g:
            g.step(100)
            with pytest.raises(N.GBSWError) as e:
                getattr(g, read)()
            assert e.value.status == TIMEOUT
    monkeypatch.delenv("GBSW_FAULT")
    with SW(inp.params(), inp.H, inp.eta0) as g:
        g.step(100)
        got = g.get_state()
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(got[f], want[f]), f


# the whole solve in one launch; checks as kernels of their own with the rows
# in registers; and in shared memory (one row and plane per tile, so that a
# tile looks at its neighbours' flags as soon as it has published its own)
@pytest.mark.parametrize("shape", [(72, 48, 40), (256, 80, 96), (8192, 8, 4)])
@pytest.mark.parametrize("kw", [dict(tol=1e-6, max_iter=200), dict(tol=-1.0, max_iter=20)])
def test_solves_that_give_up_are_reported(N, monkeypatch, shape, kw):
    import torch
    from paper_1711_04471_gb300.les import poisson_solve
    b = rhs(*shape)
    first = torch.zeros_like(b)
    s0 = poisson_solve(first, b, 4.0, **kw)
    monkeypatch.setenv("GBSW_FAULT", "sync_timeout")
    with pytest.raises(N.GBSWError) as e:
        poisson_solve(torch.zeros_like(b), b, 4.0, **kw)
    assert e.value.status == TIMEOUT
    monkeypatch.delenv("GBSW_FAULT")
    again = torch.zeros_like(b)
    assert poisson_solve(again, b, 4.0, **kw) == s0
    assert torch.equal(again, first)


def test_a_finished_tile_does_not_hide_anothers_timeout(N, monkeypatch):
    """A right-hand side whose square sum is below 1e-60 is solved by the first
    check, so the last block to come to its barrier finishes while the others
    give up.  Should that be the first block, the one that writes the solve's
    result (its subnormal values take longer), the report must be the same."""
    import torch
    from paper_1711_04471_gb300.les import poisson_solve
    b = torch.zeros((96, 96, 128))
    b[:8, :8] = 1e-40           # the first of 12 x 12 tiles
    b = b.cuda()
    p = torch.zeros_like(b)
    monkeypatch.setenv("GBSW_FAULT", "sync_timeout")
    for _ in range(1000):
        with pytest.raises(N.GBSWError) as e:
            poisson_solve(p, b, 4.0)
        assert e.value.status == TIMEOUT


def test_a_torn_state_stays_reported_until_it_is_replaced(N, monkeypatch):
    from paper_1711_04471_gb300.sw import SW
    inp = inputs.sw_hump(n=500)
    with SW(inp.params(), inp.H, inp.eta0) as g:
        g.step(7)
        start = g.get_state()
        g.step(100)
        want, vol = g.get_state(), g.volume()

    def refused(call):
        with pytest.raises(N.GBSWError) as e:
            call()
        assert e.value.status == TIMEOUT

    with SW(inp.params(), inp.H, inp.eta0) as g:
        monkeypatch.setenv("GBSW_FAULT", "sync_timeout")
        g.step(100)
        refused(g.volume)
        monkeypatch.delenv("GBSW_FAULT")
        for call in (g.get_state, g.volume, lambda: g.step(1), lambda: g.autotune(10), g.get_state):
            refused(call)
        g.set_state(eta=start["eta"], u=start["u"])     # v is still torn
        refused(g.volume)
        g.set_state(eta=start["eta"], u=start["u"], v=start["v"])
        g.step(100)
        got = g.get_state()
        assert g.volume() == vol
        # a timeout that nobody has asked about yet does not outlive the state it tore
        monkeypatch.setenv("GBSW_FAULT", "sync_timeout")
        g.step(100)
        monkeypatch.delenv("GBSW_FAULT")
        g.set_state(eta=start["eta"], u=start["u"], v=start["v"])
        g.step(100)
        again = g.get_state()
        assert g.volume() == vol
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(got[f], want[f]), f
        assert np.array_equal(again[f], want[f]), f


def test_autotune_does_not_keep_or_report_a_trial_that_gave_up(N, monkeypatch):
    from paper_1711_04471_gb300.sw import SW
    inp = inputs.sw_hump(n=500)
    with SW(inp.params(), inp.H, inp.eta0) as a, SW(inp.params(), inp.H, inp.eta0) as b:
        a.step(100)
        want, vol = a.get_state(), a.volume()
        monkeypatch.setenv("GBSW_FAULT", "sync_timeout")
        b.autotune(trial_steps=12)
        b.step(100)                  # launches: they have no waits
        got = b.get_state()
        assert b.volume() == vol
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(got[f], want[f]), f


def test_a_fixed_solve_that_gave_up_leaves_no_stencil(N, monkeypatch):
    """The final residual of a fixed-count solve stores the stencil of p for
    the next solve's first one.  After a solve that gave up, the next forms it
    anew: a context whose p is written back (which drops the stencil) and one
    whose p is left alone go on alike."""
    from paper_1711_04471_gb300.les import LES
    p0 = np.random.default_rng(3).standard_normal((42, 50, 74))
    out = []
    for write_back in (True, False):
        with LES(72, 48, 40) as les:
            les.set_fixed_iterations(20)
            les.set("p", p0)
            monkeypatch.setenv("GBSW_FAULT", "sync_timeout")
            with pytest.raises(N.GBSWError) as e:
                les.step(1)
            assert e.value.status == TIMEOUT
            monkeypatch.delenv("GBSW_FAULT")
            if write_back:
                les.set("p", les.get("p"))
            les.step(2)
            out.append([les.get(f) for f in ("p", "u", "v", "w")])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("shape", [(72, 48, 40), (256, 80, 96), (8192, 8, 4)])
def test_solves_without_room_for_the_cooperative_kernel(N, monkeypatch, shape):
    """The half-sweep launches take over, with the same iterates; the residual
    norms are FP64 sums in another order."""
    import torch
    from paper_1711_04471_gb300.les import poisson_solve
    b = rhs(*shape)
    for kw in (dict(tol=1e-6, max_iter=200), dict(tol=-1.0, max_iter=21)):
        p, q = torch.zeros_like(b), torch.zeros_like(b)
        want = poisson_solve(p, b, 4.0, **kw)
        monkeypatch.setenv("GBSW_FAULT", "occupancy")
        got = poisson_solve(q, b, 4.0, **kw)
        monkeypatch.delenv("GBSW_FAULT")
        assert got[:2] == want[:2] and abs(got[2] - want[2]) <= 1e-12 * want[2]
        assert torch.equal(p, q)


def test_steps_without_room_for_the_cooperative_kernel(N, monkeypatch):
    from paper_1711_04471_gb300.sw import SW
    inp = inputs.sw_hump(n=300)
    out = []
    for fault in ("", "occupancy"):
        monkeypatch.setenv("GBSW_FAULT", fault)
        with SW(inp.params(), inp.H, inp.eta0) as g:
            g.step(50)
            out.append(g.get_state())
    for f in ("eta", "u", "v", "wet"):
        assert np.array_equal(out[0][f], out[1][f]), f
