"""The workloads this library is timed on: what a user has it do, through
its public entry points, over the sizes its own tests, benchmark and
configurations use.

Kinds of case (see ``listed`` for what each listed one stands for):

``sw``        SW.step on one FP32 shallow-water grid, then the state on the host
``ensemble``  SWBatch.step over grids of uneven sizes, then volumes and states
``sw64``      SW64.step, the FP64 variant, then the state
``les``       LES.step: the urban LES, with a fixed SOR count or to a tolerance,
              from the previous pressure or with the learned warm start
``poisson``   poisson_solve on device tensors, to the default tolerance
``train``     UNet.train_step, then the parameters
``infer``     UNet.forward
"""
from __future__ import annotations

import math
import os
import random

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DEV = "cuda"


def listed():
    return [
        # The 100 x 100 hump basin in bursts of 30 steps, each followed by the
        # whole state: an interactive or coupled run.  Launches and copies count.
        dict(name="sw-hump-100", kind="sw", nx=100, ny=100, steps=30, basin="hump", tuned=False),
        # The paper's smallest grid, tuned once as the benchmark does, 1000 of
        # its 10,000 steps between two outputs.
        dict(name="sw-paper-500", kind="sw", nx=500, ny=500, steps=1000, basin="paper", tuned=True),
        # A ragged wet/dry grid of a few MB, as constructed (no tuning).
        dict(name="sw-ragged-1237x1501", kind="sw", nx=1237, ny=1501, steps=300, basin="wetdry", tuned=False),
        # The headline grid: 4096 x 4096 wet/dry, larger than any cache.
        dict(name="sw-wetdry-4096", kind="sw", nx=4096, ny=4096, steps=300, basin="wetdry", tuned=False),
        # An ensemble of uneven grids (sides 64 .. 1024), advanced together
        # between two outputs.
        dict(name="ensemble-20", kind="ensemble", members=20, draw=1002, nmin=64, nmax=1024, steps=600),
        # The FP64 variant on a ragged grid: a precision study.
        dict(name="sw64-700x501", kind="sw64", nx=700, ny=501, steps=100, basin="wetdry"),
        # The paper's UFLES setup: 300 x 300 x 90, 50 SOR iterations per step.
        dict(name="les-paper-300x300x90", kind="les", nx=300, ny=300, nz=90, steps=10, mode="fixed", iters=50,
             restart=False),
        # The benchmark's LES step: 256 x 256 x 128 to a 1e-6 residual with the
        # learned warm start, restarted from a checkpoint.
        dict(name="les-learned-256x256x128", kind="les", nx=256, ny=256, nz=128, steps=1, mode="learned", iters=0,
             restart=True),
        # A small street-canyon domain to the default tolerance from the
        # previous pressure: thousands of short sweeps.
        dict(name="les-plain-72x48x40", kind="les", nx=72, ny=48, nz=40, steps=2, mode="plain", iters=0, restart=True),
        # The stand-alone pressure solve with its default arguments.
        dict(name="poisson-160x96x64", kind="poisson", nx=160, ny=96, nz=64),
        # A training step of the warm-start network as its recipe runs it:
        # 32 coarse grids of 16 x 16 x 8.
        dict(name="train-32x8x16x16", kind="train", n=32, D=8, H=16, W=16),
        # The same on one large crop.
        dict(name="train-1x64x128x128", kind="train", n=1, D=64, H=128, W=128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(v):
    return v + (v & 1)


def draw(rng):
    kind = rng.choice(["sw", "sw", "ensemble", "sw64", "les", "les", "poisson", "poisson", "train", "infer"])
    if kind == "sw":
        nx, ny = _log(rng, 64, 4096), _log(rng, 64, 4096)
        steps = max(10, min(1000, int(3e9 / (nx * ny)))) + rng.randrange(0, 7)
        return dict(kind=kind, nx=nx, ny=ny, steps=steps, basin=rng.choice(["hump", "wetdry"]),
                    tuned=rng.random() < 0.25)
    if kind == "ensemble":
        return dict(kind=kind, members=rng.randrange(8, 21), draw=rng.randrange(1, 10 ** 6), nmin=64,
                    nmax=rng.choice([256, 512, 1024]), steps=rng.randrange(200, 600))
    if kind == "sw64":
        nx, ny = _log(rng, 64, 1024), _log(rng, 64, 1024)
        return dict(kind=kind, nx=nx, ny=ny, steps=max(10, min(300, int(3e7 / (nx * ny)))), basin="wetdry")
    if kind == "les":
        mode = rng.choice(["fixed", "fixed", "plain", "learned"])
        if mode == "fixed":
            nx, ny, nz = _log(rng, 32, 320), _even(_log(rng, 32, 320)), _log(rng, 16, 96)
            return dict(kind=kind, nx=nx, ny=ny, nz=nz, steps=rng.randrange(2, 10), mode=mode,
                        iters=rng.choice([20, 50, 100]), restart=True)
        if mode == "plain":
            nx, ny, nz = _log(rng, 24, 112), _even(_log(rng, 24, 112)), _log(rng, 16, 64)
            return dict(kind=kind, nx=nx, ny=ny, nz=nz, steps=rng.randrange(1, 3), mode=mode, iters=0,
                        restart=True)
        return dict(kind=kind, nx=256, ny=128 * rng.choice([1, 2]), nz=64 * rng.choice([1, 2]), steps=rng.randrange(1, 3),
                    mode=mode, iters=0, restart=True)
    if kind == "poisson":
        return dict(kind=kind, nx=_log(rng, 16, 176), ny=_even(_log(rng, 16, 176)), nz=_log(rng, 12, 96))
    if kind == "train":
        H, W = rng.choice([(16, 16), (32, 32), (64, 64)])
        D = 4 * rng.randrange(2, 13)
        return dict(kind=kind, n=_log(rng, 1, max(1, (1 << 20) // (D * H * W))), D=D, H=H, W=W)
    H, W = rng.choice([(16, 16), (32, 32), (64, 64), (128, 128)])
    return dict(kind="infer", n=rng.randrange(1, 5), D=4 * rng.randrange(2, 17), H=H, W=W)


# --------------------------------------------------------------- inputs


def _basin(basin, nx, ny, rng):
    """(params, H, eta0): a hump basin (its depth and place vary a little
    with the seed) or 15 % dry random bathymetry with a 0.5 m perturbation
    of the surface, both as separable sums (one matrix product each)."""
    x, y = np.arange(nx) + 0.5, np.arange(ny) + 0.5
    dx, dt = (1.0, 0.01) if basin == "paper" else (10.0, 0.1)
    if basin in ("hump", "paper"):
        n = min(nx, ny)
        sig = 5.0 if basin == "hump" else n / 20.0
        cx, cy = nx / 2 + rng.uniform(-0.1, 0.1) * nx, ny / 2 + rng.uniform(-0.1, 0.1) * ny
        eta = np.outer(np.exp(-((y - cy) ** 2) / (2 * sig * sig)), np.exp(-((x - cx) ** 2) / (2 * sig * sig)))
        H = np.full((ny, nx), 10.0 + rng.uniform(-0.5, 0.5))
    else:
        k = 32
        s = 0.06 * math.sqrt(nx * ny) * rng.uniform(0.5, 1.5, k)
        gx = np.exp(-((x[None] - rng.uniform(0, nx, k)[:, None]) ** 2) / (2 * s[:, None] ** 2))
        gy = np.exp(-((y[None] - rng.uniform(0, ny, k)[:, None]) ** 2) / (2 * s[:, None] ** 2))
        wl = np.exp(rng.uniform(math.log(min(64.0, min(nx, ny) / 4)), math.log(min(512.0, min(nx, ny))), 8))
        ang, ph = rng.uniform(0, 2 * math.pi, 8), rng.uniform(0, 2 * math.pi, 8)
        kx, ky = 2 * math.pi / wl * np.cos(ang), 2 * math.pi / wl * np.sin(ang)
        px, py = kx[:, None] * x[None] + ph[:, None], ky[:, None] * y[None]
        eta = np.cos(py).T @ np.cos(px) - np.sin(py).T @ np.sin(px)
        eta *= 0.5 / np.abs(eta).max()
        H = -60.0 * (gy.T @ gx)
        # the level that leaves 15 % of the cells dry; at most 60 m deep
        t = max(1, int(math.sqrt(nx * ny / 250000)))
        H -= np.quantile((H + eta)[::t, ::t], 0.15)
        np.minimum(H, 60.0, out=H)
    params = dict(nx=nx, ny=ny, dx=dx, dy=dx, dt=dt, g=9.81, eps=0.05, hmin=0.05)
    return params, H, np.maximum(eta, -H)


def _sizes(case):
    r = random.Random(case["draw"])
    return [int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** r.random())) for _ in range(case["members"])]


def _ensemble(case, seed):
    from paper_1711_04471_gb300 import inputs
    rng = np.random.default_rng(seed)
    out = []
    for n in _sizes(case):
        p, H, eta = _basin("wetdry", n, n, rng)
        x = np.arange(n) + 0.5
        g = np.exp(-((x - n / 2) ** 2) / 50.0)
        out.append(inputs.SWInput(n, n, p["dx"], p["dy"], p["dt"], H, np.maximum(eta + np.outer(g, g), -H)))
    return out


def _buildings(case, seed):
    from paper_1711_04471_gb300 import inputs
    return inputs.les_buildings(case["nx"], case["ny"], case["nz"], dx=4.0, seed=1003 + seed)


def _rhs(case, seed):
    """A smooth random right-hand side plus cell noise, and a zero guess."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    noise = torch.randn((nz, ny, nx), generator=g, device=DEV)
    low = torch.randn((1, 1, 6, 6, 6), generator=g, device=DEV)
    smooth = torch.nn.functional.interpolate(low, size=(nz, ny, nx), mode="trilinear")[0, 0]
    return (smooth + 0.25 * noise).contiguous()


def _pairs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    shape = (case["n"], case["D"], case["H"], case["W"])
    return torch.randn(shape + (2,), generator=g, device=DEV), 0.3 * torch.randn(shape, generator=g, device=DEV)


LAYERS = [(2, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 32), (64, 16), (32, 16)]


def _weights(seed):
    r = np.random.default_rng(seed + 7)
    parts = []
    for ci, co in LAYERS:
        parts += [r.standard_normal(27 * co * ci) * math.sqrt(2.0 / (27 * ci)), 0.01 * r.standard_normal(co)]
    parts += [0.25 * r.standard_normal(16), np.zeros(1)]
    return np.concatenate(parts).astype(np.float32)


# --------------------------------------------------------------- prepare and run


def _pinned(shape):
    return torch.empty(shape, dtype=torch.float32, pin_memory=True).numpy()


def prepare(case, seed):
    stream = torch.cuda.current_stream()
    kind = case["kind"]
    if kind == "sw":
        from paper_1711_04471_gb300.sw import SW
        p, H, eta = _basin(case["basin"], case["nx"], case["ny"], np.random.default_rng(seed))
        sw = SW(p, H, eta, stream=stream)
        if case["tuned"]:
            sw.autotune(trial_steps=120)
        nx, ny = case["nx"], case["ny"]
        return dict(case=case, sw=sw, eta=_pinned((ny, nx)), u=_pinned((ny, nx + 1)), v=_pinned((ny + 1, nx)))
    if kind == "sw64":
        from paper_1711_04471_gb300.sw import SW64
        p, H, eta = _basin(case["basin"], case["nx"], case["ny"], np.random.default_rng(seed))
        return dict(case=case, sw=SW64(p, H, eta, stream=stream))
    if kind == "ensemble":
        from paper_1711_04471_gb300.sw import SWBatch
        return dict(case=case, b=SWBatch(_ensemble(case, seed), stream=stream))
    if kind == "les":
        from paper_1711_04471_gb300.les import LES
        les = LES(case["nx"], case["ny"], case["nz"], _buildings(case, seed), stream=stream,
                  **(dict(check_every=500, max_iter=400000) if case["mode"] == "learned" else {}))
        st = dict(case=case, les=les)
        if case["mode"] == "fixed":
            les.set_fixed_iterations(case["iters"])
        elif case["mode"] == "learned":
            from paper_1711_04471_gb300.unet import UNet
            st["net"] = UNet(seed=0, stream=stream)
            st["net"].set_params(np.load(os.path.join(ROOT, "paper_1711_04471_gb300", "data", "unet_warmstart.npy")))
            les.set_warm_start(st["net"])
            les.step(3, stats=False)
        if case["restart"]:
            st["checkpoint"] = les.get_state()
        return st
    if kind == "poisson":
        b = _rhs(case, seed)
        return dict(case=case, b=b, p=torch.zeros_like(b), stream=stream)
    from paper_1711_04471_gb300.unet import UNet
    net = UNet(seed=0, stream=stream)
    net.set_params(_weights(seed))
    x, t = _pairs(case, seed)
    return dict(case=case, net=net, x=x, t=t)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sw":
        sw = state["sw"].step(case["steps"])
        vol = sw.volume()
        out = sw.get_state(eta=state["eta"], u=state["u"], v=state["v"], want=("eta", "u", "v"))
        return dict(eta=out["eta"], u=out["u"], v=out["v"], volume=vol)
    if kind == "sw64":
        return state["sw"].step(case["steps"]).get_state()
    if kind == "ensemble":
        b = state["b"]
        b.step(case["steps"])
        return dict(volumes=b.volumes(), states=[b.get_state(m) for m in range(case["members"])])
    if kind == "les":
        les = state["les"]
        if case["restart"]:             # every pass takes the same steps
            les.set_state(state["checkpoint"])
        if case["mode"] == "fixed":     # without a restart a pass goes on from the last one
            les.step(case["steps"], stats=False)
            return dict(u=les.get("u"), v=les.get("v"), w=les.get("w"), p=les.get("p"))
        stats = les.step(case["steps"])
        out = les.get_state()
        out["iters"] = [s["iters"] for s in stats]
        return out
    if kind == "poisson":
        from paper_1711_04471_gb300.les import poisson_solve
        p = state["p"].zero_()
        status, iters, _ = poisson_solve(p, state["b"], 4.0, stream=state["stream"])
        return dict(p=p, status=status, iters=iters)
    net = state["net"]
    if kind == "infer":
        return net.forward(state["x"])
    return dict(loss=net.train_step(state["x"], state["t"], 1e-3), params=net.get_params())


def work(case):
    """Inputs read once, outputs written once, and the arithmetic of the
    method (per cell and step: about 45 operations for 2DSW; about 420 for
    the LES predictor and 13 for an SOR update)."""
    kind = case["kind"]
    if kind in ("sw", "sw64"):
        cells = case["nx"] * case["ny"]
        return dict(bytes=(4 if kind == "sw" else 8) * 7 * cells, flops=45 * cells * case["steps"])
    if kind == "ensemble":
        cells = sum(n * n for n in _sizes(case))
        return dict(bytes=28 * cells, flops=45 * cells * case["steps"])
    if kind == "les":
        cells = case["nx"] * case["ny"] * case["nz"]
        its = case["iters"] if case["mode"] == "fixed" else 1000  # to a tolerance: of the order of 1000
        fields = 16 if case["mode"] == "fixed" else 88
        return dict(bytes=fields * cells + 24 * cells, flops=case["steps"] * cells * (420 + 13 * its))
    if kind == "poisson":
        cells = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=12 * cells, flops=13 * 1000 * cells)
    vox = case["n"] * case["D"] * case["H"] * case["W"]
    scale = [1, 1, 8, 8, 64, 64, 8, 1]
    fwd = sum(54 * ci * co / s for (ci, co), s in zip(LAYERS, scale)) * vox
    return dict(bytes=12 * vox + (0 if kind == "infer" else 3 * 806000), flops=fwd * (1 if kind == "infer" else 3))


# --------------------------------------------------------------- 64-bit results


def _sw_exact(p, H, eta, steps):
    H = torch.as_tensor(H, dtype=torch.float64, device=DEV)
    eta = torch.maximum(torch.as_tensor(eta, dtype=torch.float64, device=DEV), -H)
    u, v = torch.zeros_like(H), torch.zeros_like(H)
    rx, ry, q = p["dt"] / p["dx"], p["dt"] / p["dy"], 0.25 * p["eps"]

    def face(vel, c, e0, e1, w0, w1):
        a = vel - c * (e1 - e0)
        return torch.where((w0 & w1) | (w0 & (a > 0)) | (w1 & (a < 0)), a, torch.zeros_like(a))

    for _ in range(steps):
        h = H + eta
        wet = h > p["hmin"]
        u = torch.nn.functional.pad(face(u[:, :-1], p["g"] * rx, eta[:, :-1], eta[:, 1:], wet[:, :-1], wet[:, 1:]),
                                    (0, 1))
        v = torch.nn.functional.pad(face(v[:-1], p["g"] * ry, eta[:-1], eta[1:], wet[:-1], wet[1:]), (0, 0, 0, 1))
        F = torch.zeros_like(H)
        G = torch.zeros_like(H)
        F[:, :-1] = u[:, :-1].clamp(min=0) * h[:, :-1] + u[:, :-1].clamp(max=0) * h[:, 1:]
        G[:-1] = v[:-1].clamp(min=0) * h[:-1] + v[:-1].clamp(max=0) * h[1:]
        div = rx * F + ry * G
        div[:, 1:] -= rx * F[:, :-1]
        div[1:] -= ry * G[:-1]
        es = eta - div
        m = wet.to(torch.float64)
        a, cnt = m * es, torch.zeros_like(m)
        s = torch.zeros_like(m)
        for src, acc in ((a, s), (m, cnt)):
            acc[:, :-1] += src[:, 1:]
            acc[:, 1:] += src[:, :-1]
            acc[:-1] += src[1:]
            acc[1:] += src[:-1]
        eta = torch.where(wet, es + q * (s - cnt * es), es)
    return H, eta, u, v


def _sw_outputs(p, H, eta, u, v):
    area = p["dx"] * p["dy"]
    h = H + eta
    vol = (float(h.sum()) * area, float(h[h > p["hmin"]].sum()) * area)
    return dict(eta=eta, u=torch.nn.functional.pad(u, (1, 0)), v=torch.nn.functional.pad(v, (0, 0, 1, 0))), vol


class _Poisson:
    """The 7-point operator (Neumann at the inflow, ground and lid, p = 0 on
    the outflow face, periodic in y) and red-black SOR on it."""

    def __init__(self, nx, ny, nz, dx):
        k, j, i = torch.meshgrid(*[torch.arange(1, n + 1, device=DEV) for n in (nz, ny, nx)], indexing="ij")
        self.d = (6.0 - (i == 1).double() - (k == 1).double() - (k == nz).double() + (i == nx).double())
        self.red = ((i + j + k) % 2 == 0)
        self.h2 = dx * dx

    def near(self, p):
        s = torch.roll(p, 1, 1) + torch.roll(p, -1, 1)
        s[:, :, 1:] += p[:, :, :-1]
        s[:, :, :-1] += p[:, :, 1:]
        s[1:] += p[:-1]
        s[:-1] += p[1:]
        return s

    def sor(self, p, b, omega, iters):
        for _ in range(iters):
            for c in (self.red, ~self.red):
                gs = (self.near(p) - self.h2 * b) / self.d
                p = torch.where(c, p + omega * (gs - p), p)
        return p

    def rho(self, p, b):
        return float((b - (self.near(p) - self.d * p) / self.h2).norm() / b.norm())

    def solve(self, p, b, omega, tol, every, most=100000):
        it = 0
        while self.rho(p, b) > tol and it < most:
            p = self.sor(p, b, omega, every)
            it += every
        return p


def _les_exact(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dx, dt, nu, alpha, beta, l2 = 4.0, 0.025, 1.5e-5, -100.0, -10.0, (0.1 * 4.0) ** 2
    sol = torch.as_tensor(_buildings(case, seed), device=DEV) != 0
    nil = torch.zeros_like(sol[:, :, :1])
    fu = sol | torch.cat([sol[:, :, 1:], nil], 2)
    fv = sol | torch.roll(sol, -1, 1)
    fw = torch.zeros_like(sol)
    fw[:-1] = sol[:-1] | sol[1:]
    zc = (torch.arange(1, nz + 1, device=DEV, dtype=torch.float64) - 0.5) * dx
    uin = 5.0 * torch.log(zc / 0.1) / math.log(10.0 / 0.1)
    shape = (nz + 2, ny + 2, nx + 2)
    u, v, w, p, gu, gv, gw = (torch.zeros(shape, dtype=torch.float64, device=DEV) for _ in range(7))
    I = (slice(1, -1),) * 3
    u[I] = torch.where(fu, torch.zeros((), dtype=torch.float64, device=DEV), uin[:, None, None].expand(nz, ny, nx))
    u[1:-1, 1:-1, 0] = torch.where(sol[:, :, 0], 0.0, uin[:, None])
    solver = _Poisson(nx, ny, nz, dx)
    old = None
    r = 1.0 / dx

    def at(a, x=0, y=0, z=0):  # interior-sized view shifted by (x, y, z)
        return a[1 + z:nz + 1 + z, 1 + y:ny + 1 + y, 1 + x:nx + 1 + x]

    def mid(a, *s):  # the mean of a at the cell and at the cell shifted by s
        return 0.5 * (at(a, *s[0]) + at(a, *s[1]))

    def periodic(a):
        a[:, 0], a[:, -1] = a[:, -2].clone(), a[:, 1].clone()

    for step in range(case["steps"]):
        pi = p[I]
        pe = torch.cat([pi[:, :, 1:], -pi[:, :, -1:]], 2)
        u[I] -= dt * r * (pe - pi)
        v[I] -= dt * r * (torch.roll(pi, -1, 1) - pi)
        w[1:-2, 1:-1, 1:-1] -= dt * r * (pi[1:] - pi[:-1])
        for a, first in ((u, uin[:, None]), (v, None), (w, None)):
            a[1:-1, 1:-1, 0] = first if first is not None else -a[1:-1, 1:-1, 1]
            a[1:-1, 1:-1, -1] = a[1:-1, 1:-1, -2]
            periodic(a)
        for a in (u, v):
            a[0], a[-1] = -a[1], a[-2].clone()
        w[0] = 0.0
        w[-2:] = 0.0
        C, E, N, T = (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)
        Wn, S, B = (-1, 0, 0), (0, -1, 0), (0, 0, -1)
        Fu = -r * (mid(u, C, E) ** 2 - mid(u, Wn, C) ** 2 + mid(u, C, N) * mid(v, C, E)
                   - mid(u, S, C) * mid(v, S, (1, -1, 0)) + mid(u, C, T) * mid(w, C, E)
                   - mid(u, B, C) * mid(w, B, (1, 0, -1)))
        Fv = -r * (mid(v, C, E) * mid(u, C, N) - mid(v, Wn, C) * mid(u, Wn, (-1, 1, 0)) + mid(v, C, N) ** 2
                   - mid(v, S, C) ** 2 + mid(v, C, T) * mid(w, C, N) - mid(v, B, C) * mid(w, B, (0, 1, -1)))
        Fw = -r * (mid(w, C, E) * mid(u, C, T) - mid(w, Wn, C) * mid(u, Wn, (-1, 0, 1)) + mid(w, C, N) * mid(v, C, T)
                   - mid(w, S, C) * mid(v, S, (0, -1, 1)) + mid(w, C, T) ** 2 - mid(w, B, C) ** 2)
        for F, G, a, f in ((Fu, gu, u, fu), (Fv, gv, v, fv), (Fw, gw, w, fw)):
            G[I] += torch.where(f, dt * a[I], 0.0)
            F += torch.where(f, alpha * G[I] + beta * a[I], 0.0)
        # strain on its natural points, on the interior and one cell below and left of it
        def lo(a, x, y, z, sx, sy, sz):
            return a[1 - sz + z:nz + 1 + z, 1 - sy + y:ny + 1 + y, 1 - sx + x:nx + 1 + x]

        def edge(a, b, ax, bx, s):  # 0.5 (d a + d b) / dx at the edges
            return 0.5 * r * ((lo(a, *ax, *s) - lo(a, 0, 0, 0, *s)) + (lo(b, *bx, *s) - lo(b, 0, 0, 0, *s)))

        e12 = edge(u, v, N, E, (1, 1, 0))
        e13 = edge(u, w, T, E, (1, 0, 1))
        e23 = edge(v, w, T, N, (0, 1, 1))
        a12 = e12[:, 1:, 1:] ** 2 + e12[:, :-1, 1:] ** 2 + e12[:, 1:, :-1] ** 2 + e12[:, :-1, :-1] ** 2
        a13 = e13[1:, :, 1:] ** 2 + e13[:-1, :, 1:] ** 2 + e13[1:, :, :-1] ** 2 + e13[:-1, :, :-1] ** 2
        a23 = e23[1:, 1:] ** 2 + e23[:-1, 1:] ** 2 + e23[1:, :-1] ** 2 + e23[:-1, :-1] ** 2
        s11, s22, s33 = (r * (at(a) - at(a, *s)) for a, s in ((u, Wn), (v, S), (w, B)))
        ne = torch.zeros(shape, dtype=torch.float64, device=DEV)
        ne[I] = l2 * torch.sqrt(2.0 * (s11 ** 2 + s22 ** 2 + s33 ** 2) + a12 + a13 + a23)
        ne[:, :, 0], ne[:, :, -1] = ne[:, :, 1].clone(), ne[:, :, -2].clone()
        periodic(ne)
        ne[0], ne[-1] = ne[1].clone(), ne[-2].clone()
        ne += nu

        def edge_nu(e, s, n1, n2, n12):
            return 0.5 * e * (lo(ne, 0, 0, 0, *s) + lo(ne, *n1, *s) + lo(ne, *n2, *s) + lo(ne, *n12, *s))

        t12 = edge_nu(e12, (1, 1, 0), E, N, (1, 1, 0))
        t13 = edge_nu(e13, (1, 0, 1), E, T, (1, 0, 1))
        t23 = edge_nu(e23, (0, 1, 1), N, T, (0, 1, 1))
        pad = torch.nn.functional.pad
        t11 = 2.0 * r * ne[1:-1, 1:-1, 1:] * (u[1:-1, 1:-1, 1:] - u[1:-1, 1:-1, :-1])
        t22 = 2.0 * r * ne[1:-1, 1:, 1:-1] * (v[1:-1, 1:, 1:-1] - v[1:-1, :-1, 1:-1])
        t33 = 2.0 * r * ne[1:, 1:-1, 1:-1] * (w[1:, 1:-1, 1:-1] - w[:-1, 1:-1, 1:-1])
        Fu += r * ((t11[:, :, 1:] - t11[:, :, :-1]) + (t12[:, 1:, 1:] - t12[:, :-1, 1:]) + (t13[1:, :, 1:] - t13[:-1, :, 1:]))
        Fv += r * ((t12[:, 1:, 1:] - t12[:, 1:, :-1]) + (t22[:, 1:] - t22[:, :-1]) + (t23[1:, 1:] - t23[:-1, 1:]))
        Fw += r * ((t13[1:, :, 1:] - t13[1:, :, :-1]) + (t23[1:, 1:] - t23[1:, :-1]) + (t33[1:] - t33[:-1]))
        Fw[-1] = 0.0
        F = (Fu, Fv, Fw)
        for q, a in enumerate((u, v, w)):
            inc = dt * (F[q] if old is None else 1.5 * F[q] - 0.5 * old[q])
            if q == 2:
                inc[-1] = 0.0
            a[I] += inc
        old = F
        vs = torch.roll(v[I], 1, 1)
        b = ((at(u) - at(u, *Wn)) + (at(v) - vs) + (at(w) - at(w, *B))) / (dx * dt)
        if case["mode"] == "fixed":
            p[I] = solver.sor(p[I], b, 1.8, case["iters"])
        else:
            p[I] = solver.solve(p[I].clone(), b, 1.8, 1e-6, 10)
    # between steps the library keeps no ghost layer but the inflow face
    for a in (u, v, w, p):
        keep = a.clone()
        a.zero_()
        a[I] = keep[I]
    u[1:-1, 1:-1, 0] = uin[:, None]
    out = dict(u=u, v=v, w=w, p=p)
    if case["mode"] == "fixed":
        return out
    for n, a in zip(("fu_old", "fv_old", "fw_old"), old):
        out[n] = pad(a, (1, 1) * 3)
    return dict(out, gu=gu, gv=gv, gw=gw, step=None, iters=None)


def _net(flat, x):
    o = 0
    P = []
    for ci, co in LAYERS:
        n = 27 * ci * co
        P.append((flat[o:o + n].view(3, 3, 3, co, ci).permute(3, 4, 0, 1, 2), flat[o + n:o + n + co]))
        o += n + co
    F = torch.nn.functional
    c = lambda l, a: F.relu(F.conv3d(a, P[l][0], P[l][1], padding=1))  # noqa: E731
    up = lambda a: F.interpolate(a, scale_factor=2, mode="nearest")  # noqa: E731
    a = x.permute(0, 4, 1, 2, 3)
    s1 = c(1, c(0, a))
    s2 = c(3, c(2, F.avg_pool3d(s1, 2)))
    b3 = c(5, c(4, F.avg_pool3d(s2, 2)))
    d2 = c(6, torch.cat([up(b3), s2], 1))
    d1 = c(7, torch.cat([up(d2), s1], 1))
    return torch.einsum("ncdhw,c->ndhw", d1, flat[o:o + 16]) + flat[o + 16]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("sw", "sw64"):
        p, H, eta = _basin(case["basin"], case["nx"], case["ny"], np.random.default_rng(seed))
        out, vol = _sw_outputs(p, *_sw_exact(p, H, eta, case["steps"]))
        return dict(out, wet=None) if kind == "sw64" else dict(out, volume=vol)
    if kind == "ensemble":
        states, vols = [], []
        for m in _ensemble(case, seed):
            out, vol = _sw_outputs(m.params(), *_sw_exact(m.params(), m.H, m.eta0, case["steps"]))
            states.append(out)
            vols.append(vol)
        return dict(volumes=tuple(np.array(c) for c in zip(*vols)), states=states)
    if kind == "les":
        return None if case["mode"] == "learned" else _les_exact(case, seed)
    if kind == "poisson":
        b = _rhs(case, seed).double()
        solver = _Poisson(case["nx"], case["ny"], case["nz"], 4.0)
        return dict(p=solver.solve(torch.zeros_like(b), b, 1.8, 1e-6, 10), status=None, iters=None)
    x, t = _pairs(case, seed)
    flat = torch.as_tensor(_weights(seed), device=DEV).double()
    with torch.backends.cudnn.flags(enabled=False):
        if kind == "infer":
            return _net(flat, x.double())
        flat.requires_grad_(True)
        loss = ((_net(flat, x.double()) - t.double()) ** 2).mean()
        g, = torch.autograd.grad(loss, flat)
    # one Adam step from zero moments
    m, v = 0.1 * g / (1 - 0.9), 0.001 * g * g / (1 - 0.999)
    return dict(loss=float(loss), params=(flat - 1e-3 * m / (v.sqrt() + 1e-8)).detach())
