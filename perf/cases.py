"""The work that a user of this library has it do, as measurable cases.

Every case is one use of the public entry points (``Solver``, ``Batch``, ``Pairwise``,
``Multigrid``, ``WarmStartNet`` and the ``gabp_*`` functions) on synthetic problems of the kinds
the library is built for: a Matern field on a 2-D grid, observed along satellite-like tracks or
at scattered points with independent noise.  ``listed()`` names the fixed cases, ``draw()`` gives
others of the same ranges, ``prepare()`` makes what a program holds before the call, ``run()`` is
one pass, ``work()`` what a pass cannot do without and ``exact()`` the same result in plain
FP64 torch, without the library.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch
import torch.nn.functional as F

from paper_2404_12968_gb300 import (Batch, Multigrid, Pairwise, Solver, WarmStartNet, gabp_batch_marginals,
                                    gabp_pw_marginals, gabp_wsnet_gradients)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WEIGHTS = os.path.join(ROOT, "paper_2404_12968_gb300", "weights", "wsnet_512.npy")
F64 = torch.float64

# kind     what one pass is
# window   a new analysis window from host arrays: create, iterate, residual, marginals, destroy
# steps    a context that is kept: cold (or learned) start, iterate, residual, marginals
# batch    a kept batch of uneven problems, iterated on; its residuals and every member's marginals
# pairwise the paper's pairwise re-weighted messages on a kept context
# mg       multigrid warm start and the early-stopping rule, as the grid-size sweep runs them
# train    loss and gradients of the warm-start network on a batch of samples


def _case(kind, name=None, **kw):
    c = {"kind": kind, "nx": 64, "ny": 64, "kappa": 0.1, "alpha": 2, "tracks": 0, "per_track": 0, "points": 0,
         "sigma_lo": 0.05, "sigma_hi": 0.05, "prec": "fp32", "iters": 100, "damping": 0.3, "var": False,
         "start": "cold"}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem of the configurations, solved from scratch in FP64: all latency
        _case("window", "window-64-fp64", kappa=0.3, points=500, sigma_lo=0.1, sigma_hi=0.1, prec="fp64", iters=200,
              damping=0.5, var=True),
        # a global 1-degree analysis (361 x 181, an odd width) to the default tolerance (iters 0)
        _case("window", "window-361x181", nx=361, ny=181, tracks=8, per_track=400, points=500, iters=0, var=True),
        # a global temperature field of 2500 x 1500 nodes, about 8 % of them observed along tracks
        _case("window", "window-2500x1500", nx=2500, ny=1500, kappa=0.05, tracks=48, per_track=6250, iters=100),
        # the learned warm start's evaluation problem, to the default tolerance
        _case("steps", "learned-2048", nx=2048, ny=2048, kappa=0.03, tracks=48, per_track=3413, iters=0,
              start="learned"),
        # a regional grid whose width is not a multiple of four, a fixed number of iterations
        _case("steps", "steps-1601x1201", nx=1601, ny=1201, kappa=0.05, tracks=32, per_track=2000, points=20000,
              iters=200, var=True),
        # the benchmark's workload and step: 100 iterations, residual, means in device memory
        _case("steps", "steps-4096", nx=4096, ny=4096, kappa=0.02, tracks=96, per_track=12500, points=200000,
              sigma_lo=0.02, sigma_hi=0.1, iters=100),
        # FP64 messages (ill-conditioned small kappa) on a mid-size grid
        _case("steps", "steps-512-fp64", nx=512, ny=512, kappa=0.02, tracks=12, per_track=853, prec="fp64", iters=100,
              var=True),
        # the alpha = 4 prior (13-slot cell factors)
        _case("steps", "alpha4-2048", nx=2048, ny=2048, kappa=0.05, alpha=4, tracks=48, per_track=3413, points=50000,
              iters=50, damping=0.5),
        # an ensemble of uneven members, sides log-uniform in [128, 1024]
        _case("batch", "batch-16", count=16, lo=128, hi=1024, iters=100, var=True),
        # the paper's own message passing on its synthetic setting (5 % of the grid points observed)
        _case("pairwise", "pairwise-512", nx=512, ny=512, frac=0.05, iters=200, c=10.0, rate=0.6, var=True),
        # one entry of the grid-size x density sweep: multigrid from a 32 x 32 base, early stop
        _case("mg", "multigrid-512", nx=512, ny=512, frac=0.05, levels=5),
        # one training step's gradients at the shape the shipped network was trained with
        _case("train", "train-8x512", nx=512, ny=512, count=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["window", "window", "steps", "steps", "steps", "steps", "batch", "pairwise", "mg", "train"])
    kappa = round(rng.uniform(0.02, 0.3), 4)
    if kind in ("window", "steps"):
        prec = "fp64" if rng.random() < 0.3 else "fp32"
        alpha = 4 if kind == "steps" and rng.random() < 0.2 else 2
        top = 700 if prec == "fp64" else 1500 if alpha == 4 else 3000
        nx, ny = _log(rng, 48, top), _log(rng, 48, top)
        start = "learned" if kind == "steps" and prec == "fp32" and alpha == 2 and rng.random() < 0.2 else "cold"
        iters = rng.randint(20, 60) if alpha == 4 else rng.randint(30, 200)
        if start == "learned" or (alpha == 2 and nx * ny < 1 << 18 and rng.random() < 0.25):
            iters, kappa = 0, max(kappa, 0.08)
        m = rng.choice([0.01, 0.03, 0.08]) * nx * ny
        tracks = rng.randint(2, 32)
        return _case(kind, nx=nx, ny=ny, kappa=kappa, alpha=alpha, tracks=tracks, per_track=int(m / tracks) + 1,
                     points=rng.choice([0, nx * ny // 100]), sigma_lo=0.02, sigma_hi=rng.choice([0.02, 0.1]),
                     prec=prec, iters=iters, damping=0.5 if alpha == 4 else rng.choice([0.3, 0.5]),
                     var=rng.random() < 0.5, start=start)
    if kind == "batch":
        lo = _log(rng, 64, 256)
        return _case("batch", count=rng.randint(2, 24), lo=lo, hi=rng.randint(lo + 32, 900), iters=rng.randint(30, 100),
                     var=rng.random() < 0.5)
    if kind == "pairwise":
        return _case("pairwise", nx=_log(rng, 64, 1200), ny=_log(rng, 64, 1200), frac=rng.choice([0.01, 0.05, 0.1]),
                     iters=rng.randint(50, 200), c=rng.choice([10.0, 20.0]), rate=0.6,
                     prec="fp64" if rng.random() < 0.25 else "fp32", var=rng.random() < 0.5)
    if kind == "mg":
        levels = rng.randint(3, 5)
        side = 32 * 2 ** (levels - 1) + rng.choice([0, 0, rng.randint(-9, 9)])
        return _case("mg", nx=side, ny=side, frac=rng.choice([0.05, 0.1]), levels=levels)
    return _case("train", nx=8 * rng.randint(16, 64), ny=8 * rng.randint(16, 64), count=rng.randint(1, 8))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------

def _field_at(x, y, kappa, alpha, gen, feats=192):
    """A draw from the Matern prior at scattered points, by random Fourier features: wave numbers
    from its spectral density ~ (kappa^2 + |w|^2)^-alpha, marginal variance of the continuum."""
    dev = x.device
    u = torch.rand(feats, generator=gen, dtype=F64, device=dev).clamp_(1e-6, 1 - 1e-6)
    r = kappa * torch.sqrt((1.0 - u) ** (-1.0 / (alpha - 1)) - 1.0)
    r = r.clamp(max=math.pi)
    th = 2.0 * math.pi * torch.rand(feats, generator=gen, dtype=F64, device=dev)
    ph = 2.0 * math.pi * torch.rand(feats, generator=gen, dtype=F64, device=dev)
    var = 1.0 / (4.0 * math.pi * kappa ** 2) if alpha == 2 else 1.0 / (12.0 * math.pi * kappa ** 6)
    f = torch.zeros_like(x)
    for wx, wy, p in zip((r * torch.cos(th)).tolist(), (r * torch.sin(th)).tolist(), ph.tolist()):
        f += torch.cos(wx * x + wy * y + p)
    return f * math.sqrt(2.0 * var / feats)


def _problem(nx, ny, kappa, alpha, tracks, per_track, points, lo, hi, gen):
    """Observations along wrapped straight tracks (one sample per 1.5 cells) and at scattered
    points: (xy (m, 2), y, noise variances) as host float64 arrays."""
    dev = gen.device
    rnd = lambda n: torch.rand(n, generator=gen, dtype=F64, device=dev)  # noqa: E731
    wx, wy = nx - 1.0, ny - 1.0
    th, x0, y0 = math.pi * rnd(tracks), wx * rnd(tracks), wy * rnd(tracks)
    t = 1.5 * torch.arange(per_track, dtype=F64, device=dev)
    tx = torch.remainder(x0[:, None] + t * torch.cos(th)[:, None], wx).reshape(-1)
    ty = torch.remainder(y0[:, None] + t * torch.sin(th)[:, None], wy).reshape(-1)
    x = torch.cat([tx, wx * rnd(points)]).clamp(0.0, wx)
    y = torch.cat([ty, wy * rnd(points)]).clamp(0.0, wy)
    s = lo + (hi - lo) * rnd(x.numel())
    v = _field_at(x, y, kappa, alpha, gen) + s * torch.randn(x.numel(), generator=gen, dtype=F64, device=dev)
    return torch.stack([x, y], 1).cpu().numpy(), v.cpu().numpy(), (s * s).cpu().numpy()


def _lattice_problem(nx, ny, frac, gen):
    """The paper's synthetic setting: a fraction of the grid points observed (noise 0.01), Matern
    prior of lengthscale 0.15 and standard deviation 1.1 on the unit square; returns
    (kappa, gamma, xy, y, noise variances) at unit spacing."""
    dev = gen.device
    side = max(nx, ny)
    h, kappa = 1.0 / side, math.sqrt(2.0) / 0.15
    gamma = h * h / (1.1 ** 2 * 4.0 * math.pi * kappa * kappa) / h ** 4
    m = int(round(frac * nx * ny))
    idx = torch.randperm(nx * ny, generator=gen, device=dev)[:m].sort().values
    x, y = (idx % nx).to(F64), (idx // nx).to(F64)
    f = _field_at(x, y, kappa * h, 2, gen) / math.sqrt(gamma)
    v = f + 0.01 * torch.randn(m, generator=gen, dtype=F64, device=dev)
    return kappa * h, gamma, torch.stack([x, y], 1).cpu().numpy(), v.cpu().numpy(), np.full(m, 1e-4)


def _members(case, gen):
    """The members of a batch: uneven sides (an even spread over the logarithm of the range, shuffled),
    kappa and numbers of tracks."""
    out = []
    for i, (k, t) in enumerate(torch.rand((case["count"], 2), generator=gen, dtype=F64, device=gen.device).tolist()):
        u = (0.5 + 0.6180339887498949 * i) % 1.0
        side = int(round(case["lo"] * (case["hi"] / case["lo"]) ** u))
        kappa, tracks = 0.02 + 0.18 * k, 4 + int(28.999 * t)
        xy, y, nv = _problem(side, side, kappa, 2, tracks, int(2.5 * side / 1.5), 0, 0.05, 0.05, gen)
        out.append((side, kappa, xy, y, nv))
    return out


class _Member:
    """One batch member, in the form ``Batch`` takes."""

    def __init__(self, side, kappa, xy, y, nv):
        self.nx = self.ny = side
        self.kappa, self.obs_x, self.obs_y, self.y, self.noise_var = kappa, xy[:, 0], xy[:, 1], y, nv


def _gen(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + case["nx"] * 7919 + case["ny"] * 31 + case.get("count", 0)) % (1 << 62))
    return g


def _inputs(case, seed):
    gen = _gen(case, seed)
    if case["kind"] in ("pairwise", "mg"):
        return _lattice_problem(case["nx"], case["ny"], case["frac"], gen)
    if case["kind"] == "batch":
        return _members(case, gen)
    if case["kind"] == "train":
        return _samples(case, gen)
    return (case["kappa"], 1.0) + _problem(case["nx"], case["ny"], case["kappa"], case["alpha"], case["tracks"],
                                           case["per_track"], case["points"], case["sigma_lo"], case["sigma_hi"], gen)


def _samples(case, gen):
    """Training samples: gridded observations (value, mask, log kappa + 3, zeros) in BF16 and
    smooth targets (mean / scale, log precision)."""
    B, H, W = case["count"], case["ny"], case["nx"]
    dev = gen.device
    rnd = lambda *s: torch.rand(s, generator=gen, device=dev)  # noqa: E731
    coarse = torch.randn((B, 1, H // 8, W // 8), generator=gen, device=dev)
    field = F.interpolate(coarse, size=(H, W), mode="bicubic", align_corners=False)[:, 0]
    mask = (rnd(B, H, W) < 0.06).float()
    kf = (torch.log(0.02 + 0.18 * rnd(B)) + 3.0)[:, None, None].expand(B, H, W)
    x = torch.zeros((B, H, W, 16), device=dev)
    x[..., 0] = mask * (field + 0.05 * torch.randn((B, H, W), generator=gen, device=dev))
    x[..., 1] = mask
    x[..., 2] = kf
    t = torch.stack([field, 0.5 * kf + 2.0 * F.avg_pool2d(mask[:, None], 9, 1, 4)[:, 0]], -1).contiguous()
    return x.bfloat16().contiguous(), t


def _pinned(a):
    t = torch.empty(a.shape, dtype=F64, pin_memory=True).numpy()
    t[...] = a
    return t


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------

def _solver(case, kappa, gamma, xy, y, nv):
    return Solver(nx=case["nx"], ny=case["ny"], kappa=kappa, obs_xy=xy, y=y, noise_var=nv, precision=case["prec"],
                  gamma=gamma, alpha=case["alpha"])


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    n = case["nx"] * case["ny"]
    dev = torch.device("cuda")
    if kind == "train":
        st["x"], st["t"] = _inputs(case, seed)
        st["net"] = WarmStartNet(seed=3)
        st["net"].load(WEIGHTS)
        st["grads"] = torch.empty(st["net"].nparam, dtype=torch.float32, device=dev)
        return st
    if kind == "batch":
        mem = [_Member(*q) for q in _inputs(case, seed)]
        st["batch"] = Batch(mem)
        st["out"] = [(torch.empty(q.nx * q.ny, dtype=F64, device=dev),
                      torch.empty(q.nx * q.ny, dtype=F64, device=dev) if case["var"] else None) for q in mem]
        return st
    kappa, gamma, xy, y, nv = _inputs(case, seed)
    if kind == "window":   # host arrays, pinned as a program streaming windows holds them
        st.update(kappa=kappa, xy=_pinned(xy), y=_pinned(y), nv=_pinned(nv), mean=_pinned(np.zeros(n)),
                  vr=_pinned(np.zeros(n)) if case["var"] else None)
        return st
    solver = _solver(case, kappa, gamma, xy, y, nv)
    if kind == "pairwise":   # listed before the solver: it is released first, as the library asks
        st["pw"] = Pairwise(solver)
    st["solver"] = solver
    st["mean"] = torch.empty(n, dtype=F64, device=dev)
    st["vr"] = torch.empty(n, dtype=F64, device=dev) if case["var"] else None
    if case["start"] == "learned":
        st["net"] = WarmStartNet(seed=0)
        st["net"].load(WEIGHTS)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "train":
        xs, ts = list(st["x"].unbind(0)), list(st["t"].unbind(0))
        loss = gabp_wsnet_gradients(st["net"].handle, xs, ts, case["ny"], case["nx"], st["grads"])
        return {"loss": loss, "grads": st["grads"]}
    if kind == "batch":
        b = st["batch"]
        b.iterate(case["iters"], case["damping"])
        res = b.residuals()
        for i, (m, v) in enumerate(st["out"]):
            gabp_batch_marginals(b.handle, i, m, v)
        return {"residual": res, "mean": [m for m, _ in st["out"]], "var": [v for _, v in st["out"] if v is not None]}
    if kind == "window":
        s = _solver(case, st["kappa"], 1.0, st["xy"], st["y"], st["nv"])
        try:
            s.iterate(case["iters"] or -1, case["damping"])
            out = {"residual": s.residual(), "iterations": s.stats()["iterations"]}
            s.marginals(st["mean"], st["vr"], want_var=case["var"])
        finally:
            s.close()
        out["mean"], out["var"] = st["mean"], st["vr"]
        return out
    s = st["solver"]
    if kind == "pairwise":
        pw = st["pw"]
        pw.reset()
        pw.iterate(case["iters"], case["c"], case["rate"])
        r = pw.residual()
        gabp_pw_marginals(pw.handle, st["mean"], st["vr"])
        return {"residual": r, "mean": st["mean"], "var": st["vr"]}
    if kind == "mg":
        with Multigrid(s, case["levels"]) as mg:
            levels = mg.warm_start(case["damping"], 1e-4, 200000)["iterations"]
        t = s.iterate_early_stop(10000, case["damping"], 1e-3)
        s.marginals(st["mean"], want_var=False)
        return {"levels": levels, "iterations": t, "mean": st["mean"]}
    if case["start"] == "learned":
        s.learned_warm_start(st["net"])
    else:
        s.reset()
    s.iterate(case["iters"] or -1, case["damping"])
    out = {"residual": s.residual(), "iterations": s.stats()["iterations"]}
    s.marginals(st["mean"], st["vr"], want_var=case["var"])
    out["mean"], out["var"] = st["mean"], st["vr"]
    return out


def _m(case):
    if case["kind"] in ("pairwise", "mg"):
        return int(round(case["frac"] * case["nx"] * case["ny"]))
    return case["tracks"] * case["per_track"] + case["points"]


def work(case):
    """Bytes: per iteration every message once in and once out and the static data of every
    observation (20 B in FP32), then the outputs.  Solves to a tolerance: their usual number of
    iterations.  Flops: about 200 per node and 120 per observation and iteration (5-slot cells)."""
    kind, n, T = case["kind"], case["nx"] * case["ny"], 8 if case["prec"] == "fp64" else 4
    outs = 8.0 * n * (2 if case["var"] else 1)
    if kind == "train":
        px = case["count"] * n
        macs = 16 * 32 * 9 + 32 * 32 * 9 + (32 * 64 + 64 * 64) * 9 / 4 + (64 * 128 + 128 * 128) * 9 / 16 + \
            (128 * 256 + 256 * 256) * 9 / 64 + 256 * 128 / 64 + 128 * 128 * 9 / 16 + 128 * 64 / 16 + 64 * 64 * 9 / 4 + \
            64 * 32 / 4 + 32 * 32 * 9 + 64
        # activations of the forward pass written once and read once by the backward pass
        acts = 16 + 32 * 4 + 64 * 4 / 4 + 128 * 4 / 16 + 256 * 2 / 64 + 32 / 4 + 64 / 16 + 128 / 64
        return {"bytes": px * (2 * acts * 2 + 16.0) + 8.0 * 1.2e6, "flops": 3.0 * 2.0 * macs * px}
    if kind == "batch":
        side2 = (case["hi"] ** 2 - case["lo"] ** 2) / (2.0 * math.log(case["hi"] / case["lo"]))   # mean of side^2
        n = case["count"] * side2
        m = case["count"] * 18 * 2.5 / 1.5 * math.sqrt(side2)
        return {"bytes": case["iters"] * (16.0 * (5 * n + 4 * m) + 20.0 * m) + 8.0 * n * (2 if case["var"] else 1),
                "flops": case["iters"] * (200.0 * n + 120.0 * m)}
    m = _m(case)
    if kind == "pairwise":   # 12 messages read and written, 14 coefficients
        return {"bytes": case["iters"] * n * (12 * 4.0 * T + 14 * T) + outs, "flops": case["iters"] * n * 250.0}
    if kind == "mg":
        its = 25 + 40 / 3
        return {"bytes": its * (16.0 * (5 * n + 4 * m) + 20.0 * m) + 8.0 * n, "flops": its * (200.0 * n + 120.0 * m)}
    its = case["iters"] or (80 if case["start"] == "learned" else 250)
    slots = 13 if case["alpha"] == 4 else 5
    extra = 0.0
    if case["start"] == "learned":
        extra = 2.0 * 83e3 * n
    return {"bytes": its * (4.0 * T * (slots * n + 4 * m) + 5.0 * T * m) + outs,
            "flops": its * (40.0 * slots * n + 120.0 * m) + extra}


# ---------------------------------------------------------------------------------------
# the same results in plain FP64 torch
# ---------------------------------------------------------------------------------------

def _stencil(nx, ny, kappa, alpha, dev):
    """Offsets (dy, dx) and coefficient fields [slot][ny][nx] (0 where the node is missing) of the
    rows of L (alpha = 2) or L^2 (alpha = 4), zero-Neumann."""
    one = torch.ones((ny, nx), dtype=F64, device=dev)
    inside = lambda dy, dx: _at(one, dy, dx)  # noqa: E731  1 where node (i + dy, j + dx) exists
    four = [(0, -1), (0, 1), (-1, 0), (1, 0)]
    deg = sum(inside(*o) for o in four)
    ac = kappa * kappa + deg
    if alpha == 2:
        return [(0, 0)] + four, torch.stack([ac] + [-inside(*o) for o in four])
    offs = [(0, 0)] + four + [(-1, -1), (-1, 1), (1, -1), (1, 1)] + [(0, -2), (0, 2), (-2, 0), (2, 0)]
    a = [ac * ac + deg] + [-(ac + _at(ac, *o)) * inside(*o) for o in four] + [2.0 * inside(*o) for o in offs[5:9]] + \
        [inside(*o) for o in offs[9:]]
    return offs, torch.stack(a)


def _at(f, dy, dx):
    """g[i, j] = f[i + dy, j + dx], zero outside the grid."""
    ny, nx = f.shape
    g = torch.zeros_like(f)
    i0, i1, j0, j1 = max(0, -dy), min(ny, ny - dy), max(0, -dx), min(nx, nx - dx)
    if i0 < i1 and j0 < j1:
        g[i0:i1, j0:j1] = f[i0 + dy:i1 + dy, j0 + dx:j1 + dx]
    return g


class _Gabp:
    """Synchronous damped GaBP in FP64 on the rank-1 factors; leave-one-out sums throughout."""

    def __init__(self, nx, ny, kappa, gamma, xy, y, nv, alpha=2):
        dev = torch.device("cuda")
        self.nx, self.ny, self.n, self.gamma, self.m = nx, ny, nx * ny, gamma, len(y)
        self.offs, self.a = _stencil(nx, ny, kappa, alpha, dev)
        xy, self.y, self.v = (torch.as_tensor(q, device=dev) for q in (xy.reshape(-1, 2), y, nv))
        j0 = xy[:, 0].floor().clamp(0, max(nx - 2, 0))
        i0 = xy[:, 1].floor().clamp(0, max(ny - 2, 0))
        fu, fv = xy[:, 0] - j0, xy[:, 1] - i0
        self.w = torch.stack([(1 - fu) * (1 - fv), fu * (1 - fv), (1 - fu) * fv, fu * fv])
        b = (i0 * nx + j0).long()
        self.node = torch.stack([b, b + 1, b + nx, b + nx + 1])
        self.reset()

    def reset(self):
        self.L, self.E = self.gamma * self.a * self.a, torch.zeros_like(self.a)
        self.oL, self.oE = self.w * self.w / self.v, torch.zeros_like(self.w)

    def warm(self, mu, lam):
        ones = torch.ones(4 * self.m, dtype=F64, device=mu.device)
        deg = torch.zeros(self.n, dtype=F64, device=mu.device).index_add_(0, self.node.reshape(-1), ones)
        for u, (dy, dx) in enumerate(self.offs):
            deg += _at((self.a[u] != 0).to(F64), -dy, -dx).reshape(-1)
        lam = lam / deg
        lg, eg = lam.reshape(self.ny, self.nx), (mu * lam).reshape(self.ny, self.nx)
        for u, o in enumerate(self.offs):
            self.L[u], self.E[u] = _at(lg, *o), _at(eg, *o)
        self.oL, self.oE = lam[self.node], (mu * lam)[self.node]

    def _terms(self, P, O):
        """Per node: the incoming prior messages by slot and the sum of the observation messages."""
        inc = [_at(P[u], -dy, -dx) for u, (dy, dx) in enumerate(self.offs)]
        obs = torch.zeros(self.n, dtype=F64, device=P.device).index_add_(0, self.node.reshape(-1), O.reshape(-1))
        return inc, obs.reshape(self.ny, self.nx)

    @staticmethod
    def _loo(t, last):
        """Leave-one-out sums of the list t, the term `last` always included; and the total."""
        pre = [None]
        for q in t:
            pre.append(q if pre[-1] is None else pre[-1] + q)
        out, suf = [None] * len(t), last
        for u in range(len(t) - 1, -1, -1):
            out[u] = suf if pre[u] is None else pre[u] + suf
            suf = suf + t[u]
        return out, pre[-1]

    @staticmethod
    def _factor(a, var, r, lam, eta):
        """Messages of rank-1 factors over K slots (dimension 0)."""
        a2 = a * a
        lam = torch.where(lam > 1e-20 * a2, lam, 1e-20 * a2)
        ok = a2 > 0
        rl = torch.where(ok, 1.0 / lam, torch.zeros_like(lam))
        t, p = a2 * rl, a * eta * rl
        K = a.shape[0]
        preV, preM = [var], [torch.zeros_like(t[0])]
        for u in range(K - 1):
            preV.append(preV[-1] + t[u])
            preM.append(preM[-1] + p[u])
        L, E = torch.empty_like(a), torch.empty_like(a)
        sV = sM = 0.0
        for u in range(K - 1, -1, -1):
            V = preV[u] + sV
            L[u], E[u] = a2[u] / V, a[u] * (r - preM[u] - sM) / V
            sV, sM = sV + t[u], sM + p[u]
        return L, E

    def beliefs(self):
        iL, oL = self._terms(self.L, self.oL)
        iE, oE = self._terms(self.E, self.oE)
        return (sum(iE) + oE).reshape(-1), (sum(iL) + oL).reshape(-1)

    def step(self, beta):
        iL, tL = self._terms(self.L, self.oL)
        iE, tE = self._terms(self.E, self.oE)
        lL, sL = self._loo(iL, tL)
        lE, sE = self._loo(iE, tE)
        cl = torch.stack([_at(lL[u], *o) for u, o in enumerate(self.offs)])
        ce = torch.stack([_at(lE[u], *o) for u, o in enumerate(self.offs)])
        L, E = self._factor(self.a, torch.full_like(sL, 1.0 / self.gamma), 0.0, cl, ce)
        if self.m:
            cl = sL.reshape(-1)[self.node] + (tL.reshape(-1)[self.node] - self.oL)
            ce = sE.reshape(-1)[self.node] + (tE.reshape(-1)[self.node] - self.oE)
            l, e = self._factor(self.w, self.v, self.y, cl, ce)
            self.oL, self.oE = beta * self.oL + (1 - beta) * l, beta * self.oE + (1 - beta) * e
        self.L, self.E = beta * self.L + (1 - beta) * L, beta * self.E + (1 - beta) * E

    def apply(self, x):
        """A x and b of the posterior."""
        x = x.reshape(self.ny, self.nx)
        z = sum(self.a[u] * _at(x, *o) for u, o in enumerate(self.offs))
        r = self.gamma * sum(_at(self.a[u] * z, -o[0], -o[1]) for u, o in enumerate(self.offs)).reshape(-1)
        b = torch.zeros_like(r)
        if self.m:
            hx = (self.w * x.reshape(-1)[self.node]).sum(0)
            r.index_add_(0, self.node.reshape(-1), (self.w * (hx / self.v)).reshape(-1))
            b.index_add_(0, self.node.reshape(-1), (self.w * (self.y / self.v)).reshape(-1))
        return r, b

    def residual(self, mu=None):
        if mu is None:
            e, l = self.beliefs()
            mu = e / l
        ax, b = self.apply(mu)
        return float(torch.linalg.vector_norm(ax - b) / torch.linalg.vector_norm(b))

    def solve(self, iters, beta, tol=1e-5, every=50, top=200000):
        """`iters` steps, or (0) until the residual is at most tol; the number of steps."""
        done = 0
        while iters == 0 and done < top:
            r = self.residual()
            if not r > tol:
                return done
            for _ in range(every):
                self.step(beta)
            done += every
        for _ in range(iters):
            self.step(beta)
        return iters or done

    def early_stop(self, beta, tau=1e-3):
        ref, t = None, 0
        while t < 10000:
            o = [q.clone() for q in (self.L, self.E, self.oL, self.oE)]
            self.step(beta)
            t += 1
            d = sum(float((p - q).abs().sum()) for p, q in zip((self.L, self.E, self.oL, self.oE), o))
            if t == 2:
                ref = d
            elif t > 2 and d < tau * ref:
                break
        return t


def _exact_pairwise(case, kappa, gamma, xy, y, nv):
    g = _Gabp(case["nx"], case["ny"], kappa, gamma, xy, y, nv)
    offs = [(0, -1), (0, 1), (-1, 0), (1, 0), (-1, -1), (1, 1), (-1, 1), (1, -1), (0, -2), (0, 2), (-2, 0), (2, 0)]
    shape = (g.ny, g.nx)

    def coef(o):
        """P between node i and node i + o."""
        s = torch.zeros(shape, dtype=F64, device=g.a.device)
        for u, ou in enumerate(g.offs):
            for v, ov in enumerate(g.offs):
                if (ov[0] - ou[0], ov[1] - ou[1]) == o:
                    s += gamma * _at(g.a[u] * g.a[v], -ou[0], -ou[1])
        s = s.reshape(-1)
        for cu in range(4):
            for cv in range(4):
                if ((cv >> 1) - (cu >> 1), (cv & 1) - (cu & 1)) == o:
                    s.index_add_(0, g.node[cu], g.w[cu] * g.w[cv] / g.v)
        return s.reshape(shape)

    P0, P = coef((0, 0)), [coef(o) for o in offs]
    h = g.apply(torch.zeros(g.n, dtype=F64, device=P0.device))[1].reshape(shape)
    c, rate = case["c"], case["rate"]
    a = [torch.zeros_like(P0) for _ in offs]     # a[d][j]: the message of j to j + offs[d]
    b = [torch.zeros_like(P0) for _ in offs]
    for _ in range(case["iters"]):
        ia, ib = [_at(a[d], -o[0], -o[1]) for d, o in enumerate(offs)], [_at(b[d], -o[0], -o[1]) for d, o in enumerate(offs)]
        ta, tb = sum(ia), sum(ib)
        na, nb = [], []
        for d in range(12):   # the pair's message back arrives from the opposite direction d ^ 1
            al = P0 + c * (ta - ia[d ^ 1]) + (c - 1) * ia[d ^ 1]
            be = h + c * (tb - ib[d ^ 1]) + (c - 1) * ib[d ^ 1]
            q = P[d] / c
            na.append((1 - rate) * a[d] - rate * q * q / al)
            nb.append((1 - rate) * b[d] - rate * be * q / al)
        a, b = na, nb
    prec = P0 + c * sum(_at(a[d], -o[0], -o[1]) for d, o in enumerate(offs))
    mu = ((h + c * sum(_at(b[d], -o[0], -o[1]) for d, o in enumerate(offs))) / prec).reshape(-1)
    return {"residual": g.residual(mu), "mean": mu, "var": (1.0 / prec).reshape(-1) if case["var"] else None}


def _exact_mg(case, kappa, gamma, xy, y, nv):
    lv = {}
    for k in range(case["levels"]):
        s = 1 << k
        nx, ny = (case["nx"] + s - 1) // s, (case["ny"] + s - 1) // s
        q = np.minimum(xy / s, np.array([nx - 1.0, ny - 1.0]))
        lv[k] = _Gabp(nx, ny, kappa * s, gamma / (s * s), q, y, nv)
    have, its = None, [0] * case["levels"]
    for k in range(case["levels"] - 1, -1, -1):
        g = lv[k]
        start = None
        if have is not None:   # marginals of the parent nodes
            c = have[0]
            i = torch.arange(g.ny, device=g.a.device).div(2, rounding_mode="floor").clamp(max=c.ny - 1)
            j = torch.arange(g.nx, device=g.a.device).div(2, rounding_mode="floor").clamp(max=c.nx - 1)
            start = [q.reshape(c.ny, c.nx)[i][:, j].reshape(-1) for q in have[1:]]
        if k == 0:
            if start:
                g.warm(*start)
            t = g.early_stop(case["damping"])
            e, l = g.beliefs()
            return {"levels": None, "iterations": None, "mean": e / l}
        beta = case["damping"]
        for _ in range(4):
            g.warm(*start) if start else g.reset()
            best, res = math.inf, math.inf
            for q in range(4001):
                res = g.residual()
                if not math.isfinite(res) or res <= 1e-4 or res > 1e6 * best:
                    break
                best = min(best, res)
                for _ in range(50):
                    g.step(beta)
            if math.isfinite(res) and res < 1.0:
                e, l = g.beliefs()
                have = (g, e / l, l)
                break
            beta = 0.5 * (1.0 + beta)
        else:
            have = (g, *start) if start else None


_NET = [(16, 32, 3, 1), (32, 32, 3, 1), (32, 64, 3, 1), (64, 64, 3, 1), (64, 128, 3, 1), (128, 128, 3, 1),
        (128, 256, 3, 1), (256, 256, 3, 1), (256, 128, 1, 0), (128, 128, 3, 1), (128, 64, 1, 0), (64, 64, 3, 1),
        (64, 32, 1, 0), (32, 32, 3, 1)]   # input and output channels, side of the kernel, ReLU


def _net(params, x):
    """The warm-start network (an encoder-decoder with additive skips) in the type of its input
    [B][C][H][W]; `params` is the flat parameter vector, weights [cout][tap][cin] then bias."""
    at, P = 0, []
    for ci, co, k, _ in _NET:
        w = params[at:at + co * k * k * ci].reshape(co, k, k, ci).permute(0, 3, 1, 2)
        at += co * k * k * ci
        P.append((w, params[at:at + co]))
        at += co
    hw, hb = params[at:at + 64].reshape(2, 32, 1, 1), params[at + 64:at + 66]

    def L(i, q):
        o = F.conv2d(q, P[i][0], P[i][1], padding=_NET[i][2] // 2)
        return torch.relu(o) if _NET[i][3] else o

    up = lambda q: F.interpolate(q, scale_factor=2, mode="nearest")  # noqa: E731
    s0 = L(1, L(0, x))
    s1 = L(3, L(2, F.avg_pool2d(s0, 2)))
    s2 = L(5, L(4, F.avg_pool2d(s1, 2)))
    b3 = L(7, L(6, F.avg_pool2d(s2, 2)))
    d2 = L(9, up(L(8, b3)) + s2)
    d1 = L(11, up(L(10, d2)) + s1)
    d0 = L(13, up(L(12, d1)) + s0)
    return F.conv2d(d0, hw, hb)


def _params():
    return torch.as_tensor(np.load(WEIGHTS).astype(np.float64), device="cuda")


def _learned_start(g, kappa):
    """Initial beliefs from the network on the gridded observations."""
    H, W = (g.ny + 7) // 8 * 8, (g.nx + 7) // 8 * 8
    scale = float(g.y.std())
    fu, fv = g.w[1] + g.w[3], g.w[2] + g.w[3]
    near = g.node[0] + (fu >= 0.5).long() + g.nx * (fv >= 0.5).long()
    s = torch.zeros(g.n, dtype=F64, device=g.y.device).index_add_(0, near, g.y / scale)
    c = torch.zeros_like(s).index_add_(0, near, torch.ones_like(g.y))
    x = torch.zeros((1, 16, H, W), dtype=F64, device=s.device)
    x[0, 0, :g.ny, :g.nx] = (s / c.clamp(min=1)).reshape(g.ny, g.nx)
    x[0, 1, :g.ny, :g.nx] = (c > 0).to(F64).reshape(g.ny, g.nx)
    x[0, 2] = math.log(kappa) + 3.0
    with torch.no_grad():
        o = _net(_params(), x)[0, :, :g.ny, :g.nx].reshape(2, -1)
    g.warm(scale * o[0], torch.exp(o[1].clamp(-10.0, 15.0)))


def exact(case, seed):
    kind, n = case["kind"], case["nx"] * case["ny"]
    if kind == "train":
        x, t = _inputs(case, seed)
        p = _params().requires_grad_(True)
        total, count = 0.0, t.numel() // 2
        for b in range(case["count"]):   # one sample at a time: the activations fit
            o = _net(p, x[b].to(F64).permute(2, 0, 1)[None])[0].permute(1, 2, 0)
            loss = (o - t[b].to(F64)).square().sum() / count
            loss.backward()
            total += float(loss.detach())
        return {"loss": total, "grads": p.grad}
    if kind == "batch":
        out = {"residual": [], "mean": [], "var": []}
        for side, kappa, xy, y, nv in _inputs(case, seed):
            g = _Gabp(side, side, kappa, 1.0, xy, y, nv)
            g.solve(case["iters"], case["damping"])
            e, l = g.beliefs()
            out["residual"].append(g.residual())
            out["mean"].append(e / l)
            if case["var"]:
                out["var"].append(1.0 / l)
        out["residual"] = np.array(out["residual"])
        return out
    kappa, gamma, xy, y, nv = _inputs(case, seed)
    if kind == "pairwise":
        return _exact_pairwise(case, kappa, gamma, xy, y, nv)
    if kind == "mg":
        return _exact_mg(case, kappa, gamma, xy, y, nv)
    g = _Gabp(case["nx"], case["ny"], kappa, gamma, xy, y, nv, case["alpha"])
    if case["start"] == "learned":
        _learned_start(g, kappa)
    g.solve(case["iters"], case["damping"])
    e, l = g.beliefs()
    mu, var = e / l, 1.0 / l if case["var"] else None
    if kind == "window":
        mu, var = mu.cpu().numpy(), var.cpu().numpy() if case["var"] else None
    return {"residual": g.residual(), "iterations": None, "mean": mu, "var": var}
