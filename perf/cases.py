"""Timed cases of the library's public entry points: what a vortex-particle program asks of it, from one small
evaluation to a clustered field of 2^24 particles, in both forms, on both trees, forward and backward.

``listed()`` names the cases, ``draw(rng)`` gives one more of the same ranges, ``prepare(case, seed)`` makes the
inputs and the handle on the GPU, ``run(state)`` is one pass, ``work(case)`` the bytes and operations it cannot do
without, and ``exact(case, seed)`` the same outputs by direct summation in 64 bits (where that is affordable).

Inputs follow the repository's workloads: sigma = 0.5 / sqrt(N) and about 64 particles per leaf for random fields,
sigma = 2 h for Lamb-Oseen lattices, and a tree depth of round(log4(N / 64)).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1008_2410_gb300 import api, model

DIRECT_PAIRS = 6.0e10  # most pairs that exact() sums directly
DT = 1e-3  # advection step: a particle of the Lamb-Oseen vortex moves about a tenth of the lattice spacing


def _depth(n: int) -> int:
    return max(2, int(round(math.log(n / 64.0, 4))))


def _case(name, kind, n, field, p, precision, **kw):
    c = {"name": name, "kind": kind, "n": n, "field": field, "p": p, "precision": precision, "depth": _depth(n),
         "leaf_capacity": 0, "tile_threads": 0, "tile_targets": 0, "square": True, "graph": True, "nsys": 1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest system a program steps: all launch latency (one graph replay)
        _case("uniform_4k_mixed", "velocity", 4096, "uniform", 12, "mixed"),
        # the plain form on the Lamb-Oseen lattice, called as the defaults are (no graph)
        _case("lattice_16k_fp64", "velocity", 16384, "lattice", 12, "fp64", graph=False),
        # an odd size with the bounding-box root square, every default of the precision form
        _case("uniform_100k_mixed_bbox", "velocity", 100003, "uniform", 14, "mixed", square=False, graph=False),
        # the benchmark's evaluation, with the near-field tile that its tuner keeps
        _case("uniform_1m_mixed", "velocity", 1 << 20, "uniform", 17, "mixed", tile_threads=256, tile_targets=4),
        # the same field in the plain form, which the precision form is checked against
        _case("uniform_1m_fp64", "velocity", 1 << 20, "uniform", 17, "fp64"),
        # the same call on page-locked host arrays: copies in and out are part of it
        _case("host_1m_mixed", "host", 1 << 20, "uniform", 17, "mixed", tile_threads=256, tile_targets=4),
        # clustered field on the uniform tree (dense leaves: the symmetric near-field tile)
        _case("patches_16m_mixed", "velocity", 1 << 24, "patches", 20, "mixed", tile_threads=128, tile_targets=4),
        # clustered field on the adaptive tree
        _case("patches_4m_adaptive_mixed", "velocity", 1 << 22, "patches", 20, "mixed", depth=10, leaf_capacity=48),
        # many independent systems of uneven size in one evaluation
        _case("batched_64_mixed", "batched", 4500000, "uniform", 14, "mixed", nsys=64),
        # one gradient step through the autograd function: evaluation, loss on the velocities, exact adjoint
        _case("gradient_1m_fp64", "gradient", 1 << 20, "uniform", 17, "fp64", graph=False),
        # the adjoint alone with its FP32 near field, at an odd size
        _case("adjoint_120k_mixed", "adjoint", 120007, "uniform", 14, "mixed", graph=False),
        # one Runge-Kutta step (midpoint rule) of a vortex whose root square follows the particles
        _case("advect_160k_mixed", "advect", 160000, "lattice", 14, "mixed", square=False),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["velocity_mixed", "velocity_mixed", "velocity_fp64", "velocity_fp64", "host", "patches", "adaptive",
                       "batched", "gradient", "adjoint", "advect"])
    p = rng.randint(10, 20)
    if kind == "velocity_mixed":
        n = _log_size(rng, 4000, 1 << 22)
        return _draw_case("velocity", n, "uniform", p, "mixed", rng, tile=rng.choice([(0, 0), (256, 4)]))
    if kind == "velocity_fp64":
        n = _log_size(rng, 4000, 1 << 20)
        return _draw_case("velocity", n, rng.choice(["uniform", "lattice"]), p, "fp64", rng)
    if kind == "host":
        n = _log_size(rng, 20000, 1 << 20)
        return _draw_case("host", n, "uniform", p, rng.choice(["mixed", "mixed", "fp64"]), rng)
    if kind == "patches":
        n = _log_size(rng, 1 << 18, 1 << 23)
        return _draw_case("velocity", n, "patches", p, "mixed", rng, tile=(128, 4))
    if kind == "adaptive":
        n = _log_size(rng, 20000, 1 << 23)
        precision = "fp64" if n < 1 << 20 and rng.random() < 0.5 else "mixed"
        return _draw_case("velocity", n, "patches", p, precision, rng, depth=_depth(n) + 2,
                          leaf_capacity=rng.choice([32, 48, 64]))
    if kind == "batched":
        nsys = rng.randint(4, 64)
        return _draw_case("batched", nsys * _log_size(rng, 12000, 70000), "uniform", p, rng.choice(["mixed", "mixed", "fp64"]),
                          rng, nsys=nsys)
    if kind == "gradient":
        return _draw_case("gradient", _log_size(rng, 4000, 1 << 19), "uniform", p, "fp64", rng, graph=False)
    if kind == "adjoint":
        return _draw_case("adjoint", _log_size(rng, 4000, 1 << 20), "uniform", p, rng.choice(["mixed", "fp64"]), rng,
                          graph=False)
    return _draw_case("advect", _log_size(rng, 10000, 1 << 20), "lattice", p, rng.choice(["mixed", "mixed", "fp64"]), rng,
                      square=False)


def _draw_case(kind, n, field, p, precision, rng, tile=(0, 0), **kw):
    c = _case("", kind, n, field, p, precision, tile_threads=tile[0], tile_targets=tile[1],
              **{"graph": rng.random() < 0.7, "square": rng.random() < 0.7, **kw})
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs

def _uniform(n, gen):
    """n uniform points in [0, 1)^2, gamma ~ N(0, 1) / n."""
    x, y = (torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) for _ in range(2))
    return x, y, torch.randn(n, generator=gen, device="cuda", dtype=torch.float64) / n


def _patches(n, gen):
    """n points in 8 Gaussian patches (std 0.05, centres in [0.2, 0.8]^2, circulations +-1) in a random order."""
    c = 0.2 + 0.6 * torch.rand((8, 2), generator=gen, device="cuda", dtype=torch.float64)
    k = torch.randint(0, 8, (n,), generator=gen, device="cuda")
    c = c[k]
    z = c + 0.05 * torch.randn((n, 2), generator=gen, device="cuda", dtype=torch.float64)
    z = torch.where((z < 0.0) | (z >= 1.0), 2.0 * c - z, z).clamp_(0.0, 1.0 - 1e-9)
    gamma = torch.where(k % 2 == 0, 8.0 / n, -8.0 / n).to(torch.float64)
    return z[:, 0].contiguous(), z[:, 1].contiguous(), gamma


def _lattice(n, gen):
    """Lamb-Oseen vortex (circulation 1, core about 0.2) on a lattice of spacing h, first n points of it, each moved
    by up to h / 20; gamma = h^2 omega."""
    side = math.isqrt(n - 1) + 1
    h = 2.0 / side
    i = torch.arange(n, device="cuda")
    move = torch.rand((2, n), generator=gen, device="cuda", dtype=torch.float64) * 0.1 - 0.05
    x = -1.0 + ((i % side) + 0.5 + move[0]) * h
    y = -1.0 + ((i // side) + 0.5 + move[1]) * h
    core2 = float((0.2 + 0.02 * torch.rand(1, generator=gen, device="cuda", dtype=torch.float64)) ** 2)
    return x, y, h * h / (math.pi * core2) * torch.exp(-(x * x + y * y) / core2)


FIELDS = {"uniform": _uniform, "patches": _patches, "lattice": _lattice}


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    n = case["n"]
    if case["kind"] == "batched":
        # sizes log-uniform over a factor of 64 (capped at a quarter of all), summing to n
        s = np.exp(np.random.RandomState(int(seed) % (1 << 31)).uniform(0.0, math.log(64.0), case["nsys"]))
        s = np.minimum(s, s.sum() / 4.0)
        off = np.concatenate([[0], np.round(np.cumsum(s) / s.sum() * n)]).astype(np.int64)
        x, y, g = _uniform(n, gen)
        sizes = np.diff(off)
        g = g * torch.from_numpy(np.repeat(n / sizes, sizes)).cuda()
        return x, y, g, off
    return (*FIELDS[case["field"]](n, gen), gen)


def _sigma(case, n=None):
    n = n or case["n"]
    if case["field"] == "lattice":
        return 2.0 * (2.0 / (math.isqrt(n - 1) + 1))
    return 0.5 / math.sqrt(n)


def _square(case):
    return (-1.0, -1.0, 2.0) if case["field"] == "lattice" else (0.0, 0.0, 1.0)


def _targets(x, y, g, gen, f):
    """Velocities u* of circulations perturbed by 1 %: what a fit of the circulations compares with."""
    n = g.numel()
    return f.velocity(x, y, g + 0.01 * torch.randn(n, generator=gen, device="cuda", dtype=torch.float64) / n)


def prepare(case, seed):
    f = api.FMM(case["depth"], case["p"], _sigma(case), precision=case["precision"],
                domain=_square(case) if case["square"] else None, graph=case["graph"],
                leaf_capacity=case["leaf_capacity"])
    if case["tile_threads"]:
        f.set_p2p_tile(case["tile_threads"], case["tile_targets"])
    s = {"kind": case["kind"], "f": f}
    x, y, g, more = _inputs(case, seed)
    if case["kind"] == "host":
        x, y, g = (t.cpu().pin_memory() for t in (x, y, g))
    s.update(x=x, y=y, g=g)
    if case["kind"] in ("velocity", "host", "batched"):
        s.update(u=torch.empty_like(x, pin_memory=case["kind"] == "host"),
                 v=torch.empty_like(x, pin_memory=case["kind"] == "host"))
    if case["kind"] == "batched":
        sizes = np.diff(more)
        s.update(off=more, kw={"depths": [_depth(int(k)) for k in sizes], "sigmas": [0.5 / math.sqrt(k) for k in sizes],
                               "domains": [(0.0, 0.0, 1.0)] * case["nsys"] if case["square"] else None})
    if case["kind"] == "gradient":
        s["us"], s["vs"] = _targets(x, y, g, more, f)
        for t in (x, y, g):
            t.requires_grad_(True)
    if case["kind"] == "adjoint":
        f.set_adjoint_precision(case["precision"])
        s["gu"], s["gv"] = (torch.randn(x.numel(), generator=more, device="cuda", dtype=torch.float64) / x.numel()
                            for _ in range(2))
    return s


def run(s):
    f, x, y, g = s["f"], s["x"], s["y"], s["g"]
    kind = s["kind"]
    if kind == "velocity":
        return f.velocity(x, y, g, s["u"], s["v"])
    if kind == "host":
        return f.velocity_host(x, y, g, s["u"], s["v"])
    if kind == "batched":
        return f.velocity_batched(s["off"], x, y, g, u=s["u"], v=s["v"], **s["kw"])
    if kind == "adjoint":
        return f.adjoint(x, y, g, s["gu"], s["gv"])
    if kind == "advect":
        f.advect(x, y, g, DT, 1, order=2)
        return x, y
    u, v = api.fmm_velocity(x, y, g, f)
    loss = 0.5 * ((u - s["us"]).square().sum() + (v - s["vs"]).square().sum())
    dg, dx, dy = torch.autograd.grad(loss, (g, x, y))
    return u.detach(), v.detach(), dg, dx, dy


# ---------------------------------------------------------------- work

def _near_pairs(case, n, depth):
    """Ordered pairs of adjacent leaves' particles, from the field's density (patches: 8 Gaussians of std 0.05)."""
    if case["leaf_capacity"]:
        return 6.0 * case["leaf_capacity"] * n  # leaves between a quarter full and full, 9 leaves' worth of neighbours
    w = 2.0 ** -depth
    if case["field"] == "patches":
        return n * n * 9.0 * w * w * (1.0 + 1.0 / (8.0 * 4.0 * math.pi * 0.05 ** 2))
    return n * n * (3.0 * w - 2.0 * w * w) ** 2


def _evaluation_flops(case, n, depth):
    cells = n / case["leaf_capacity"] * 2.0 if case["leaf_capacity"] else 4.0 ** depth
    f = model.flops(n, n / cells, max(2, round(math.log(cells, 4))), case["p"], near_pairs=_near_pairs(case, n, depth))
    return float(sum(f.values()))


def work(case):
    n = case["n"]
    if case["kind"] == "batched":
        # all systems have about 64 particles a leaf: one field of n particles at that occupancy
        return {"bytes": 40.0 * n, "flops": _evaluation_flops(case, n, _depth(n))}
    one = _evaluation_flops(case, n, case["depth"])
    # adjoint: two sweeps (circulations and output gradients) and the near field with the kernel's Jacobian (the
    # kernel's 22 operations and 26 for its derivatives and their products)
    back = one + _evaluation_flops(case, n, case["depth"]) + 26.0 * _near_pairs(case, n, case["depth"])
    return {"velocity": {"bytes": 40.0 * n, "flops": one}, "host": {"bytes": 40.0 * n, "flops": one},
            "advect": {"bytes": 40.0 * n, "flops": 2.0 * one}, "adjoint": {"bytes": 64.0 * n, "flops": back},
            "gradient": {"bytes": 80.0 * n, "flops": one + back}}[case["kind"]]


# ---------------------------------------------------------------- direct sums in 64 bits

def _direct(x, y, g, sigma):
    """(u, v) of Eq. 7: the Gaussian-regularised Biot-Savart kernel summed over all pairs."""
    n = x.numel()
    u, v = torch.empty_like(x), torch.empty_like(x)
    rows = max(1, int(2 ** 27 // n))
    for a in range(0, n, rows):
        dx, dy = x[a:a + rows, None] - x[None, :], y[a:a + rows, None] - y[None, :]
        r2 = dx * dx + dy * dy
        k = torch.where(r2 > 0.0, -torch.expm1(r2 * (-0.5 / sigma ** 2)) / (2.0 * math.pi * r2), 0.0)
        u[a:a + rows] = -((dy * k) @ g)
        v[a:a + rows] = (dx * k) @ g
    return u, v


def _direct_adjoint(x, y, g, gu, gv, sigma):
    """Gradients of sum(gu u + gv v) by (gamma, x, y) of the same sum."""
    n = x.numel()
    dg, dx_, dy_ = (torch.empty_like(x) for _ in range(3))
    rows = max(1, int(2 ** 27 // n))
    k2 = 0.5 / sigma ** 2
    for a in range(0, n, rows):
        t = slice(a, min(n, a + rows))
        dx, dy = x[t, None] - x[None, :], y[t, None] - y[None, :]
        r2 = dx * dx + dy * dy
        safe = torch.where(r2 > 0.0, r2, 1.0)
        om = -torch.expm1(-k2 * r2)
        f = om / (2.0 * math.pi * safe)  # K = (-dy, dx) f(r^2), f = 0 at r = 0 as K is
        fp = torch.where(r2 > 0.0, (k2 * torch.exp(-k2 * r2) * r2 - om) / (2.0 * math.pi * safe * safe), 0.0)
        cu, cv = gu[t, None] * g[None, :] - g[t, None] * gu[None, :], gv[t, None] * g[None, :] - g[t, None] * gv[None, :]
        dg[t] = (dy * f) @ gu - (dx * f) @ gv
        dx_[t] = (-cu * 2.0 * dx * dy * fp + cv * (f + 2.0 * dx * dx * fp)).sum(1)
        dy_[t] = (-cu * (f + 2.0 * dy * dy * fp) + cv * 2.0 * dx * dy * fp).sum(1)
    return dg, dx_, dy_


def exact(case, seed):
    n, kind = case["n"], case["kind"]
    sums = {"advect": 2, "gradient": 5, "adjoint": 3}.get(kind, 1)
    if kind == "batched":
        x, y, g, off = _inputs(case, seed)
        sizes = np.diff(off).astype(np.float64)
        if float((sizes * sizes).sum()) > DIRECT_PAIRS:
            return None
        parts = [_direct(x[a:b], y[a:b], g[a:b], 0.5 / math.sqrt(b - a)) for a, b in zip(off[:-1], off[1:])]
        return torch.cat([q[0] for q in parts]), torch.cat([q[1] for q in parts])
    if sums * float(n) * n > DIRECT_PAIRS:
        return None
    x, y, g, gen = _inputs(case, seed)
    sigma = _sigma(case)
    if kind == "advect":
        u, v = _direct(x, y, g, sigma)
        u, v = _direct(x + 0.5 * DT * u, y + 0.5 * DT * v, g, sigma)
        return x + DT * u, y + DT * v
    if kind == "adjoint":
        gu, gv = (torch.randn(n, generator=gen, device="cuda", dtype=torch.float64) / n for _ in range(2))
        return _direct_adjoint(x, y, g, gu, gv, sigma)
    u, v = _direct(x, y, g, sigma)
    if kind != "gradient":
        return u.cpu() if kind == "host" else u, v.cpu() if kind == "host" else v
    us, vs = _direct(x, y, g + 0.01 * torch.randn(n, generator=gen, device="cuda", dtype=torch.float64) / n, sigma)
    return (u, v, *_direct_adjoint(x, y, g, u - us, v - vs, sigma))
