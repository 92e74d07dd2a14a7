"""The plain form's near field and its adjoint where fixed-point pairs could differ from FP64 ones in single particles that
a norm over all of them hides: coincident particles, weak charges, particles close to a coordinate axis."""
import numpy as np
import pytest

import fmm_inputs as fi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1008_2410_gb300 import api, build

    build.build()
    return api


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("sigma", [0.05, 0.01, 1e-4])  # every pair close; close pairs listed; close pairs in FP64
@pytest.mark.parametrize("copies", [2, 5])
def test_adjoint_of_coincident_particles(lib, oracle, sigma, copies):
    """Coincident particles do not act on one another, in the adjoint too. Tolerance 1e-11 relative L2 over the coincident
    particles alone: sums of a thousand terms with one more level of products, each within a few 2^-53 of its size."""
    w = fi.uniform(3000, seed_index=141, depth=2, p=12, sigma=sigma)
    same = np.arange(40 * copies).reshape(40, copies)
    w.x[same], w.y[same] = w.x[same[:, :1]], w.y[same[:, :1]]
    r = np.random.default_rng(8)
    gu, gv = r.standard_normal(w.n) / w.n, r.standard_normal(w.n) / w.n
    f = lib.FMM(w.depth, w.p, w.sigma, precision="fp64", domain=w.domain)
    got = f.adjoint(dev(w.x), dev(w.y), dev(w.gamma), dev(gu), dev(gv))
    f.sync()
    ref = oracle.fmm_adjoint(w.x, w.y, w.gamma, w.sigma, w.depth, w.p, gu, gv, domain=w.domain)
    for a, b in zip(got, ref):
        a, b = a.cpu().numpy()[same.ravel()], b[same.ravel()]
        assert np.linalg.norm(a - b) < 1e-11 * np.linalg.norm(b)


# ---------------------------------------------------------------- each particle against direct sums in long double

Q = np.longdouble
TWO_PI = 2 * Q("3.14159265358979323846264338327950288")


def blob(x):
    """F(x) = (1 - e^-x) / x and F'(x): Taylor series below 1, the formulas from there on."""
    F, D = np.zeros_like(x), np.zeros_like(x)
    m = x < 1
    t = np.ones_like(x[m])  # (-x)^k / (k + 1)!
    for k in range(40):
        F[m] += t
        D[m] -= t * (k + 1) / (k + 2)
        t = t * -x[m] / (k + 2)
    X = x[~m]
    F[~m] = (1 - np.exp(-X)) / X
    D[~m] = ((1 + X) * np.exp(-X) - 1) / (X * X)
    return F, D


def pairs(w):
    """Displacements, F k2 and 2 F' k2^2 of every pair (targets by rows); zero for coincident ones. Depth 1: all near."""
    x, y = w.x.astype(Q), w.y.astype(Q)
    a, b = x[:, None] - x[None, :], y[:, None] - y[None, :]
    k2 = 1 / (2 * Q(w.sigma) ** 2)
    F, D = blob(((a * a + b * b) * k2).ravel())
    F, D = F.reshape(a.shape) * k2, D.reshape(a.shape) * 2 * k2 * k2
    same = (a == 0) & (b == 0)
    F[same] = D[same] = 0
    return a, b, F, D


def bound(n):
    """An FP64 sum of n terms, each within a few 2^-53 of its size, is off by less than (n + 8) 2^-53 sum |terms|."""
    return (n + 8) * 2.0 ** -53 / (2 * np.pi)


def close_to_axes(ratio, spread):
    """300 particles within a few spread * sigma of the origin, leaves of width 1 / 8 = sigma / ratio."""
    r = fi.rng(142)
    w = fi.uniform(300, seed_index=143, depth=1, p=4, sigma=0.125 * ratio)
    w.x, w.y = (spread * w.sigma * r.standard_normal(w.n) for _ in range(2))
    w.domain = (-0.125, -0.125, 0.25)
    return w


def weak_around_strong(weak, apart, sigma=1 / 32):
    """Two particles of charge 1, apart * sigma from each other, among 574 of the order of weak."""
    w = fi.uniform(576, seed_index=144, depth=1, p=4, sigma=sigma)
    w.gamma = weak * fi.rng(145).standard_normal(w.n)
    w.gamma[:2] = 1.0
    w.x[1], w.y[1] = w.x[0] + apart * w.sigma, w.y[0]
    return w


EXACT = [
    ("uniform", lambda: fi.uniform(1500, seed_index=146, depth=1, p=4)),
    ("axes_16", lambda: close_to_axes(1 / 16, 2.0)),
    ("axes_16_tight", lambda: close_to_axes(1 / 16, 1e-4)),
    ("axes_60", lambda: close_to_axes(1 / 60, 2.0)),
    ("axes_60_tight", lambda: close_to_axes(1 / 60, 1e-2)),
    ("axes_500", lambda: close_to_axes(2e-3, 2.0)),
    ("axes_1e5", lambda: close_to_axes(1e-5, 2.0)),
    ("axes_1e7", lambda: close_to_axes(1e-7, 2.0)),
    ("axes_1e9", lambda: close_to_axes(1e-9, 2.0)),
    ("weak_1e-9", lambda: weak_around_strong(1e-9, 0.0)),
    ("weak_1e-12", lambda: weak_around_strong(1e-12, 0.0)),
    ("weak_1e-12_apart", lambda: weak_around_strong(1e-12, 1e-8)),
    ("weak_1e-9_narrow", lambda: weak_around_strong(1e-9, 0.0, sigma=0.2)),
]


@pytest.mark.parametrize("name,make", EXACT, ids=[c[0] for c in EXACT])
def test_each_velocity(lib, name, make):
    w = make()
    f = lib.FMM(w.depth, w.p, w.sigma, precision="fp64", domain=w.domain)
    u, v = (t.cpu().numpy() for t in f.velocity_near(dev(w.x), dev(w.y), dev(w.gamma)))
    f.sync()
    a, b, F, _ = pairs(w)
    g = w.gamma.astype(Q)
    tu, tv = -b * F * g, a * F * g
    err = np.maximum(abs(u - tu.sum(1) / (TWO_PI)), abs(v - tv.sum(1) / (TWO_PI)))
    size = np.maximum(abs(tu).sum(1), abs(tv).sum(1))
    worst = float((err / size).max())
    print(f"{name}: {worst / bound(w.n):.2e} of the bound")
    assert worst < bound(w.n)


def test_gradient_of_charges_far_from_one(lib):
    """Charges of 1e-188 with gradients of 1e200; every tenth target 1e-119 times as strong in both (its charge times the
    unit of the others' is below FP64's range, its gradient is not). Tolerance 1e-11 relative L2 over those, as for the
    other adjoint tests (the same sums, scaled)."""
    w = fi.uniform(1500, seed_index=148, depth=1, p=4)
    r = fi.rng(149)
    g, gu, gv = r.standard_normal((3, w.n))
    s = np.ones(w.n)
    s[::10] = 1e-119
    f = lib.FMM(w.depth, w.p, w.sigma, precision="fp64", domain=w.domain)
    got = [t.cpu().numpy() for t in f.adjoint(dev(w.x), dev(w.y), dev(g * s * 1e-188), dev(gu * s * 1e200), dev(gv * s * 1e200))]
    f.sync()
    a, b, F, D = pairs(w)
    g, gu, gv = (t.astype(Q) * s for t in (g, gu, gv))
    cu = g[None, :] * gu[:, None] - g[:, None] * gu[None, :]
    cv = g[None, :] * gv[:, None] - g[:, None] * gv[None, :]
    J1, J2, ab = F + b * b * D, F + a * a * D, a * b * D
    ref = (F * (gu[None, :] * b - gv[None, :] * a)).sum(1), (cv * J2 - cu * ab).sum(1), (cv * ab - cu * J1).sum(1)
    # in units of 1e200 (dgamma), 1e-188 1e200 1e-119 = 1e-107 (dx, dy of the weak targets)
    for q, t, unit, strength in zip(got, ref, (1e200, 1e-107, 1e-107), (1.0, 1e-119, 1e-119)):
        q, t = q[::10] / unit, t[::10] / strength / TWO_PI
        assert np.linalg.norm((q - t).astype(float)) < 1e-11 * np.linalg.norm(t.astype(float))


@pytest.mark.parametrize("grads", ["normal", "like_charges"])
@pytest.mark.parametrize("name,make", EXACT, ids=[c[0] for c in EXACT])
def test_each_gradient(lib, name, make, grads):
    w = make()
    r = fi.rng(147)
    gu, gv = r.standard_normal(w.n), r.standard_normal(w.n)
    if grads == "like_charges":  # strong and weak like gamma, of either sign
        gu, gv = gu * abs(w.gamma), gv * abs(w.gamma)
    f = lib.FMM(w.depth, w.p, w.sigma, precision="fp64", domain=w.domain)
    got = [t.cpu().numpy() for t in f.adjoint(dev(w.x), dev(w.y), dev(w.gamma), dev(gu), dev(gv))]
    f.sync()
    a, b, F, D = pairs(w)
    g, gu, gv = (t.astype(Q) for t in (w.gamma, gu, gv))
    cu = g[None, :] * gu[:, None], g[:, None] * gu[None, :]
    cv = g[None, :] * gv[:, None], g[:, None] * gv[None, :]
    J1, J2, ab = F + b * b * D, F + a * a * D, a * b * D  # -dKu/db, dKv/da, dKv/db = -dKu/da
    dg = F * (gu[None, :] * b - gv[None, :] * a)
    dx = (cv[0] - cv[1]) * J2 - (cu[0] - cu[1]) * ab
    dy = (cv[0] - cv[1]) * ab - (cu[0] - cu[1]) * J1
    size_g = (F * (abs(gu[None, :] * b) + abs(gv[None, :] * a))).sum(1)
    size_xy = ((abs(cu[0]) + abs(cu[1]) + abs(cv[0]) + abs(cv[1])) * (F + (a * a + b * b) * abs(D))).sum(1)
    worst = [float((abs(q - t.sum(1) / TWO_PI) / s).max()) / bound(w.n)
             for q, t, s in zip(got, (dg, dx, dy), (size_g, size_xy, size_xy))]
    print(f"{name} {grads}: {worst} of the bound")
    assert max(worst) < 1.0
