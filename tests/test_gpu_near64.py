"""The plain form's near field against the oracle where its split between fixed-point and FP64 pairs can go wrong: few
and many sources, leaves of one to many hundred targets, leaves narrow and wide against sigma, charges of wide range,
offset and tiny squares, coincident particles. Tolerance 1e-12 relative L2: up to a few thousand terms per target,
each within a few 2^-53 of its size, against partial cancellation of signed charges."""
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


def near(lib, w):
    f = lib.FMM(w.depth, w.p, w.sigma, precision="fp64", domain=w.domain)
    u, v = f.velocity_near(dev(w.x), dev(w.y), dev(w.gamma))
    f.sync()
    return np.concatenate([u.cpu().numpy(), v.cpu().numpy()])


def scaled(w, scale, x0, y0):
    w.x, w.y, w.sigma = w.x * scale + x0, w.y * scale + y0, w.sigma * scale
    w.domain = (x0, y0, scale * (1 + 1e-12))
    return w


def charges(w, kind):
    r = np.random.default_rng(5)
    if kind == "strong":  # one in 700 a hundred million times the others
        w.gamma[::700] *= 1e8
    elif kind == "zeros":
        w.gamma[r.random(w.n) < 0.9] = 0.0
    elif kind == "one_sign":
        w.gamma = np.abs(w.gamma) * 1e-150
    elif kind == "lognormal":
        w.gamma = np.exp(3.0 * r.standard_normal(w.n)) * np.where(r.random(w.n) < 0.5, -1.0, 1.0)
    return w


CASES = [
    ("sources_95_97", lambda: fi.uniform(170, seed_index=81, depth=2, p=4, sigma=0.004)),
    ("one_per_leaf", lambda: fi.uniform(900, seed_index=82, depth=5, p=4, sigma=0.001)),
    ("leaf_63_to_65", lambda: fi.uniform(16384, seed_index=83, depth=4, p=4)),
    ("leaf_hundreds", lambda: fi.uniform(20000, seed_index=84, depth=3, p=4)),
    ("leaf_thousands", lambda: fi.clustered(9000, seed_index=85, depth=2, p=4)),
    ("narrow_all_close", lambda: fi.uniform(6000, seed_index=86, depth=4, p=4, sigma=0.05)),
    ("cut_at_leaf_diagonal", lambda: fi.uniform(6000, seed_index=87, depth=3, p=4, sigma=0.125 * 2 ** 1.5 / 75 ** 0.5)),
    ("wide_leaves", lambda: fi.uniform(6000, seed_index=88, depth=3, p=4, sigma=1e-6)),
    ("tiny_square_offset", lambda: scaled(fi.uniform(8000, seed_index=89, depth=3, p=4), 3.7e-9, 1.25, -0.5)),
    ("huge_square", lambda: scaled(fi.uniform(8000, seed_index=90, depth=3, p=4), 3.0e40, -1e40, 2e40)),
    ("square_beyond_range", lambda: scaled(fi.uniform(3000, seed_index=91, depth=3, p=4), 3.0e70, 0.0, 0.0)),
    ("strong_few", lambda: charges(fi.uniform(12000, seed_index=92, depth=4, p=4), "strong")),
    ("mostly_zero", lambda: charges(fi.uniform(12000, seed_index=93, depth=3, p=4), "zeros")),
    ("one_sign_tiny", lambda: charges(fi.uniform(12000, seed_index=94, depth=4, p=4), "one_sign")),
    ("lognormal", lambda: charges(fi.uniform(12000, seed_index=95, depth=4, p=4), "lognormal")),
]


@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_near64_matches_oracle(lib, oracle, name, make):
    w = make()
    if name == "leaf_thousands":  # coincident particles
        w.x[100:104], w.y[100:104] = w.x[100], w.y[100]
    got = near(lib, w)
    uo, vo, _ = oracle.fmm(w.x, w.y, w.gamma, w.sigma, w.depth, w.p, domain=w.domain, parts="near")
    ref = np.concatenate([uo, vo])
    assert np.linalg.norm(got - ref) < 1e-12 * np.linalg.norm(ref)


def test_near64_infinite_charge_stays_with_its_neighbours(lib):
    w = fi.uniform(4000, seed_index=96, depth=3, p=4)
    w.gamma[17] = np.inf
    n = w.n
    got = near(lib, w)
    ix, iy = np.floor(w.x * 8).astype(int), np.floor(w.y * 8).astype(int)
    touched = (np.abs(ix - ix[17]) <= 1) & (np.abs(iy - iy[17]) <= 1)
    touched[17] = False  # a particle does not act on itself
    finite = np.isfinite(got[:n]) & np.isfinite(got[n:])
    assert np.array_equal(finite, ~touched)


ADJ_CASES = ["sources_95_97", "leaf_63_to_65", "leaf_hundreds", "narrow_all_close", "cut_at_leaf_diagonal", "wide_leaves",
             "tiny_square_offset", "strong_few", "mostly_zero", "one_sign_tiny"]  # the oracle overflows beyond 1e70


@pytest.mark.parametrize("grads", ["normal", "outliers", "charges"])
@pytest.mark.parametrize("name", ADJ_CASES)
def test_adjoint_near64_matches_oracle(lib, oracle, name, grads):
    """The adjoint on a tree of depth 1 (all near field) and on the case's own tree, against the oracle's transposed
    stages. The gradients of a target are sums of the same length as above with one more level of products: 1e-11."""
    if (name, grads) == ("strong_few", "charges"):
        pytest.skip("cu cancels products 1e16 times the result: FP64's residue of it is 1e-9 of the result")
    for depth in (1, None):
        w = dict(CASES)[name]()
        w.p = 12
        if depth is not None:
            w.depth = depth
        r = np.random.default_rng(7)
        gu, gv = r.standard_normal(w.n) / w.n, r.standard_normal(w.n) / w.n
        if grads == "outliers":
            gu[::500] *= 1e6
        elif grads == "charges":  # gu proportional to gamma: cu vanishes pair by pair
            gu = 3.0 * w.gamma
        f = lib.FMM(w.depth, w.p, w.sigma, precision="fp64", domain=w.domain)
        got = f.adjoint(dev(w.x), dev(w.y), dev(w.gamma), dev(gu), dev(gv))
        f.sync()
        ref = oracle.fmm_adjoint(w.x, w.y, w.gamma, w.sigma, w.depth, w.p, gu, gv, domain=w.domain)
        for a, b in zip(got, ref):
            assert np.linalg.norm(a.cpu().numpy() - b) < 1e-11 * np.linalg.norm(b)
