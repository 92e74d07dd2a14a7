"""Adaptive leaves' U and W lists against the oracle where they can go wrong: capacities of one (a leaf per particle), leaves
with more neighbours than a list holds (a coarse leaf beside a very fine patch), leaves of level 1, odd and even range ends
of the packed pairs, coincident particles. Tolerances as for the other adaptive parity tests: 1e-12 in the plain form,
1e-6 in the precision form (relative L2)."""
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


def fine_patch(n, seed, std):
    """Half the particles within a few std of a point beside a leaf edge, half spread out: coarse leaves with many fine
    neighbours."""
    r = fi.rng(seed)
    m = n // 2
    x = np.concatenate([0.5 + std * r.standard_normal(m), r.random(n - m)])
    y = np.concatenate([0.25 + std * r.standard_normal(m), r.random(n - m)])
    return np.clip(x, 0, 0.9999), np.clip(y, 0, 0.9999), r.standard_normal(n) / n


CASES = [
    ("cap1", lambda: fi.two_scale(900, 301), 6, 1, 12),
    ("cap3", lambda: fi.two_scale(2000, 302), 8, 3, 12),
    ("many_neighbours", lambda: fine_patch(6000, 303, 1e-3), 11, 4, 12),
    ("level1", lambda: fine_patch(300, 304, 1e-2), 4, 120, 12),
    ("odd_ranges", lambda: fi.two_scale(5001, 305), 9, 17, 16),
]


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-6)])
@pytest.mark.parametrize("name,make,L,B,p", CASES, ids=[c[0] for c in CASES])
def test_adaptive_lists(lib, oracle, name, make, L, B, p, precision, tol):
    x, y, g = make()
    x[5], y[5] = x[4], y[4]  # coincident
    f = lib.FMM(L, p, 2e-3, precision=precision, domain=(0.0, 0.0, 1.0), leaf_capacity=B)
    u, v = f.velocity(dev(x), dev(y), dev(g))
    f.sync()
    ref = np.concatenate(oracle.adaptive_fmm(x, y, g, 2e-3, L, B, p, domain=(0.0, 0.0, 1.0)))
    got = np.concatenate([u.cpu().numpy(), v.cpu().numpy()])
    assert np.linalg.norm(got - ref) < tol * np.linalg.norm(ref)
