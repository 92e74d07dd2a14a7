"""Memory of the adaptive leaves' U and W lists, and the walk that takes over where they have no room. Tolerances as for the
other adaptive parity tests: 1e-12 in the plain form, 1e-6 in the precision form (relative L2)."""
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


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_memory_of_the_lists_is_bounded(lib, precision):
    """The workspace grows by at most 256 MB (and the workspace's eighth of it, and 16 MB for the granularity of allocations)
    as the capacity falls (more leaves, more lists), for 2^21 particles."""
    w = fi.uniform(1 << 21, seed_index=171, depth=9, p=8)
    x, y, g = dev(w.x), dev(w.y), dev(w.gamma)
    u, v = torch.empty_like(x), torch.empty_like(x)
    used = []
    for capacity in (128, 128, 8, 1):  # the first for the modules
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        f = lib.FMM(w.depth, w.p, w.sigma, precision=precision, domain=w.domain, leaf_capacity=capacity)
        f.velocity(x, y, g, u, v)
        f.sync()
        used.append(free - torch.cuda.mem_get_info()[0])
        f.close()
    assert max(used[2:]) < used[1] + (304 << 20), used


def spikes(m, L, seed):
    """m tight clusters of 129, and around each a single particle in every sibling of the boxes that hold it: with 128 to a
    leaf, many leaves of one particle."""
    r = fi.rng(seed)
    c = 0.01 + 0.98 * r.random((m, 2))
    z = [np.repeat(c, 129, axis=0) + 1e-7 * r.standard_normal((129 * m, 2))]
    for l in range(4, L + 1):
        box = np.floor(c * 2 ** l).astype(int)
        for s in ((1, 0), (0, 1), (1, 1)):
            z.append(((box ^ np.array(s)) + 0.25 + 0.5 * r.random((m, 2))) / 2 ** l)
    z = np.concatenate(z)
    return z[:, 0].copy(), z[:, 1].copy(), r.standard_normal(len(z)) / len(z)


def leaves(x, y, L, capacity):
    """Non-empty leaves of the adaptive tree on the unit square."""
    n, split = 0, None
    for l in range(L + 1):
        key = np.floor(x * 2 ** l).astype(int) * 2 ** l + np.floor(y * 2 ** l).astype(int)
        live = np.ones(x.size, bool) if split is None else split
        k, inv, cnt = np.unique(key[live], return_inverse=True, return_counts=True)
        over = cnt > capacity if l < L else np.zeros(cnt.size, bool)
        n += int((~over).sum())
        split = live.copy()
        split[live] = over[inv]
    return n


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("mixed", 1e-6)])
def test_more_leaves_than_lists(lib, oracle, precision, tol):
    x, y, g = spikes(128, 11, 172)
    assert leaves(x, y, 11, 128) > 1.2 * max(x.size / 16 + 1024, x.size / 10)  # room for lists
    f = lib.FMM(11, 12, 2e-3, precision=precision, domain=(0.0, 0.0, 1.0), leaf_capacity=128)
    u, v = f.velocity(dev(x), dev(y), dev(g))
    f.sync()
    ref = np.concatenate(oracle.adaptive_fmm(x, y, g, 2e-3, 11, 128, 12, domain=(0.0, 0.0, 1.0)))
    got = np.concatenate([u.cpu().numpy(), v.cpu().numpy()])
    assert np.linalg.norm(got - ref) < tol * np.linalg.norm(ref)
