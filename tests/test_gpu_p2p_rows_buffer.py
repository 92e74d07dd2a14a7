"""The near field with a warp per leaf and source row where its buffers are smaller than the tiles (four-leaf tiles, 1025 to
4096 leaves of 64 to 111 particles): the same bits as in a batch of more leaves, where another kernel runs."""
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


# the smallest occupancy, rows beyond the buffer here and there, larger buffers, the largest, dense and empty leaves, the
# split coordinates of wide leaves
CASES = [
    ("u64", lambda: fi.uniform(4096 * 64, seed_index=181, depth=6, p=8)),
    ("u79", lambda: fi.uniform(4096 * 79 + 5, seed_index=182, depth=6, p=8)),
    ("u95", lambda: fi.uniform(4096 * 95, seed_index=183, depth=6, p=8)),
    ("u111", lambda: fi.uniform(4096 * 111 + 17, seed_index=184, depth=6, p=8)),
    ("patches", lambda: fi.patches(1 << 18, seed_index=185, depth=6, p=8)),
    ("split", lambda: fi.uniform(4096 * 70, seed_index=186, depth=6, p=8, sigma=1e-6)),
]


@pytest.mark.parametrize("kt", [2, 4])
@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_small_buffers_give_the_same_bits(lib, name, make, kt):
    w = make()
    big = fi.uniform(5000, seed_index=187, depth=6, p=8, sigma=0.001)  # 4096 more leaves
    f = lib.FMM(w.depth, w.p, w.sigma, precision="mixed", domain=w.domain)
    f.set_p2p_tile(256, kt)
    u, v = f.velocity_near(dev(w.x), dev(w.y), dev(w.gamma))
    uf, vf = f.velocity_far(dev(w.x), dev(w.y), dev(w.gamma))
    f.sync()
    fb = lib.FMM(w.depth, w.p, w.sigma, precision="mixed")
    fb.set_p2p_tile(256, kt)
    off = [0, w.n, w.n + big.n]
    ub, vb = fb.velocity_batched(off, *(dev(np.concatenate([getattr(w, k), getattr(big, k)])) for k in ("x", "y", "gamma")),
                                 depths=[w.depth, big.depth], sigmas=[w.sigma, big.sigma], domains=[w.domain, big.domain])
    fb.sync()
    # the batch sums the near and far parts in FP32
    for near, far, both in ((u, uf, ub), (v, vf, vb)):
        assert torch.equal((near.float() + far.float()).double(), both[: w.n])
