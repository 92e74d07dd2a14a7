"""The symmetric near field (tile 128) of trees with more than 1024 leaves: persistent blocks in order of falling work, heavy
leaves to a block and the others to a warp each. A small system evaluated alone (a block per leaf) equals, to the last bit,
the same system in a batch that goes there: beside enough work for its leaves to run on single warps, beside so little that
they are the heavy ones, and beside a system whose near field is another kernel's."""
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


# several passes with remainders, one pass, few particles and empty leaves, dense leaves, more than 1024 leaves alone too
CASES = [
    ("d3_312", lambda: fi.uniform(20000, seed_index=151, depth=3, p=8)),
    ("d3_131", lambda: fi.uniform(8400, seed_index=152, depth=3, p=8)),
    ("d2_300", lambda: fi.uniform(4800, seed_index=153, depth=2, p=8)),
    ("d4_200", lambda: fi.uniform(51200, seed_index=154, depth=4, p=8)),
    ("d4_few", lambda: fi.uniform(600, seed_index=155, depth=4, p=8)),
    ("d3_dense", lambda: fi.clustered(12000, seed_index=156, depth=3, p=8)),
    ("d6_clustered", lambda: fi.clustered(60001, seed_index=157, depth=6, p=8)),
    ("d3_split", lambda: fi.uniform(9000, seed_index=158, depth=3, p=8, sigma=1e-5)),  # not this kernel's
]
# 4096 leaves each: of 640 particles (a warp's share of the work is above a CASES leaf's), of one, of one and not this kernel's
BESIDE = {
    "much": lambda: fi.uniform(4096 * 640, seed_index=159, depth=6, p=8),
    "little": lambda: fi.uniform(5000, seed_index=160, depth=6, p=8),
    "split": lambda: fi.uniform(5000, seed_index=161, depth=6, p=8, sigma=1e-6),
}


@pytest.mark.parametrize("kt", [2, 4])
@pytest.mark.parametrize("beside", list(BESIDE))
@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_ordered_blocks_and_warps_give_the_same_bits(lib, name, make, beside, kt):
    w, big = make(), BESIDE[beside]()
    f = lib.FMM(w.depth, w.p, w.sigma, precision="mixed", domain=w.domain)
    f.set_p2p_tile(128, kt)
    u, v = f.velocity_near(dev(w.x), dev(w.y), dev(w.gamma))
    uf, vf = f.velocity_far(dev(w.x), dev(w.y), dev(w.gamma))
    f.sync()
    fb = lib.FMM(w.depth, w.p, w.sigma, precision="mixed")
    fb.set_p2p_tile(128, kt)
    off = [0, w.n, w.n + big.n]
    ub, vb = fb.velocity_batched(off, *(dev(np.concatenate([getattr(w, k), getattr(big, k)])) for k in ("x", "y", "gamma")),
                                 depths=[w.depth, big.depth], sigmas=[w.sigma, big.sigma], domains=[w.domain, big.domain])
    fb.sync()
    # the batch sums the near and far parts in FP32
    for near, far, both in ((u, uf, ub), (v, vf, vb)):
        assert torch.equal((near.float() + far.float()).double(), both[: w.n])
