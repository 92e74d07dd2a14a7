"""The symmetric near field (tile 128) gives a heavy leaf to a block and the others to a warp each, in order of falling
work; what is heavy depends on the whole call, so a system evaluated alone (its heavy leaves to blocks) equals, to the
last bit, the same system in a batch with enough work beside it to put its leaves on single warps."""
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


# leaves just above the least heavy work, of several passes with remainders, of less than one round of a block's chunks
# and of more; dense leaves (blocks both times); nothing heavy; empty leaves; a depth without neighbours' neighbours
CASES = [
    ("d3_312", lambda: fi.uniform(20000, seed_index=121, depth=3, p=8)),
    ("d3_131", lambda: fi.uniform(8400, seed_index=122, depth=3, p=8)),
    ("d2_300", lambda: fi.uniform(4800, seed_index=123, depth=2, p=8)),
    ("d4_200", lambda: fi.uniform(51200, seed_index=124, depth=4, p=8)),
    ("d4_few", lambda: fi.uniform(600, seed_index=125, depth=4, p=8)),
    ("d3_dense", lambda: fi.clustered(12000, seed_index=126, depth=3, p=8)),
    ("d6_clustered", lambda: fi.clustered(100001, seed_index=127, depth=6, p=8)),
]


@pytest.mark.parametrize("kt", [2, 4])
@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_blocks_and_warps_give_the_same_bits(lib, name, make, kt):
    w = make()
    big = fi.uniform(1 << 18, seed_index=128, depth=3, p=8)  # 64 leaves of 4096
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


def test_tile_set_after_the_first_evaluation(lib):
    w = fi.clustered(30000, seed_index=129, depth=5, p=8)
    x, y, g = dev(w.x), dev(w.y), dev(w.gamma)
    f = lib.FMM(w.depth, w.p, w.sigma, precision="mixed", domain=w.domain)
    f.velocity(x, y, g)
    f.set_p2p_tile(128, 4)
    u, v = f.velocity(x, y, g)
    f.set_p2p_tile(64, 4)
    f.velocity(x, y, g)
    fs = lib.FMM(w.depth, w.p, w.sigma, precision="mixed", domain=w.domain)
    fs.set_p2p_tile(128, 4)
    us, vs = fs.velocity(x, y, g)
    torch.cuda.synchronize()
    assert torch.equal(u, us) and torch.equal(v, vs)
