"""The precision form's near field with a warp per leaf and source row: its sums are those of the kernel for larger
trees to the last bit, so a system evaluated alone (few leaves) equals the same system inside a batch of many leaves."""
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


# leaves of a few, of just over a pass (remainders), of several passes and tiles; one dense leaf; empty leaves; the
# split coordinates of wide leaves; no boundary bands
CASES = [
    ("d2_32", lambda: fi.uniform(512, seed_index=101, depth=2, p=8)),
    ("d3_few", lambda: fi.uniform(200, seed_index=102, depth=3, p=8)),
    ("d4_33_to_97", lambda: fi.uniform(16500, seed_index=103, depth=4, p=8)),
    ("d3_130", lambda: fi.uniform(8400, seed_index=104, depth=3, p=8)),
    ("d2_600", lambda: fi.uniform(9700, seed_index=105, depth=2, p=8)),
    ("d3_dense", lambda: fi.clustered(12000, seed_index=106, depth=3, p=8)),
    ("d4_split", lambda: fi.uniform(9000, seed_index=107, depth=4, p=8, sigma=1e-4)),
    ("d4_no_bands", lambda: fi.uniform(9000, seed_index=108, depth=4, p=8, sigma=0.04)),
]


@pytest.mark.parametrize("tile", [(32, 4), (64, 4), (64, 2), (256, 4), (256, 2)])
@pytest.mark.parametrize("name,make", CASES, ids=[c[0] for c in CASES])
def test_few_leaves_match_many_leaves_bitwise(lib, name, make, tile):
    w = make()
    big = fi.uniform(5000, seed_index=109, depth=6, p=8, sigma=0.001)  # 4096 more leaves of one particle
    f = lib.FMM(w.depth, w.p, w.sigma, precision="mixed", domain=w.domain)
    f.set_p2p_tile(*tile)
    u, v = f.velocity_near(dev(w.x), dev(w.y), dev(w.gamma))
    uf, vf = f.velocity_far(dev(w.x), dev(w.y), dev(w.gamma))
    f.sync()
    fb = lib.FMM(w.depth, w.p, w.sigma, precision="mixed")
    fb.set_p2p_tile(*tile)
    off = [0, w.n, w.n + big.n]
    ub, vb = fb.velocity_batched(off, *(dev(np.concatenate([getattr(w, k), getattr(big, k)])) for k in ("x", "y", "gamma")),
                                 depths=[w.depth, big.depth], sigmas=[w.sigma, big.sigma], domains=[w.domain, big.domain])
    fb.sync()
    # the batch sums the near and far parts in FP32
    for near, far, both in ((u, uf, ub), (v, vf, vb)):
        assert torch.equal((near.float() + far.float()).double(), both[: w.n])
