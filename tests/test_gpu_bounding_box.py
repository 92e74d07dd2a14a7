"""The bounding-box square of one system (a part per block, met by a second kernel) equals that of the general kernels,
which take the same system in a batch: the evaluations agree (precision form: to the last bit)."""
import numpy as np
import pytest

import fmm_inputs as fi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [1, 2, 33, 511, 513, 4097, 155649, 400001])
def test_one_system_equals_the_same_in_a_batch(n, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1008_2410_gb300 import api, build

    build.build()
    w = fi.uniform(n, seed_index=141, depth=2, p=4)
    x, y = 3.0 * w.x - 7.0, -0.5 * w.y  # both signs, the extent on one side
    x[n // 2], y[n - 1] = -9.0, 2.5  # the extremes in the middle and last
    depth = 2 if n < 1000 else (3 if n < 10000 else 6)
    f = api.FMM(depth, 4, 1e-3, precision=precision)
    one = f.velocity(dev(x), dev(y), dev(w.gamma))
    f.sync()
    fb = api.FMM(depth, 4, 1e-3, precision=precision)
    two = fb.velocity_batched([0, n, 2 * n], *(dev(np.concatenate([a, b])) for a, b in ((x, x), (y, y), (w.gamma, w.gamma))),
                              depths=[depth] * 2, sigmas=[1e-3] * 2)
    fb.sync()
    for a, b in zip(one, two):
        # (one particle: a square of side 1e-300, which the precision form answers with NaN)
        same = dict(rtol=0.0, atol=0.0, equal_nan=True)
        torch.testing.assert_close(b[:n], b[n:], **same)
        if precision == "fp64":
            same["atol"] = 1e-12 * b.abs().max().item()
        torch.testing.assert_close(a, b[:n], **same)
