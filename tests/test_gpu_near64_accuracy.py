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
