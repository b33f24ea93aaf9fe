"""set_state and get_state at the edges of their tiles of 64 elements, for values at the
edges of the two formats: the result is, bit for bit, what the conversions give on the
host (FP32 tiers: h + B rounded to nearest even, less the bed rounded alike).
"""
import numpy as np
import pytest

import paper_1403_1661_gb300 as P
from paper_1403_1661_gb300 import _native as nat
from workloads import meshes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_1661_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32tc"])
@pytest.mark.parametrize("N,K", [(1, 1), (1, 64), (2, 63), (2, 65), (3, 128), (4, 129), (4, 700), (5, 33)])
def test_round_trip(precision, N, K):
    nx = (K + 5) // 6 + 1
    vx, vy, tri = meshes.graded_jittered_rect(0.0, 1e3, 0.0, 200.0, nx, 3, ratio=2.0, jitter=0.1, seed=K)
    mesh = P.Mesh(vx, vy, tri[:K])
    s = P.Solver(mesh, N, precision=precision)
    rng = np.random.default_rng(100 * N + K)
    shape = (K, s.Np)
    B = -10.0 * rng.random(shape)
    h = rng.random(shape) * 5.0
    hu, hv = rng.standard_normal((2, *shape))
    # ties of the 24-bit rounding both ways, a carry into the exponent, zeros of both
    # signs, subnormal and smallest normal floats, the largest ones
    odd = np.array([1 + 2.0**-24, 1 + 3 * 2.0**-24, 1 + 2.0**-24 + 2.0**-52, 2 - 2.0**-26, -(2 - 2.0**-25), 0.0, -0.0,
                    2.0**-126, 2.0**-126 * (1 - 2.0**-25), 3e-39, -1e-45, 1e-60, 2.0**127 * (2 - 2.0**-23), 1.7e38])
    hu.flat[:min(odd.size, hu.size)] = odd[:hu.size]
    hv.flat[::5] = rng.choice(odd, hv.flat[::5].shape)
    s.set_bathymetry(B)
    s.set_state(h, hu, hv)
    got = s.get_state()
    T = np.float64 if precision == "fp64" else np.float32
    ref = ((h + B).astype(T).astype(np.float64) - B.astype(T).astype(np.float64), hu.astype(T).astype(np.float64),
           hv.astype(T).astype(np.float64))
    for g, r in zip(got, ref):
        assert np.array_equal(g.view(np.int64), r.view(np.int64))
    for bad in (np.nan, np.inf, -np.inf):
        x = hv.copy()
        x.flat[-1] = bad
        with pytest.raises(nat.SWEError):
            s.set_state(h, hu, x)
    for g, r in zip(s.get_state()[:3], ref):   # a refused state leaves the old one
        assert np.array_equal(g, r)
    s.close()
