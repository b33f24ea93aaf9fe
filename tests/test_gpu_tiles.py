"""Element counts at the edges of the stage kernels' warp tiles (2, 8 or 16 elements
per tile, by tier and order): fewer elements than a tile, exactly one, one more, and a
last tile with a single element, against the FP64 oracle.

R and one macro step (three levels, PP + TVB, a partly dry beach) within the bounds
derived from the arithmetic: R 1e-11 / 2e-5 / 2e-4 of max|R| (FP64, FP32, FP32 with
tensor cores), states 1e-11 / 2e-5 / 8e-5 of max h and of max h sqrt(g max h).
"""
import numpy as np
import pytest

from tests.gpu_helpers import both, state_errors
from workloads import meshes, scenarios as sc

pytestmark = pytest.mark.gpu

TOL_R = {"fp64": 1e-11, "fp32": 2e-5, "fp32tc": 2e-4}
TOL_Q = {"fp64": 1e-11, "fp32": 2e-5, "fp32tc": 8e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_1661_gb300 import build
    build.build()


def _scenario(N, K):
    """The first K triangles of a graded, jittered strip, the bed rising out of the water."""
    nx = (K + 5) // 6 + 1
    def mesh():
        vx, vy, tri = meshes.graded_jittered_rect(0.0, 40e3, 0.0, 6e3, nx, 3, ratio=6.0, jitter=0.15, seed=K)
        cx, _ = meshes.centroids(vx, vy, tri)
        return vx, vy, tri[np.argsort(cx, kind="stable")[::-1][:K]]
    s = sc.Scenario(name=f"tiles_N{N}_K{K}", mesh=mesh, N=N, g=9.81, h0=1e-3, cfl=0.4, nlevels=3,
                    limiter_mask=sc.LIM_PP | sc.LIM_TVB, tvb_M=1e-3,
                    bathymetry=lambda x, y, cx=None, cy=None: -60.0 + 62.0 * (x / 40e3) ** 2 + 1e-4 * y, init=None)

    def init(x, y, cx, cy, B):
        h = np.maximum(0.0, 0.5 * np.exp(-((x - 30e3) ** 2) / 4e7) - B)
        return h, 0.2 * h, -0.1 * h
    s.init = init
    return s


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp32tc"])
@pytest.mark.parametrize("N,K", [(1, 5), (1, 33), (2, 1), (2, 2), (2, 3), (2, 17), (2, 64), (3, 8), (3, 9), (3, 65),
                                 (4, 1), (4, 7), (4, 16), (4, 31), (4, 97), (5, 15), (5, 32), (5, 33)])
def test_tile_edges(precision, N, K):
    scn = _scenario(N, K)
    om, ref, model, integ, s = both(scn, precision)
    q = integ.q_end
    R, Ro = s.rhs().cpu().numpy().astype(np.float64), model.rhs(q[0], q[1], q[2])
    scale = max(np.abs(Ro).max(), 1e-300)
    assert np.abs(R - Ro).max() <= TOL_R[precision] * scale
    for _ in range(2 ** (integ.L - 1)):
        integ.substep()
    s.step(1)
    hmax = np.abs(integ.q_end[0]).max()
    eh, em, _ = state_errors(s, integ)
    assert eh <= TOL_Q[precision] * hmax
    assert em <= TOL_Q[precision] * hmax * np.sqrt(scn.g * hmax)
    assert not s.stats()["nonfinite"]
    s.close()
