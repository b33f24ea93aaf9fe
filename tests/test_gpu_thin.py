"""Films of water near the bottom of the number range: velocities are hu / h, whatever the
product of the two depths at a face, and nothing turns non-finite.
"""
import numpy as np
import pytest

from workloads import meshes

pytestmark = pytest.mark.gpu


def _rhs(precision, N, scheme, h0, depth):
    import paper_1403_1661_gb300 as P
    vx, vy, tri = meshes.graded_jittered_rect(0.0, 1.0, 0.0, 1.0, 8, 8, ratio=1.0, jitter=0.1, seed=4)
    s = P.Solver(P.Mesh(vx, vy, tri), N, precision=precision, h0=h0, scheme=scheme)
    x, y = s.mesh.node_coords(N)
    h = depth * (1.0 + 0.2 * x + 0.1 * y)
    s.set_bathymetry(np.zeros_like(h))
    s.set_state(h, 0.3 * h, 0.1 * h * (1.0 + x))
    R = s.rhs().cpu().numpy().astype(np.float64)
    s.close()
    return R


@pytest.mark.parametrize("N,scheme", [(1, "cubature"), (2, "cubature"), (4, "cubature"), (3, "cubature_2n"),
                                      (5, "collocation")])
def test_fp64_depths_whose_product_underflows(N, scheme):
    # gravity is negligible at both depths (sqrt(g h) < 1e-49 against speeds of 0.3), so R is
    # proportional to the depth; FP64 rounding of R at these orders: below 1e-12 of max|R|
    a, b = (_rhs("fp64", N, scheme, 0.1 * d, d) / d for d in (1e-100, 1e-170))
    assert np.isfinite(b).all()
    assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()


@pytest.mark.parametrize("precision", ["fp32", "fp32tc"])
@pytest.mark.parametrize("N,scheme", [(1, "cubature"), (3, "cubature"), (4, "collocation"), (2, "cubature_2n")])
def test_fp32_subnormal_depths(precision, N, scheme):
    # a film of subnormal depth over a subnormal threshold: no velocity, and no infinity from
    # a reciprocal that takes such a depth for zero
    R = _rhs(precision, N, scheme, 2e-39, 5e-39)
    assert np.isfinite(R).all()
