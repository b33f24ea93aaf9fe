"""The stage kernels at launch shapes in which every warp takes several tiles, one after the
other (a tile's connectivity and geometry then arrive while the tile before it commits): the
state is that of the default shape, bit for bit, alone and in a batch. The mesh has more
tiles of 16 elements than one CTA of seven warps per SM, and a last tile of one element.
"""
import numpy as np
import pytest

from workloads import scenarios as sc

pytestmark = pytest.mark.gpu


def _solver(N, precision, **kw):
    import torch
    import paper_1403_1661_gb300 as P
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    K = 16 * (7 * sms + sms // 2) + 1
    ny = 40
    scn = sc.tsunami(nx=K // (2 * ny) + 1, ny=ny, N=N, nlevels=4)
    vx, vy, tri = scn.build_mesh()
    order = np.argsort(vx[tri].mean(axis=1), kind="stable")[::-1][:K]   # the shore's end of the strip
    s = P.solver_from_scenario(scn, precision=precision, mesh_arrays=(vx, vy, tri[np.sort(order)]), **kw)
    assert s.K == K
    return s


def _state(s):
    s.step(2)
    q = s.get_state()
    s.close()
    return q


CASES = [(N, "cubature") for N in (2, 3, 4, 5)] + [(3, "collocation"), (5, "collocation"), (2, "cubature_2n"),
                                                   (4, "cubature_2n")]


@pytest.mark.parametrize("N,scheme", CASES)
def test_tensor_core_shapes_agree(N, scheme):
    import paper_1403_1661_gb300 as P
    want = _state(_solver(N, "fp32tc", scheme=scheme))
    assert np.isfinite(want[0]).all()
    for ctas, warps in ((1, 1), (1, 3), (1, 7), (0, 2)):
        s = _solver(N, "fp32tc", scheme=scheme)
        s.set_launch_config({"ctas_per_sm": ctas, "tc_warps": warps})
        for u, v in zip(want, _state(s)):
            assert np.array_equal(u, v)
    s = _solver(N, "fp32tc", scheme=scheme)
    s.set_tc_warps(3)
    b = P.Batch([s], max_macro=2)
    b.step(2)
    for u, v in zip(want, s.get_state()):
        assert np.array_equal(u, v)
    b.close()


@pytest.mark.parametrize("precision,N", [("fp32tc", 2), ("fp32tc", 4), ("fp32tc", 5), ("fp32", 3), ("fp32", 5)])
def test_compensated_shapes_agree(precision, N):
    want = _state(_solver(N, precision, compensated=True))
    s = _solver(N, precision, compensated=True)
    s.set_launch_config({"ctas_per_sm": 1, "tc_warps": 1 if precision == "fp32tc" else None})
    for u, v in zip(want, _state(s)):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("precision,N", [("fp32", 2), ("fp32", 4), ("fp64", 2), ("fp64", 3), ("fp64", 5)])
def test_simt_shapes_agree(precision, N):
    want = _state(_solver(N, precision))
    s = _solver(N, precision)
    s.set_launch_config(1)
    for u, v in zip(want, _state(s)):
        assert np.array_equal(u, v)
