"""FP64 at N = 2: the stage kernel takes sixteen lanes per element on small active sets and
four on large ones (the batch kernel and the operators-in-global variant always four); the
two are the same arithmetic, bit for bit, on both sides of the line (eight warps of two
elements per SM).
"""
import numpy as np
import pytest

from workloads import scenarios as sc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_1661_gb300 import build
    build.build()


@pytest.mark.parametrize("scheme", ["cubature", "collocation", "cubature_2n"])
@pytest.mark.parametrize("side", ["few", "below", "at", "above"])
def test_lane_counts_agree(scheme, side):
    import torch
    import paper_1403_1661_gb300 as P
    from paper_1403_1661_gb300 import _native as nat
    line = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    K = {"few": 3, "below": line - 1, "at": line, "above": line + 1}[side]
    ny = 6
    scn = sc.tsunami(nx=(K + 2 * ny - 1) // (2 * ny), ny=ny, N=2, nlevels=4)
    vx, vy, tri = scn.build_mesh()
    cx = vx[tri].mean(axis=1)
    arrays = (vx, vy, tri[np.sort(np.argsort(cx, kind="stable")[::-1][:K])])
    a, b = (P.solver_from_scenario(scn, precision="fp64", mesh_arrays=arrays, scheme=scheme) for _ in range(2))
    assert a.K == K
    assert torch.equal(a.rhs_variant(nat.SWE_RHS_FUSED_SIMT), a.rhs_variant(nat.SWE_RHS_GLOBAL_OPS))
    batch = P.Batch([b])
    a.step(2)
    batch.step(2)
    for u, v in zip(a.get_state(), b.get_state()):
        assert np.array_equal(u, v)
    batch.close()
