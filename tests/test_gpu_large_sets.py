"""The FP32 stage kernel with one thread per element, which large active sets take, against
the kernel with four lanes per element, which the others take: a mesh gives the same R and
the same state bit for bit when elements that it shares no face with are added, enough that
the sets change the kernel. The sizes: the last one on the one side of the line, the first
on the other (a last block of one thread), and one at which every block takes several
elements and the sets of a step lie on both sides.
"""
import numpy as np
import pytest

from workloads import scenarios as sc

pytestmark = pytest.mark.gpu

BLOCKS = {2: 2, 3: 7}   # blocks of 128 elements per SM from which a set takes the kernel
CASES = [(2, "cubature", False), (3, "cubature", False), (2, "collocation", False), (3, "collocation", True),
         (2, "cubature_2n", True), (3, "cubature_2n", False), (2, "cubature", True), (3, "cubature", True)]


def _run(scn, vx, vy, tri, scheme, comp, K):
    import paper_1403_1661_gb300 as P
    nv, rest = len(vx), K - len(tri)
    if rest:
        vx, vy, tri = np.tile(vx, 2), np.tile(vy, 2), np.concatenate([tri, tri[:rest] + nv])
    s = P.solver_from_scenario(scn, precision="fp32", scheme=scheme, compensated=comp, mesh_arrays=(vx, vy, tri))
    assert s.K == K
    if comp:   # open boundaries
        s.set_farfield((100.0, 0.0, 0.0))
    r = s.rhs().cpu().numpy()
    s.step(3)
    out = [r, *s.get_state()[:3]]
    s.close()
    return out


@pytest.mark.parametrize("N,scheme,comp", CASES)
def test_large_sets_agree(N, scheme, comp):
    import torch
    edge = 128 * (BLOCKS[N] * torch.cuda.get_device_properties(0).multi_processor_count - 1)
    n = 7 * edge // 10 | 1
    ny = 40
    scn = sc.tsunami(nx=n // (2 * ny) + 1, ny=ny, N=N, nlevels=4)
    vx, vy, tri = scn.build_mesh()
    order = np.argsort(vx[tri].mean(axis=1), kind="stable")[::-1][:n]   # the shore's end of the strip
    tri = tri[np.sort(order)]
    want = _run(scn, vx, vy, tri, scheme, comp, n)
    assert np.isfinite(want[0]).all() and (comp or all(np.isfinite(x).all() for x in want))
    for K in (edge, edge + 1, 14 * edge // 10):
        got = _run(scn, vx, vy, tri, scheme, comp, K)
        for w, g in zip(want, got):
            w, g = w.reshape(-1, n, w.shape[-1]), g.reshape(-1, K, g.shape[-1])
            assert np.array_equal(w, g[:, :n], equal_nan=True)
