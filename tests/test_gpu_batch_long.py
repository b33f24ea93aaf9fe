"""A batch created for long calls: its tickets pass 2^31, its workspace stays small (one
record per phase, none per ticket), and its steps are those of the solvers alone.
"""
import numpy as np
import pytest

from workloads import scenarios as sc

pytestmark = pytest.mark.gpu


def test_long_calls_need_one_record_per_phase():
    import paper_1403_1661_gb300 as P
    from paper_1403_1661_gb300 import _native as nat
    import ctypes as C
    scns = [sc.hump_square(n=170, N=2), sc.dam_break(nx=320, ny=32, N=2)]   # 57,800 and 20,480 elements
    alone = [P.solver_from_scenario(s, precision="fp32") for s in scns]
    mixed = [P.solver_from_scenario(s, precision="fp32") for s in scns]
    macro = 600_000
    assert macro * sum(-(-s.K // 16) for s in mixed) > 2**31
    handles = (C.c_void_p * 2)(*[s.handle.value for s in mixed])
    nbytes = C.c_size_t()
    nat.check(nat.lib().swe_batch_workspace_bytes(handles, 2, macro, C.byref(nbytes)), "swe_batch_workspace_bytes")
    assert 3 * macro * 48 <= nbytes.value < 3 * macro * 48 + 4096   # hump: the stage; dam: the stage and the limiter
    b = P.Batch(mixed, max_macro=macro)
    for n in ([3, 5], [4, 0], [1, 1]):
        assert (b.step(n) == 0).all()
        for s, k in zip(alone, n):
            s.step(k)
    for s, t in zip(alone, mixed):
        for u, v in zip(s.get_state(), t.get_state()):
            assert np.array_equal(u, v)
    b.close()
