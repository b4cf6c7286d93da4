"""The waits of the multigrid cycle's own kernels: bounded by the limit that pb_set_wait_limit sets,
as those of the PCG kernels are."""
import time

import numpy as np
import pytest

from test_gpu_hierarchy_memory import _uniform, env  # noqa: F401

pytestmark = pytest.mark.gpu


class _View:
    def __init__(self, ptr, n):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<f4", "data": (ptr, False), "version": 3}


@pytest.mark.parametrize("how", ["alone", "batch", "engine"])
def test_wait_limit_reaches_the_cycle(env, how):  # noqa: F811
    """With no polls allowed the first kernel of the cycle gives up: the solve ends with its
    status, and the cycle's result, which was cleared when the hierarchy was made, is never
    written.  With the limit back the same system solves to the bits of another that never saw it."""
    import torch
    pb, h = env
    opts = pb.SolveOpts(precision=pb.MIXED, rtol=1e-10)
    twin, n = _uniform(pb)
    pb.pb_set_tuning(twin, pb.MIXED, 1, 8)  # by shape: no timing runs under the short limit
    ref = pb.pb_solve(twin, opts)
    phi = pb.pb_get_phi(twin)
    s, _ = _uniform(pb)
    before = h.count(4 * n)
    try:
        pb.pb_set_wait_limit(0)
        if how == "alone":
            status = pb.pb_solve(s, opts, check=False)["status"]
        elif how == "batch":
            status = pb.pb_solve_batch([s], opts, check=False)[0]["status"]
        else:
            with pb.Engine(capacity=2, opts=opts) as eng:
                eng.submit(s)
                got, end = [], time.time() + 60
                while not got and time.time() < end:
                    got = eng.wait(timeout_s=0.05)
                status = got[0]["stats"]["status"]
        assert status == -5
        v = [p for p, (_, b) in h.live.items() if b == 4 * n][before + 4]  # after the solver's four vectors
        v = torch.as_tensor(_View(v, n), device="cuda")
        assert not bool(v.any())
    finally:
        pb.pb_set_wait_limit(-1)
    st = pb.pb_solve(s, opts)
    assert bool(v.any())
    assert st["iters_inner"] == ref["iters_inner"] and np.array_equal(pb.pb_get_phi(s), phi)
    del v
