"""The slab code of the split solve against the single solve, on grids too thin for a multigrid
hierarchy: there both run the Jacobi-preconditioned PCG, so one slab gives the single solve's bits
and more slabs differ by the order of their sums only."""
import numpy as np
import pytest

import pb_inputs
from test_gpu_hierarchy_memory import _uniform, env  # noqa: F401

pytestmark = pytest.mark.gpu


# thin in each direction; rows shorter and longer than a tile, planes for several ranks
@pytest.mark.parametrize("n", [(8, 40, 33), (141, 8, 50), (70, 35, 8)])
def test_slabs_are_the_single_jacobi_solve(env, n):  # noqa: F811
    pb, _ = env
    atoms = pb_inputs.globular_molecule(12, seed=302)
    atoms[:, :3] -= atoms[:, :3].mean(0)
    h = 18.0 / (min(n) - 1)
    spec = pb.GridSpec(n=n, origin=tuple(-0.5 * h * (m - 1) for m in n), h=h, fill=0.0)
    s = pb.pb_assemble_coeffs(pb.pb_build_grid(spec, atoms), pb.Params(bc=pb.BC_DH))
    opts = pb.SolveOpts(precision=pb.MIXED, rtol=1e-10)
    ref = pb.pb_solve(s, opts)
    phi = pb.pb_get_phi(s)
    assert ref["status"] == 0
    for ranks in (1, 2, 3, 5):
        st = pb.pb_solve_split(s, ranks, opts)
        got = pb.pb_get_phi(s)
        if ranks == 1:
            assert st["iters_inner"] == ref["iters_inner"] and st["true_rel_res"] == ref["true_rel_res"]
            assert np.array_equal(got, phi)
        # FP32 dot products differ in their last bits: the residual of an iteration by far less than
        # it falls in one
        assert abs(st["iters_inner"] - ref["iters_inner"]) <= 2 + ref["iters_inner"] // 25
        assert st["status"] == 0 and st["true_rel_res"] <= 1e-10
        # residuals of 1e-10 and a condition number under 1e3 on these grids
        assert np.linalg.norm(got - phi) <= 1e-7 * np.linalg.norm(phi)


def test_ranks_build_no_hierarchy(env):  # noqa: F811
    """Several ranks need none (a vector and 3 B a node); the single solve after them takes its own."""
    pb, h = env
    opts = pb.SolveOpts(precision=pb.MIXED, rtol=1e-10)
    twin, n = _uniform(pb)
    ref = pb.pb_solve(twin, opts)
    s, _ = _uniform(pb)
    before = h.count(4 * n)
    st = pb.pb_solve_split(s, 2, opts)
    assert st["status"] == 0 and st["iters_inner"] > 60
    assert h.count(4 * n) == before + 4  # the solver's own vectors
    st = pb.pb_solve(s, opts)
    assert st["iters_inner"] == ref["iters_inner"] and np.array_equal(pb.pb_get_phi(s), pb.pb_get_phi(twin))
