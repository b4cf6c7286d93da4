"""Multigrid preconditioner of the mixed-precision solver: the solution does not depend on
it (true residual under the oracle's operator), and it is at work on every grid that has a
hierarchy, whatever the sizes, spacings and permittivities."""
import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_09323_gb300 import build
    build.build()
    import paper_2502_09323_gb300 as pb
    return pb


# n, eps_in, eps_out, hierarchy.  Sizes around the tile (64 x 16 fine, 32 x 8 coarse nodes), the
# coarsening (n - 1 even or odd on each level) and the bottom kernel's limits; 8 nodes on an axis
# and the long thin grid keep the Jacobi preconditioner.
CASES = [
    ((9, 9, 9), 2.0, 80.0, True),
    ((10, 12, 11), 2.0, 80.0, True),
    ((33, 33, 33), 2.0, 80.0, True),
    ((33, 33, 33), 80.0, 2.0, True),
    ((35, 34, 37), 1.0, 1000.0, True),
    ((65, 17, 18), 2.0, 80.0, True),
    ((66, 16, 35), 4.0, 4.0, True),
    ((131, 31, 9), 2.0, 80.0, True),
    ((8, 20, 20), 2.0, 80.0, False),
    ((9, 9, 4000), 2.0, 80.0, False),
]


@pytest.mark.parametrize("n,ein,eout,hierarchy", CASES)
def test_solution_and_iterations(pb, orc, n, ein, eout, hierarchy):
    atoms = pb_inputs.globular_molecule(12, seed=77)
    atoms[:, :3] -= atoms[:, :3].mean(0)
    h = 18.0 / (min(n) - 1)
    g = orc.Grid(n, tuple(-0.5 * h * (m - 1) for m in n), h)
    gg = pb.pb_build_grid(pb.GridSpec(n=n, origin=tuple(g.origin), h=h, fill=0.0), atoms)
    s = pb.pb_assemble_coeffs(gg, pb.Params(eps_in=ein, eps_out=eout, bc=pb.BC_COULOMB))
    st = pb.pb_solve(s, pb.SolveOpts(precision=pb.MIXED, rtol=1e-10))
    assert st["status"] == 0 and st["true_rel_res"] <= 1e-10
    phi, bc, f = (pb.pb_get_array(s, k) for k in ("phi", "bc", "rhs"))
    coef = {k: pb.pb_get_array(s, k) for k in ("Wx", "Wy", "Wz", "diag")}
    r = f - orc.apply(g, coef, phi - bc)
    assert np.linalg.norm(r) <= 1.01e-10 * np.linalg.norm(f)
    # V(1,1) takes 26 iterations to 1e-10 on such grids (CPU prototype); Jacobi over 100 on 33^3
    if hierarchy:
        assert st["iters_inner"] <= 60
    # alone, in a batch and as the one rank of a split solve: the same bits
    st2 = pb.pb_solve_batch([s], pb.SolveOpts(precision=pb.MIXED, rtol=1e-10))[0]
    assert st2["iters_inner"] == st["iters_inner"] and np.array_equal(pb.pb_get_phi(s), phi)
    st3 = pb.pb_solve_split(s, 1, pb.SolveOpts(precision=pb.MIXED, rtol=1e-10))
    assert st3["iters_inner"] == st["iters_inner"] and np.array_equal(pb.pb_get_phi(s), phi)


# h_bulk (one to four levels of refinement from 0.25 A), explicit coarse bricks (0: automatic),
# lattice correction; the four-level tree keeps the Jacobi preconditioner
OCTREES = [(0.5, 0, True), (1.0, 0, True), (1.0, 7, True), (2.0, 0, True), (2.0, 4, True), (4.0, 0, False)]


@pytest.mark.parametrize("h_bulk,n0,lattice", OCTREES)
def test_octree_solution_and_iterations(pb, h_bulk, n0, lattice):
    atoms = pb_inputs.globular_molecule(25, seed=78)
    o = tuple(atoms[:, :3].mean(0) - 4.0 * h_bulk * n0)
    spec = pb.OctreeSpec(h_fine=0.25, h_bulk=h_bulk, refine_dist=6.0 if h_bulk > 2.0 else 3.0, n0=n0, origin=o)
    s = pb.pb_assemble_coeffs(pb.pb_build_grid(spec, atoms), pb.Params(bc=pb.BC_DH))
    # the plain FP64 solver (Jacobi, FP64 operator) on the same system
    ref = pb.pb_solve(s, pb.SolveOpts(precision=pb.FP64, rtol=1e-12))
    phi64 = pb.pb_get_phi(s)
    st = pb.pb_solve(s, pb.SolveOpts(precision=pb.MIXED, rtol=1e-12))
    phi = pb.pb_get_phi(s)
    assert ref["status"] == 0 and st["status"] == 0 and st["true_rel_res"] <= 1e-12
    # two solutions of relative residual 1e-12: their difference is at most the condition number
    # (under 1e4 here) times that
    assert np.linalg.norm(phi - phi64) <= 1e-8 * np.linalg.norm(phi64)
    if lattice:
        assert st["iters_inner"] <= 80  # 13 to 21 per 1e-6 in the CPU prototype
    st2 = pb.pb_solve_batch([s], pb.SolveOpts(precision=pb.MIXED, rtol=1e-12))[0]
    assert st2["iters_inner"] == st["iters_inner"] and np.array_equal(pb.pb_get_phi(s), phi)


@pytest.mark.parametrize("n,ein,eout,hierarchy", CASES)
def test_fp64_solution_and_iterations(pb, orc, n, ein, eout, hierarchy):
    """The plain FP64 solver with its own (FP64) cycle, and the operator alone in both types on
    the same grids (ragged rows, one or several blocks a plane) against the oracle's."""
    atoms = pb_inputs.globular_molecule(12, seed=79)
    atoms[:, :3] -= atoms[:, :3].mean(0)
    h = 18.0 / (min(n) - 1)
    g = orc.Grid(n, tuple(-0.5 * h * (m - 1) for m in n), h)
    gg = pb.pb_build_grid(pb.GridSpec(n=n, origin=tuple(g.origin), h=h, fill=0.0), atoms)
    s = pb.pb_assemble_coeffs(gg, pb.Params(eps_in=ein, eps_out=eout, bc=pb.BC_COULOMB))
    st = pb.pb_solve(s, pb.SolveOpts(precision=pb.FP64, rtol=1e-11))
    assert st["status"] == 0 and st["true_rel_res"] <= 1e-11
    if hierarchy:
        assert st["iters_inner"] <= 60
    phi, bc, f = (pb.pb_get_array(s, k) for k in ("phi", "bc", "rhs"))
    coef = {k: pb.pb_get_array(s, k) for k in ("Wx", "Wy", "Wz", "diag")}
    r = f - orc.apply(g, coef, phi - bc)
    assert np.linalg.norm(r) <= 1.01e-11 * np.linalg.norm(f)
    import torch
    x = pb_inputs.random_field(g.N, seed=80)
    y = orc.apply(g, coef, np.where(np.asarray(coef["diag"]) > 0, x, 0.0))
    xd = torch.from_numpy(x).cuda()
    y64 = pb.pb_apply(s, xd).cpu().numpy()
    assert np.abs(y64 - y).max() <= 1e-12 * np.abs(y).max()
    y32 = pb.pb_apply(s, xd.float(), pb.MIXED).cpu().numpy()
    assert np.abs(y32 - y).max() <= 1e-5 * np.abs(y).max()
