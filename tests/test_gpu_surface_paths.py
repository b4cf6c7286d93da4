"""Crossing edges, vertex weights, normals and boundary values on grids that take every path of
their kernels: rows shorter and longer than a thread's 16 edges, rows that end inside them, one
plane more than a z slab, and so many cut edges that the list for the union overflows."""
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


def _molecule(n, seed):
    a = pb_inputs.globular_molecule(n, seed=seed)
    a[:, :3] -= a[:, :3].mean(0)
    return a


def _dust(n, half, seed):
    """Small balls all over the box: most edges they cut have both ends in the solvent, more of
    them than the list holds (an eighth of the nodes and 1,024)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    a = np.zeros((n, 5))
    a[:, :3] = rng.uniform(-half, half, (n, 3))
    a[:, 3] = rng.uniform(0.1, 0.22, n)
    a[:, 4] = 0.1
    return a


CASES = [((12, 40, 33), 0.6, "mol"), ((16, 17, 18), 0.9, "mol"), ((47, 15, 16), 0.9, "mol"),
         ((41, 33, 35), 0.45, "mol"), ((24, 24, 24), 0.5, "dust"), ((9, 30, 30), 0.5, "dust")]


@pytest.mark.parametrize("n,h,kind", CASES)
def test_surface_is_the_oracles(pb, orc, n, h, kind):
    half = 0.5 * h * (min(n) - 1)
    atoms = _molecule(14, 31) if kind == "mol" else _dust(3000, half - 1.01 * h, 32)
    g = orc.Grid(n, tuple(-0.5 * h * (m - 1) for m in n), h)
    if kind == "mol":  # fit the shortest side
        atoms[:, :4] *= 0.9 * (half - 1.1 * h) / np.abs(atoms[:, :3]).max()
    gg = pb.pb_build_grid(pb.GridSpec(n=n, origin=tuple(g.origin), h=h, fill=0.0), atoms)
    inside = orc.classify(g, atoms)
    ref = orc.crossing_edges(g, atoms, inside)
    assert np.array_equal(pb.pb_get_array(gg, "inside"), inside)
    for name, key in (("cross_id", "ids"), ("cross_alpha", "alpha"), ("cross_rp", "rp"), ("cross_sign", "sign")):
        assert np.array_equal(pb.pb_get_array(gg, name), ref[key]), name
    assert np.array_equal(pb.pb_get_array(gg, "mc_weight"), orc.mc_weights(g, inside, ref))
    assert np.array_equal(pb.pb_get_array(gg, "mc_normal"), orc.mc_normals(ref, atoms))
    lB, kD = orc.units()
    coef = orc.assemble(g, inside, ref, 2.0, 80.0, kD)
    for bc, obc in ((pb.BC_DH, orc.BC_DH), (pb.BC_COULOMB, orc.BC_COULOMB), (pb.BC_ZERO, orc.BC_ZERO)):
        s = pb.pb_assemble_coeffs(gg, pb.Params(bc=bc))
        b = orc.bc_values(g, atoms, lB, 80.0, obc, kD)
        f = orc.rhs(g, atoms, lB, coef, b)
        assert np.array_equal(pb.pb_get_array(s, "diag"), np.where(orc_boundary(g), 0.0, coef["diag"]))
        # every term of a value is good to a few roundings
        assert np.abs(pb.pb_get_array(s, "bc") - b).max() <= 1e-14 * max(np.abs(b).max(), 1e-300) * len(atoms) ** 0.5
        assert np.abs(pb.pb_get_array(s, "rhs") - f).max() <= 1e-13 * np.abs(f).max()


def orc_boundary(g):
    nx, ny, nz = (int(v) for v in g.n)
    m = np.ones((nz, ny, nx), bool)
    m[1:-1, 1:-1, 1:-1] = False
    return m.reshape(-1)
