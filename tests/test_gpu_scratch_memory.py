"""Scratch that only makes a call faster: where memory has no room for it the call does without,
and gives back what it had of it."""
import numpy as np
import pytest

import pb_inputs
from test_gpu_hierarchy_memory import env  # noqa: F401

pytestmark = pytest.mark.gpu


def test_surface_sums_without_room_for_expansions(env):  # noqa: F811
    """Every allocation of the local expansions (order of the targets, balls, partial sums) refused
    in turn: the sums over all pairs, which differ by FP32 roundings."""
    pb, h = env
    atoms = pb_inputs.globular_molecule(1500, seed=53)
    g = pb.pb_build_grid(pb.OctreeSpec(h_fine=0.25, h_bulk=1.0, refine_dist=3.0), atoms)
    names = ("phi_surf", "psi_surf", "psi_n")
    ref = None
    for at in [None] + list(range(5, 12)):  # the first five: the sums and the split sources
        h.reset()
        s = pb.pb_assemble_coeffs(g, pb.Params())
        before = len(h.live)
        h.reset(refuse=lambda q, _: q == at)
        pb.pb_coulomb_terms(s, pb.CT_SURFACE)
        n = len(h.sizes)
        assert len(h.live) == before + 3 and pb.pb_last_error() == ""
        got = [pb.pb_get_array(s, k) for k in names]
        if at is None:
            ref, total = got, n
            assert total == 12
        for a, b in zip(ref, got):
            assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(a)
            assert at is None or not np.array_equal(a, b)
        s.free()


def test_transition_rows_without_room_for_kept_ones(env):  # noqa: F811
    """The rows that the counting pass of an octree's assembly keeps: refused, they are formed again,
    to the same bits; and they make room for the system's own arrays."""
    pb, h = env
    atoms = pb_inputs.globular_molecule(25, seed=54)
    g = pb.pb_build_grid(pb.OctreeSpec(h_fine=0.25, h_bulk=1.0, refine_dist=3.0), atoms)
    names = ("rhs", "diag")
    opts = pb.SolveOpts(precision=pb.FP64, rtol=1e-12)

    def assemble():
        s = pb.pb_assemble_coeffs(g, pb.Params(bc=pb.BC_ZERO))
        assert pb.pb_last_error() == ""
        out = [pb.pb_get_array(s, k) for k in names]
        pb.pb_solve(s, opts)
        return s, out + [pb.pb_get_phi(s)]

    h.reset()
    s, ref = assemble()
    sizes = list(h.sizes)
    kept = [q for q in range(len(sizes) - 1) if sizes[q] % 96 == 0 and sizes[q] and sizes[q + 1] == 2 * sizes[q]]
    assert len(kept) == 1
    k = kept[0]
    rows = sizes[k] // 96
    values = next(q for q in range(k + 2, len(sizes)) if sizes[q + 1] == 2 * sizes[q] and sizes[q] > 4 * rows)
    s.free()
    before = len(h.live)
    for at in (k, k + 1, values, values + 1):
        h.reset(refuse=lambda q, _: q == at)
        s, got = assemble()
        assert all(np.array_equal(a, b) for a, b in zip(ref, got))
        s.free()
        assert len(h.live) == before


@pytest.mark.parametrize("n", [(49, 49, 49), (16, 37, 70)])
def test_grid_without_room_for_the_candidate_list(env, n):  # noqa: F811
    pb, h = env
    atoms = pb_inputs.globular_molecule(40, seed=55)
    atoms[:, :3] -= atoms[:, :3].mean(0)
    step = 20.0 / (min(n) - 1)
    spec = pb.GridSpec(n=n, origin=tuple(-0.5 * step * (m - 1) for m in n), h=step, fill=0.0)
    names = ("cross_id", "cross_alpha", "cross_rp", "cross_sign", "mc_weight", "mc_normal")
    h.reset()
    g = pb.pb_build_grid(spec, atoms)
    ref = [pb.pb_get_array(g, k) for k in names]
    size = 8 * (n[0] * n[1] * n[2] // 8 + 1024)
    assert h.sizes.count(size) == 1
    h.reset(refuse=lambda q, sizes: sizes[q] == size)
    g = pb.pb_build_grid(spec, atoms)
    assert pb.pb_last_error() == "" and h.sizes.count(size) == 1
    assert all(np.array_equal(a, pb.pb_get_array(g, k)) for a, k in zip(ref, names))
