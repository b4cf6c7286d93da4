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
