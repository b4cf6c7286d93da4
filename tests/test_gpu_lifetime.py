"""A system keeps its grid alive: the caller may free the grid first, and the
garbage collector finalises the two in either order when both lie in a cycle."""
import gc

import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("octree", [False, True])
def test_grid_freed_before_its_systems(octree):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    atoms = pb_inputs.globular_molecule(60, seed=17)
    spec = (pb.OctreeSpec(h_fine=0.5, h_bulk=1.0, refine_dist=2.0, fill=1.8) if octree
            else pb.GridSpec(n=(33, 37, 41), origin=(-15.0, -16.0, -17.0), h=0.9))
    opts = pb.SolveOpts(precision=pb.MIXED, rtol=1e-9)

    def make():
        g = pb.pb_build_grid(spec, atoms)
        return g, [pb.pb_assemble_coeffs(g, pb.Params()) for _ in range(2)]

    def solve(s):
        pb.pb_coulomb_terms(s, pb.CT_SURFACE | pb.CT_PAIRS)
        assert pb.pb_solve(s, opts)["status"] == 0
        return pb.pb_energy(s)

    g, (a, b) = make()
    energy = solve(a)
    g.free()
    a.free()
    assert solve(b) == energy
    b.free()
    # the same through the collector: a cycle holds both
    torch.cuda.synchronize()
    gc.collect()
    before = torch.cuda.memory_allocated()
    cycle = list(make())
    cycle.append(cycle)
    del cycle
    gc.collect()
    assert torch.cuda.memory_allocated() == before
