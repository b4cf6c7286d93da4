"""Mixed-precision solves at permittivities whose products leave the range of FP32: the
preconditioner's coarse weights stay finite, as the operator's own do."""
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-25, 1e-18, 1.0, 1e18, 1e25])
@pytest.mark.parametrize("kind", ["uniform", "octree"])
def test_solve(kind, scale):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    atoms = pb_inputs.globular_molecule(20, seed=81)
    spec = (pb.GridSpec(n=(41, 41, 41), fill=1.5) if kind == "uniform"
            else pb.OctreeSpec(h_fine=0.5, h_bulk=1.0, refine_dist=3.0))
    s = pb.pb_assemble_coeffs(pb.pb_build_grid(spec, atoms), pb.Params(eps_in=2.0 * scale, eps_out=80.0 * scale))
    st = pb.pb_solve(s, pb.SolveOpts(precision=pb.MIXED, rtol=1e-8))
    assert st["status"] == 0 and st["true_rel_res"] <= 1e-8
    assert st["iters_inner"] <= 60
    assert pb.pb_solve_batch([s], pb.SolveOpts(precision=pb.MIXED, rtol=1e-8))[0]["status"] == 0
