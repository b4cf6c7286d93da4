"""Surface sums whose far atoms go through local expansions: no further from FP64 sums over all
pairs than the FP32 sums over all pairs were on the same inputs (2-norm errors of those, measured)."""
import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu

# atoms, seed, finest spacing, charges, shift, errors of Phi, Psi and Psi along the analytic
# normals with all pairs in FP32
CASES = [(20000, 33, 0.25, "", 0.0, (1.26e-7, 1.84e-7, 1.89e-7)),
         (3000, 33, 0.25, "", 1000.0, (1.26e-7, 1.79e-7, 1.83e-7)),
         (5000, 33, 0.25, "positive", 0.0, (8.78e-9, 4.08e-8, 4.88e-8)),
         (9000, 3, 0.5, "neutral", 0.0, (1.87e-7, 1.69e-7, 1.74e-7))]


@pytest.mark.parametrize("n, seed, h, charges, shift, bars", CASES)
def test_no_larger_than_all_pairs(n, seed, h, charges, shift, bars):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    atoms = pb_inputs.globular_molecule(n, seed=seed)
    atoms[:, :3] += shift
    if charges == "neutral":
        atoms[:, 4] -= atoms[:, 4].mean()
    if charges == "positive":
        atoms[:, 4] = np.abs(atoms[:, 4])
    g = pb.pb_build_grid(pb.OctreeSpec(h_fine=h, h_bulk=1.0, refine_dist=3.0), atoms)
    s = pb.pb_assemble_coeffs(g, pb.Params())
    pb.pb_coulomb_terms(s, pb.CT_SURFACE)
    arr = {k: pb.pb_get_array(s, k) for k in ("cross_sign", "cross_id", "cross_rp", "mc_normal", "phi_surf",
                                              "psi_surf", "psi_n")}
    pick = np.random.default_rng(2).choice(np.nonzero(arr["cross_sign"])[0], 20000)
    A = torch.from_numpy(atoms).cuda()
    rp = torch.from_numpy(arr["cross_rp"].reshape(-1, 3)[pick]).cuda()
    mc = torch.from_numpy(arr["mc_normal"].reshape(-1, 3)[pick]).cuda()
    d = torch.from_numpy(arr["cross_id"][pick] // g.N).cuda()
    sign = torch.from_numpy(arr["cross_sign"][pick]).cuda().double()
    exact = [[], [], []]
    for c in torch.split(torch.arange(len(pick), device="cuda"), 1000):
        v = rp[c][:, None] - A[None, :, :3]
        r = v.norm(dim=2)
        G = (A[None, :, 4, None] * v / r[..., None] ** 3).sum(1)
        exact[0].append((A[:, 4] / r).sum(1))
        exact[1].append(sign[c] * torch.gather(G, 1, d[c][:, None])[:, 0])
        exact[2].append((G * mc[c]).sum(1))
    for k, e, bar in zip(("phi_surf", "psi_surf", "psi_n"), exact, bars):
        e = torch.cat(e)
        err = torch.from_numpy(arr[k][pick]).cuda() - e
        assert float(err.norm() / e.norm()) <= bar, k
        if charges == "positive" and k == "phi_surf":  # no cancellation: each value, too
            assert float((err / e).abs().max()) <= 3.5e-8
