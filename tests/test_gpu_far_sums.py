"""Surface sums of many pairs, whose far atoms go through local expansions,
against FP64 sums over all pairs."""
import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


# a small molecule that takes the expansions, one source past a chunk, and one whose
# target blocks need two pairs of launches
@pytest.mark.parametrize("n, h, one_sign", [(1500, 0.25, False), (4097, 0.5, True), (13000, 0.25, False)])
def test_far_sums(n, h, one_sign):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    atoms = pb_inputs.globular_molecule(n, seed=31)
    if one_sign:
        atoms[:, 4] = np.abs(atoms[:, 4])
    g = pb.pb_build_grid(pb.OctreeSpec(h_fine=h, h_bulk=1.0, refine_dist=3.0), atoms)
    s = pb.pb_assemble_coeffs(g, pb.Params())
    pb.pb_coulomb_terms(s, pb.CT_SURFACE)
    arr = {k: pb.pb_get_array(s, k) for k in ("cross_sign", "cross_id", "cross_rp", "mc_normal", "phi_surf",
                                              "psi_surf", "psi_n")}
    assert len(arr["cross_id"]) * n >= 400000000  # the library's threshold
    flux = np.nonzero(arr["cross_sign"])[0]
    assert np.all(arr["phi_surf"][arr["cross_sign"] == 0] == 0.0)
    pick = np.concatenate([flux[:600], flux[-600:], np.random.default_rng(1).choice(flux, 20000)])
    A = torch.from_numpy(atoms).cuda()
    rp = torch.from_numpy(arr["cross_rp"].reshape(-1, 3)[pick]).cuda()
    mc = torch.from_numpy(arr["mc_normal"].reshape(-1, 3)[pick]).cuda()
    d = torch.from_numpy(arr["cross_id"][pick] // g.N).cuda()
    sign = torch.from_numpy(arr["cross_sign"][pick]).cuda().double()
    got = [torch.from_numpy(arr[k][pick]).cuda() for k in ("phi_surf", "psi_surf", "psi_n")]
    q = A[:, 4]
    for c in torch.split(torch.arange(len(pick), device="cuda"), 2000):
        v = rp[c][:, None] - A[None, :, :3]
        r = v.norm(dim=2)
        G = (q[None, :, None] * v / r[..., None] ** 3).sum(1)
        exact = [(q / r).sum(1), sign[c] * torch.gather(G, 1, d[c][:, None])[:, 0], (G * mc[c]).sum(1)]
        bars = [(q.abs() / r).sum(1), (q.abs() / r ** 2).sum(1), (q.abs() / r ** 2).sum(1)]
        for x, e, b in zip(got, exact, bars):  # the bar of the pair sums, as on uniform grids
            assert float(((x[c] - e).abs() / b).max()) <= 2e-6
