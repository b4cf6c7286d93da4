"""Boundary values away from the origin and at extreme screening, against sums in extended precision."""
import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu

N = (33, 27, 25)
H = 1.0


def _system(shift, **params):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    atoms = pb_inputs.globular_molecule(60, seed=41)
    atoms[:, :3] += np.array(shift) - atoms[:, :3].mean(0)
    o = [c - 0.5 * H * (m - 1) for c, m in zip(shift, N)]
    g = pb.pb_build_grid(pb.GridSpec(n=N, origin=tuple(o), h=H, fill=0.0), atoms)
    s = pb.pb_assemble_coeffs(g, pb.Params(**params))
    bc = pb.pb_get_array(s, "bc").reshape(N[::-1])
    x = [o[d] + np.arange(N[d], dtype=float) * H for d in range(3)]
    z, y, x = np.meshgrid(x[2], x[1], x[0], indexing="ij")
    edge = np.ones(N[::-1], bool)
    edge[1:-1, 1:-1, 1:-1] = False
    return atoms, np.stack([x[edge], y[edge], z[edge]], 1), bc[edge]


@pytest.mark.parametrize("shift", [(0.0, 0.0, 0.0), (100.0, -70.0, 40.0), (1000.0, -700.0, 900.0)])
@pytest.mark.parametrize("screened", [True, False])
def test_error_does_not_depend_on_the_origin(orc, shift, screened):
    import paper_2502_09323_gb300 as pb
    atoms, p, bc = _system(shift, bc=pb.BC_DH if screened else pb.BC_COULOMB)
    lB, kD = orc.units()
    L = np.longdouble
    r = np.sqrt(((p.astype(L)[:, None] - atoms[None, :, :3].astype(L)) ** 2).sum(2))
    t = (np.exp(-L(kD) * r) if screened else 1) / r * (L(lB) / 80)
    exact, scale = (t * atoms[:, 4]).sum(1), (t * np.abs(atoms[:, 4])).sum(1)
    # A term has about ten roundings of 2^-53 at most, one of them k r = 1 to 4 times over, 0.3 x 2^-53 each
    # in the mean square: 3e-16 at the very most if the 60 terms' errors had one sign; they have
    # not (a factor of sqrt(60) / 1.3), which leaves 5e-17
    assert np.linalg.norm((bc - exact).astype(float)) <= 1.5e-16 * np.linalg.norm(scale.astype(float))


@pytest.mark.parametrize("ionic", [1e10, 1e14, 1e20])
def test_strong_screening_underflows_to_zero(ionic):
    import paper_2502_09323_gb300 as pb
    _, _, bc = _system((0.0, 0.0, 0.0), bc=pb.BC_DH, ionic_strength_M=ionic)
    assert np.all(bc == 0.0)  # k r of 1e5 and more
