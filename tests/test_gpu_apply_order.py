"""pb_apply in FP32, operation by operation: the same roundings in the same order as restated in
numpy, so that its error against 64 bits cannot grow unseen."""
import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


def test_fp32_apply_rounds_in_the_stated_order(orc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    n, h = (47, 35, 40), 0.5
    atoms = pb_inputs.globular_molecule(30, seed=71)
    atoms[:, :3] -= atoms[:, :3].mean(0)
    g = pb.pb_build_grid(pb.GridSpec(n=n, origin=tuple(-0.5 * h * (m - 1) for m in n), h=h, fill=0.0), atoms)
    s = pb.pb_assemble_coeffs(g, pb.Params())
    shape, f = n[::-1], np.float32
    W = [pb.pb_get_array(s, k).reshape(shape) for k in ("Wx", "Wy", "Wz")]
    inside = pb.pb_get_array(g, "inside").reshape(shape).astype(bool)
    listed = np.zeros(3 * g.N, bool)
    listed[pb.pb_get_array(g, "cross_id")] = True
    listed = listed.reshape(3, *shape)
    x = np.random.default_rng(72).standard_normal(shape).astype(f)
    y = pb.pb_apply(s, torch.from_numpy(x.reshape(-1)).cuda(), pb.MIXED).cpu().numpy().reshape(shape)
    inner = (slice(1, -1),) * 3

    def at(a, d, o):  # the neighbour o along axis d of every interior node
        q = [slice(1, -1)] * 3
        q[2 - d] = slice(1 + o, a.shape[2 - d] - 1 + o)
        return a[tuple(q)]

    def fma(a, b, c):  # exact product; the sum in 53 bits and then in 24 (a tie lost once in 2^29)
        return (a.astype(float) * b.astype(float) + c.astype(float)).astype(f)

    x0 = np.zeros_like(x)
    x0[inner] = x[inner]
    X = x0[inner]
    pure = np.where(inside[inner], f(2.0 * h), f(80.0 * h)).astype(f)
    kp = pb.pb_get_array(s, "kappa").reshape(shape)[inner].astype(f)
    diff, w, special = [], [], np.zeros(X.shape, bool)
    for d in range(3):
        for o in (-1, 1):
            on = at(listed[d], d, -1) if o < 0 else listed[d][inner]
            v = at(W[d], d, -1) if o < 0 else W[d][inner]
            special |= on
            w.append(np.where(on, v.astype(f), pure))
            diff.append(X - at(x0, d, o))
    tree = ((diff[0] + diff[1]) + (diff[2] + diff[3])) + (diff[4] + diff[5])
    chain = kp * X
    for q in range(6):
        chain = fma(w[q], diff[q], chain)
    want = np.where(special, chain, fma(pure, tree, kp * X))
    assert special.any() and not special.all()
    got = y[inner]
    assert (got == want).mean() >= 0.9999
