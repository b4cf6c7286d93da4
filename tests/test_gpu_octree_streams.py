"""Octrees of one engine iterate on streams of their own: fewer and more of
them than streams, each with the bits of its pb_solve."""
import time

import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 8, 11])
def test_octrees_beside_each_other(count):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    opts = pb.SolveOpts(precision=pb.MIXED, rtol=1e-10)
    spec = pb.OctreeSpec(h_fine=0.5, h_bulk=1.0, refine_dist=2.0, fill=1.8)

    def system(i):
        g = pb.pb_build_grid(spec, pb_inputs.globular_molecule(30 + 25 * i, seed=700 + i))
        return pb.pb_assemble_coeffs(g, pb.Params())

    alone = []
    for i in range(count):
        s = system(i)
        alone.append((pb.pb_solve(s, opts)["iters_inner"], pb.pb_get_phi(s)))
    with pb.Engine(capacity=count, opts=opts) as eng:
        of = {eng.submit(system(i)): i for i in range(count)}
        got, t_end = [], time.time() + 60
        while len(got) < count:
            assert time.time() < t_end, "engine did not finish"
            got += eng.wait(timeout_s=0.05)
    for r in got:
        iters, phi = alone[of[r["ticket"]]]
        assert r["stats"]["status"] == 0 and r["stats"]["iters_inner"] == iters
        assert np.array_equal(pb.pb_get_phi(r["system"]), phi)
