"""An engine whose requests run their first replays while other threads of the program synchronise
the whole device, as any library in it may: no call of either fails."""
import threading
import time

import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


def test_first_replays_beside_device_synchronisations():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    opts = pb.SolveOpts(precision=pb.MIXED, rtol=1e-8)
    atoms = pb_inputs.globular_molecule(40, seed=61)
    # none, one, two and three levels above the smallest, and a small octree beside a thin grid
    specs = [pb.GridSpec(n=n, fill=0.0, h=22.0 / (min(n) - 1),
                         origin=tuple(-11.0 / (min(n) - 1) * (m - 1) for m in n))
             for n in ((8, 20, 20), (33, 33, 33), (65, 65, 65), (129, 129, 129))]
    specs.append(pb.OctreeSpec(h_fine=0.5, h_bulk=1.0, refine_dist=3.0))
    systems = [pb.pb_assemble_coeffs(pb.pb_build_grid(q, atoms), pb.Params()) for q in specs]
    phi = []
    for s in systems:
        assert pb.pb_solve(s, opts)["status"] == 0
        phi.append(pb.pb_get_phi(s))
    stop, errors, count = threading.Event(), [], [0]

    def synchronise():
        try:
            while not stop.is_set():
                torch.cuda.synchronize()
                count[0] += 1
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=synchronise) for _ in range(2)]
    for t in threads:
        t.start()
    try:
        for _ in range(10):
            with pb.Engine(capacity=4, opts=opts) as eng:
                for s in systems[::-1]:
                    eng.submit(s)
                got, end = [], time.time() + 60
                while len(got) < len(systems) and time.time() < end:
                    got += eng.wait(timeout_s=0.05)
            assert [r["stats"]["status"] for r in got] == [0] * len(systems)
            assert all(s["status"] == 0 for s in pb.pb_solve_batch(systems, opts))
    finally:
        stop.set()
        for t in threads:
            t.join()
    assert not errors and count[0] > 0
    for s, p in zip(systems, phi):
        assert np.array_equal(pb.pb_get_phi(s), p)
