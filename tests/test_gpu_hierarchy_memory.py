"""Multigrid hierarchies that cannot be built: nothing of a failed one stays on the system, and
one that memory has no room for is done without.  Allocations are refused, or misplaced, by the allocator hooks."""
import numpy as np
import pytest

import pb_inputs

pytestmark = pytest.mark.gpu


class Hooks:
    """Allocator hooks over torch's allocator that note every allocation."""

    def __init__(self, torch):
        self.torch = torch
        self.reset()
        self.live = {}  # pointer handed out: (pointer of torch, bytes)

    def reset(self, refuse=None, shift=None):
        self.sizes, self.refuse, self.shift = [], refuse, shift

    def alloc(self, ctx, nbytes, stream):
        at = len(self.sizes)
        self.sizes.append(nbytes)
        if self.refuse and self.refuse(at, self.sizes):
            return None
        off = 4 if self.shift and self.shift(at, self.sizes) else 0
        p = self.torch.cuda.caching_allocator_alloc(nbytes + off, self.torch.cuda.current_device(), stream or 0)
        self.live[p + off] = (p, nbytes)
        return p + off

    def free(self, ctx, ptr, stream):
        self.torch.cuda.caching_allocator_delete(self.live.pop(ptr, (ptr, 0))[0])

    def count(self, nbytes):
        return sum(n == nbytes for _, n in self.live.values())


@pytest.fixture
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_09323_gb300 as pb
    from paper_2502_09323_gb300 import _native as N
    h = Hooks(torch)
    pb.use_torch_allocator()
    a, f = N.ALLOC_FN(h.alloc), N.FREE_FN(h.free)
    N.check(N.lib().pb_set_allocator(a, f, None))
    yield pb, h
    torch.cuda.synchronize()
    N.check(N.lib().pb_set_allocator(*N.kept(), None))


def _uniform(pb):
    atoms = pb_inputs.globular_molecule(60, seed=51)
    s = pb.pb_assemble_coeffs(pb.pb_build_grid(pb.GridSpec(n=(49, 49, 49), fill=1.5), atoms), pb.Params())
    return s, 64 * 49 * 49  # rows of 49 are padded to 64


def test_failed_build_leaves_nothing(env):
    """A vector that a tensor map cannot take (an address that is no multiple of 16 bytes): the
    solve reports the refused map, and the hierarchy's own vector is given back."""
    pb, h = env
    s, n = _uniform(pb)
    before = h.count(4 * n)
    h.reset(shift=lambda at, sizes: sizes[at] == 4 * n and sizes.count(4 * n) == 1)  # z
    for _ in range(2):
        st = pb.pb_solve(s, pb.SolveOpts(precision=pb.MIXED), check=False)
        assert st["rc"] < 0 and "cuTensorMapEncodeTiled" in pb.pb_last_error()
        assert h.count(4 * n) == before + 4  # z, two directions and the correction
    s.free()
    assert h.count(4 * n) == 0


def _octree(pb):
    atoms = pb_inputs.globular_molecule(25, seed=52)
    g = pb.pb_build_grid(pb.OctreeSpec(h_fine=0.25, h_bulk=1.0, refine_dist=3.0), atoms)
    return pb.pb_assemble_coeffs(g, pb.Params()), g.N


# system, precision, vectors of the solver itself, allocations of the preconditioner after them
# (None: all), iterations that Jacobi exceeds and the preconditioned solver does not
KINDS = {"uniform": (_uniform, 1, 4, 4, 60), "fp64": (_uniform, 0, 11, 2, 60), "octree": (_octree, 1, 4, None, 60)}


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("batch", [False, True])
def test_without_room_for_a_hierarchy(env, kind, batch):
    pb, h = env
    make, prec, vectors, after, few = KINDS[kind]
    opts = pb.SolveOpts(precision=prec, rtol=1e-10)
    esz = 4 if prec else 8

    def solve(s):
        return pb.pb_solve_batch([s], opts)[0] if batch else pb.pb_solve(s, opts)

    s, n = make(pb)
    h.reset()
    ref = solve(s)
    sizes, phi = list(h.sizes), pb.pb_get_phi(s)
    assert ref["status"] == 0 and ref["iters_inner"] <= few
    last = [at for at, b in enumerate(sizes) if b == esz * n][vectors - 1]
    end = len(sizes) if after is None else last + 1 + after
    assert end - last - 1 >= 2
    for at in range(last + 1, end):
        s, _ = make(pb)
        h.reset(refuse=lambda q, _: q == at)
        st = solve(s)
        assert st["status"] == 0 and st["true_rel_res"] <= 1e-10 and st["iters_inner"] > few
        # residuals of 1e-10 and a condition number under 1e3 on these grids
        assert np.linalg.norm(pb.pb_get_phi(s) - phi) <= 1e-7 * np.linalg.norm(phi)
        live = sum(b for _, b in h.live.values())
        # with room again the same system takes the hierarchy
        h.reset()
        st = solve(s)
        assert st["iters_inner"] == ref["iters_inner"] and np.array_equal(pb.pb_get_phi(s), phi)
        # what was refused, and all that belongs to it, had been given back
        assert sum(b for _, b in h.live.values()) - live >= sizes[at]
        s.free()


@pytest.mark.parametrize("kind", list(KINDS))
def test_solve_after_one_that_ran_out_of_memory(env, kind):
    """Every allocation of a first solve that it cannot do without, refused in turn: the solve
    reports it, and the next one of the same system goes on from what is there."""
    pb, h = env
    make, prec, vectors, _, _ = KINDS[kind]
    opts = pb.SolveOpts(precision=prec, rtol=1e-10)
    s, n = make(pb)
    h.reset()
    ref = pb.pb_solve(s, opts)
    sizes, phi = list(h.sizes), pb.pb_get_phi(s)
    last = [at for at, b in enumerate(sizes) if b == (4 if prec else 8) * n][vectors - 1]
    for at in range(last + 1):
        s, _ = make(pb)
        h.reset(refuse=lambda q, _: q == at)
        assert pb.pb_solve(s, opts, check=False)["rc"] == -2
        h.reset()
        st = pb.pb_solve(s, opts)
        assert st["iters_inner"] == ref["iters_inner"] and np.array_equal(pb.pb_get_phi(s), phi)
        s.free()
