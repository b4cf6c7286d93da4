"""Multigrid hierarchies that cannot be built: nothing of a failed one stays on the system.
Allocations are refused, or misplaced, by the allocator hooks."""
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
