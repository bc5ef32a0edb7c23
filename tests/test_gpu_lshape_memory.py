"""Device memory of a mixed-precision handle on the L: all of it comes at set-up, as the boundary says of the allocator's
callbacks, and a handle that fits with compact float32 levels alone is still set up."""
import contextlib

import pytest
import torch

pytestmark = pytest.mark.gpu


class _Budget:
    """Allocator callbacks that count calls and hand out at most `limit` bytes at a time."""

    def __init__(self, limit=None):
        self.calls, self.held, self.peak, self.limit = 0, 0, 0, limit

    def alloc(self, nbytes, stream, ctx):
        self.calls += 1
        if self.limit is not None and self.held + nbytes > self.limit:
            return None
        self.held += nbytes
        self.peak = max(self.peak, self.held)
        return torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))

    def free(self, ptr, nbytes, stream, ctx):
        self.held -= nbytes
        torch.cuda.caching_allocator_delete(int(ptr))


@contextlib.contextmanager
def _allocator(budget):
    from paper_1502_04070_gb300 import _binding as B
    lib = B.load()
    cbs = (B.ALLOC_FN(budget.alloc), B.FREE_FN(budget.free))
    B.check(lib.stokes_set_allocator(cbs[0], cbs[1], None), "stokes_set_allocator")
    try:
        yield
    finally:
        B.check(lib.stokes_set_allocator(B.ALLOC_FN(), B.FREE_FN(), None), "stokes_set_allocator")
        budget.keep = cbs


def _arrays(levels):
    n = 2 ** levels
    gen = torch.Generator(device="cuda").manual_seed(levels)
    u, f = (torch.rand(2, 2 * n + 1, 2 * n + 1, generator=gen, device="cuda") - 0.5 for _ in range(2))
    p, g = (torch.rand(n + 1, n + 1, generator=gen, device="cuda") - 0.5 for _ in range(2))
    return u, p, f / n ** 2, g / n ** 2


LSHAPE = dict(precision="mixed", domain="lshape", coarse_level=1)


def test_calls_allocate_nothing():
    from paper_1502_04070_gb300.solver import Solver
    a = _Budget()
    u, p, f, g = _arrays(7)
    with _allocator(a):
        S = Solver(7, 1.0, **LSHAPE)
        calls = a.calls
        S.cycle(u.double(), p.double(), f.double(), g.double())
        S.smooth_f32(u, p, f, g, 1)
        S.residual_restrict_f32(u, p, f, g)
        S.solve(f.double(), g.double(), tol=0.0, max_cycles=1)
        assert a.calls == calls
        S.close()
    assert a.held == 0


def test_set_up_in_the_memory_of_compact_levels():
    from paper_1502_04070_gb300.solver import Solver
    _, _, f, g = _arrays(8)
    compact, tight = _Budget(), _Budget()
    out = []
    for budget, tma in ((compact, 14), (tight, 0)):
        with _allocator(budget):
            S = Solver(8, 1.0, tma_level=tma, **LSHAPE)
            out.append(S.solve(f.double(), g.double(), tol=0.0, max_cycles=2)[:2])
            S.close()
        tight.limit = compact.peak
    assert tight.peak <= compact.peak and tight.held == 0
    assert all(torch.equal(a, b) for a, b in zip(*out))
