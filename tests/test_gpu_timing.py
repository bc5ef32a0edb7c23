"""Timing of the finest level's smoothing steps and residuals (stokes_set_timing): the counts of a solve are
those of its steps, whichever calls came between."""
import pytest

from paper_1502_04070_gb300 import workloads
from tests._gpu import dev

pytestmark = pytest.mark.gpu


def _counts(S):
    _, smooth, _, resid = S.timing()
    return smooth + S.timing_fused()[1], resid


@pytest.mark.parametrize("k,precision", [(6, "mixed"), (5, "fp64")])
def test_counts_after_a_cycle_between_two_solves(k, precision):
    from paper_1502_04070_gb300.solver import Solver
    S = Solver(k + 1, 1e2, precision=precision)
    fn, gn = workloads.random_nodal(k, 5)
    f, g = S.load_vectors(dev(fn), dev(gn), project_g=True)
    S.set_timing(True)
    per_step = []
    for _ in range(2):
        before = _counts(S)
        rep = S.solve(f, g, tol=1e-8, max_cycles=100)[2]
        after = _counts(S)
        per_step.append([(b - a) / rep.cycles for a, b in zip(before, after)])
        S.cycle(S.zeros_u(), S.zeros_p(), f, g)
    assert per_step == [[6.0, 1.0], [6.0, 1.0]]


@pytest.mark.parametrize("k,precision,kw", [
    (1, "fp64", {}), (4, "fp64", {}), (4, "fp64", dict(coarse_level=3, nu_pre=2)), (3, "mixed", dict(gamma=2, coarse_level=2)),
    (5, "mixed", dict(inner_cycles=2)), (4, "mixed", dict(smoother="normal")), (4, "mixed", dict(domain="lshape", coarse_level=1)),
    (4, "fp64", dict(domain="lshape", coarse_level=1))])
def test_small_finest_levels_are_counted(k, precision, kw):
    """Every smoothing step of the finest level and one residual a step, also where that level's cycle is one launch
    when it is not timed; the timed solve ends at the same solution (both to 1e-9; 1e-6 of the largest value)."""
    import torch
    from paper_1502_04070_gb300.solver import Solver
    S = Solver(k + 1, 1e2, precision=precision, **kw)
    n = 2 ** (k + 1)
    gen = torch.Generator(device="cuda").manual_seed(k)
    f = torch.rand(2, 2 * n + 1, 2 * n + 1, generator=gen, device="cuda", dtype=torch.float64) - 0.5
    g = torch.zeros(n + 1, n + 1, dtype=torch.float64, device="cuda")
    u0, p0, rep0 = S.solve(f, g, tol=1e-9, max_cycles=500)
    S.set_timing(True)
    u1, p1, rep1 = S.solve(f, g, tol=1e-9, max_cycles=500)
    assert rep0.converged and rep1.converged and abs(rep0.cycles - rep1.cycles) <= 1
    steps = (kw.get("nu_pre", 3) + 3) * kw.get("inner_cycles", 1) * rep1.cycles
    assert _counts(S) == (steps, rep1.cycles)
    for a, b in ((u0, u1), (p0, p1)):
        assert float((a - b).abs().max()) <= 1e-6 * float(a.abs().max())
