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
