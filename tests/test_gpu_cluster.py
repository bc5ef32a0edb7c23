"""The cluster cycle of the small levels (csrc/cluster_cycle.cu): one multigrid iteration against the
oracle's, element by element, at the sizes where the placement of rows changes (every level held by every
CTA, one row per CTA, the highest level of the cluster, the level above it), V- and W-cycles, every coarsest
level (exact solves inside the launch and between launches), odd, zero and unequal smoothing counts, from a given
state and from zero.

Tolerances: float64 as in the parity tests (1e-11 of the largest value); float32 cycles: about 150 dependent
roundings of 2^-24 per value on the way through a cycle, doubled for the amplification by the smoother's
factors (up to 2.2): 2e-5 of the largest value of each field.
"""
import numpy as np
import pytest

from oracle import fem
from oracle import multigrid as mg
from paper_1502_04070_gb300 import workloads
from tests._gpu import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def discs():
    return fem.discretizations(7)


CONFIGS = [(1, 0, 3, 3), (2, 0, 1, 2), (1, 1, 2, 1), (2, 2, 3, 3), (2, 3, 3, 3), (1, 3, 0, 2), (2, 1, 0, 1), (1, 2, 4, 0)]


def _cycle(discs, k, beta, gamma, coarse, nu_pre, nu_post, precision, zero):
    from paper_1502_04070_gb300.solver import Solver
    H = mg.Hierarchy(k + 1, beta, discs[:k + 1], coarse_level=coarse)
    D = discs[k]
    fn, gn = workloads.random_nodal(k, 21)
    F = D.load(fn, gn, project_g=True)
    u0, p0 = workloads.random_state(k, 22)
    if zero:
        u0, p0 = np.zeros_like(u0), np.zeros_like(p0)
    prm = mg.Params(nu_pre=nu_pre, nu_post=nu_post, gamma=gamma)
    x = H.project_mean(k, H.cycle(k, D.to_vec(u0, p0), F, prm))
    S = Solver(k + 1, beta, precision=precision, gamma=gamma, coarse_level=coarse, nu_pre=nu_pre, nu_post=nu_post)
    f, g = S.load_vectors(dev(fn), dev(gn), project_g=True)
    if precision == "fp64":
        u, p = S.cycle(dev(u0), dev(p0), f, g)
    else:   # one step of a solve (a mixed-precision stokes_cycle keeps the order of operations of separate launches)
        u, p, _ = S.solve(f, g, tol=0.0, max_cycles=1, u=dev(u0), p=dev(p0))
    y = D.to_vec(host(u), host(p))
    nu = D.nu
    return [np.abs(a - b).max() / np.abs(a).max() for a, b in ((x[:nu], y[:nu]), (x[nu:], y[nu:]))]


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("gamma,coarse,nu_pre,nu_post", CONFIGS)
def test_cluster_cycle_float64(discs, k, gamma, coarse, nu_pre, nu_post):
    if coarse >= k:
        pytest.skip("coarsest level at or above the finest")
    for beta, zero in ((0.0, False), (1e4, True)):
        eu, ep = _cycle(discs, k, beta, gamma, coarse, nu_pre, nu_post, "fp64", zero)
        assert eu < 1e-11 and ep < 1e-11, (beta, eu, ep)


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("gamma,coarse,nu_pre,nu_post", CONFIGS)
def test_cluster_cycle_float32(discs, k, gamma, coarse, nu_pre, nu_post):
    if coarse >= k:
        pytest.skip("coarsest level at or above the finest")
    for beta in (1.0, 1e6):
        eu, ep = _cycle(discs, k, beta, gamma, coarse, nu_pre, nu_post, "mixed", True)
        assert eu < 2e-5 and ep < 2e-5, (beta, eu, ep)
