"""The ways a handle's small levels run (stokes_params.coop_level): in one thread-block cluster (0), as one cooperative
launch (1 .. 6) or by launches of their own (-1, the way also taken where a device holds no cluster).  The three
launch different numbers of kernels, and the last is compared with the oracle's iteration, element by element, from a
given state and from zero.

Tolerances as in test_gpu_cluster.py: 1e-11 of the largest value in float64; 2e-5 for one float32 cycle (about 150
dependent roundings of 2^-24 per value, doubled for the smoother's amplification).
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
    return fem.discretizations(6)


@pytest.mark.parametrize("gamma,coop", [(1, 5), (2, 4), (2, 3)])
def test_coop_level_selects_the_launches(gamma, coop):
    from paper_1502_04070_gb300.solver import Solver
    k = 6
    fn, gn = workloads.random_nodal(k, 3)
    launches = {}
    for cl in (0, coop, -1):
        S = Solver(k + 1, 1e2, precision="mixed", gamma=gamma, coop_level=cl)
        f, g = S.load_vectors(dev(fn), dev(gn), project_g=True)
        before = S.kernel_launches()
        S.solve(f, g, tol=0.0, max_cycles=3)
        launches[cl] = S.kernel_launches() - before
        S.close()
    assert launches[0] <= launches[coop] < launches[-1] and (coop == 5 or launches[0] < launches[coop]), launches


CONFIGS = [(1, 0, 3, 3), (2, 0, 1, 2), (2, 3, 3, 3), (1, 2, 0, 2)]


@pytest.mark.parametrize("k", [2, 4, 5])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("gamma,coarse,nu_pre,nu_post", CONFIGS)
def test_without_a_cluster(discs, k, precision, gamma, coarse, nu_pre, nu_post):
    from paper_1502_04070_gb300.solver import Solver
    coarse = min(coarse, k - 1)
    D = discs[k]
    fn, gn = workloads.random_nodal(k, 31)
    F = D.load(fn, gn, project_g=True)
    tol = 1e-11 if precision == "fp64" else 2e-5
    for beta, zero in ((1.0, False), (1e4, True)):
        if precision == "mixed" and not zero:
            continue   # the float32 cycle of a refinement step always starts from zero
        H = mg.Hierarchy(k + 1, beta, discs[:k + 1], coarse_level=coarse)
        u0, p0 = workloads.random_state(k, 32)
        if zero:
            u0, p0 = np.zeros_like(u0), np.zeros_like(p0)
        prm = mg.Params(nu_pre=nu_pre, nu_post=nu_post, gamma=gamma)
        x = H.project_mean(k, H.cycle(k, D.to_vec(u0, p0), F, prm))
        S = Solver(k + 1, beta, precision=precision, gamma=gamma, coarse_level=coarse, nu_pre=nu_pre, nu_post=nu_post,
                   coop_level=-1)
        f, g = S.load_vectors(dev(fn), dev(gn), project_g=True)
        u, p, _ = S.solve(f, g, tol=0.0, max_cycles=1, u=dev(u0), p=dev(p0))
        y = D.to_vec(host(u), host(p))
        for a, b in ((x[:D.nu], y[:D.nu]), (x[D.nu:], y[D.nu:])):
            assert np.abs(a - b).max() <= tol * np.abs(a).max(), (beta, zero)
        S.close()
