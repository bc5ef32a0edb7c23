"""The L-shaped domain on planar float32 levels (from N = 128): the first refinement step of a mixed-precision
solve from zero against one float64 cycle on the L (tested against the oracle in test_gpu_lshape.py), at the first
sizes with one, two and three planar levels, where tiles lie on the mid-lines, on the re-entrant sides and inside
the removed quadrant.

Tolerance: about 150 dependent float32 roundings per value through a cycle, doubled for the smoother's
amplification: 2e-5 of the largest value of each field.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels,gamma,nu_pre,nu_post", [(7, 1, 3, 3), (8, 1, 2, 1), (8, 1, 0, 2), (9, 1, 3, 3)])
@pytest.mark.parametrize("beta", [1e2, 1e6])
def test_lshape_planar_step(levels, gamma, nu_pre, nu_post, beta):
    from paper_1502_04070_gb300.solver import Solver
    n = 2 ** levels
    rng = np.random.default_rng(50 + levels)
    f = rng.uniform(-1.0, 1.0, size=(2, 2 * n + 1, 2 * n + 1)) / n ** 2
    g = rng.uniform(-1.0, 1.0, size=(n + 1, n + 1)) / n ** 2
    f[:, 0], f[:, -1], f[:, :, 0], f[:, :, -1], f[:, n:, n:] = 0.0, 0.0, 0.0, 0.0, 0.0
    live = np.ones_like(g)
    live[n // 2 + 1:, n // 2 + 1:] = 0.0
    g = live * (g - (live * g).sum() / live.sum())
    f, g = torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda()
    kw = dict(domain="lshape", coarse_level=1, gamma=gamma, nu_pre=nu_pre, nu_post=nu_post)
    A = Solver(levels, beta, precision="fp64", **kw)
    B = Solver(levels, beta, precision="mixed", **kw)
    ua, pa = A.cycle(A.zeros_u(), A.zeros_p(), f, g)
    ub, pb, _ = B.solve(f, g, tol=0.0, max_cycles=1)
    for x, y in ((ua, ub), (pa, pb)):
        assert float((x - y).abs().max() / x.abs().max()) < 2e-5
    assert float(ub[:, n:, n:].abs().max()) == 0.0 and float(pb[n // 2 + 1:, n // 2 + 1:].abs().max()) == 0.0


@pytest.mark.parametrize("levels", [7, 8])
def test_lshape_cycle_on_compact_levels(levels):
    # a mixed cycle, the float32 step and the restriction on the L give the same bits whatever the layout of a solve
    from paper_1502_04070_gb300.solver import Solver
    n = 2 ** levels
    gen = torch.Generator(device="cuda").manual_seed(levels)
    u, f = (torch.rand(2, 2 * n + 1, 2 * n + 1, generator=gen, device="cuda") - 0.5 for _ in range(2))
    p, g = (torch.rand(n + 1, n + 1, generator=gen, device="cuda") - 0.5 for _ in range(2))
    S = [Solver(levels, 1.0, precision="mixed", domain="lshape", coarse_level=1, tma_level=t) for t in (6, 14)]
    for beta in (1.0, 1e4):
        res = []
        for s in S:
            s.set_beta(beta)
            s.solve(f.double() / n ** 2, g.double() / n ** 2, tol=0.0, max_cycles=1)
            out = list(s.cycle(u.double(), p.double(), f.double() / n ** 2, g.double() / n ** 2))
            out += list(s.residual_restrict_f32(u, p, f, g))
            v, q = u.clone(), p.clone()
            s.smooth_f32(v, q, f, g, 2)
            res.append(out + [v, q])
        assert all(torch.equal(a, b) for a, b in zip(*res))
