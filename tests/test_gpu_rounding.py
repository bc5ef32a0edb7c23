"""Rounding of the float64 kernels that sum whole stencil rows at once, against the same sums with exact coefficients in
extended precision.  The exact coefficients are the oracle's, whose integrals are multiples of 1/6 (stiffness), h^2/360 (mass)
and h/12 (divergence), rounded to those.
"""
import numpy as np
import pytest

from oracle import fem
from tests._gpu import dev, host

pytestmark = pytest.mark.gpu


def _exact(M, unit):
    M = M.tocoo()
    k = np.rint(M.data * unit)
    assert np.abs(M.data * unit - k).max() < 1e-6
    return M.row, M.col, k.astype(np.longdouble) / np.longdouble(unit), M.shape[0]


def _times(E, x):
    row, col, val, n = E
    y = np.zeros(n, np.longdouble)
    np.add.at(y, row, val * x.astype(np.longdouble)[col])
    return y


def test_residual_rounds_no_more_than_separate_products():
    """f - A u - B^T p of order-one (u, p) and a load-sized f: the relative error (2-norm, N = 64) is at most the 1.43e-16
    that A u and B^T p summed apart have."""
    from paper_1502_04070_gb300.solver import Solver
    k, beta = 5, 1e4
    n = 2 ** (k + 1)
    d = fem.discretizations(k + 1)[-1]
    K, M, B = _exact(d.Ki, 6), _exact(d.Mi, 360 * n * n), _exact(d.Bi.T, 12 * n)
    rng = np.random.default_rng(6)
    u = rng.uniform(-1, 1, (2, 2 * n + 1, 2 * n + 1))
    f = rng.uniform(-1, 1, (2, 2 * n + 1, 2 * n + 1)) / n ** 2
    for a in (u, f):
        a[:, 0], a[:, -1], a[:, :, 0], a[:, :, -1] = 0.0, 0.0, 0.0, 0.0
    p, g = rng.uniform(-1, 1, (n + 1, n + 1)), np.zeros((n + 1, n + 1))
    S = Solver(k + 1, beta)
    ru, rp = S.residual(dev(u), dev(p), dev(f), dev(g))
    got = d.to_vec(host(ru), host(rp))[:d.nu]
    x, b = d.to_vec(u, p), d.to_vec(f, g)
    au = np.concatenate([_times(K, c) + beta * _times(M, c) for c in (x[:d.ni], x[d.ni:d.nu])])
    want = b[:d.nu].astype(np.longdouble) - au - _times(B, x[d.nu:])
    err = got.astype(np.longdouble) - want
    assert float(np.sqrt((err * err).sum() / (want * want).sum())) <= 1.43e-16


def test_load_vectors_have_exact_coefficients():
    """The load vector of a basis function is a column of the mass matrix: every entry is its multiple of h^2/360 (velocity,
    at the unknowns) and h^2/24 (pressure, off the boundary), rounded once.  N = 8; basis functions in every orientation
    class, their neighbours included."""
    from paper_1502_04070_gb300.solver import Solver
    k = 2
    n = 2 ** (k + 1)
    d = fem.discretizations(k + 1)[-1]
    S = Solver(k + 1, 1.0)
    for y in range(1, 2 * n):
        for x in range(1, 2 * n):
            fn, gn = np.zeros((2, 2 * n + 1, 2 * n + 1)), np.zeros((n + 1, n + 1))
            fn[0, y, x] = fn[1, y, x] = 1.0
            if x <= n and y <= n:
                gn[y, x] = 1.0
            f, g = [host(t) for t in S.load_vectors(dev(fn), dev(gn), project_g=False)]
            F = d.load(fn, gn)
            wf, wg = d.from_vec(F)
            for got, want, unit in ((f, wf, 360.0 * n * n), (g[1:-1, 1:-1], wg[1:-1, 1:-1], 24.0 * n * n)):
                assert np.abs(want * unit - np.rint(want * unit)).max() < 1e-9
                assert np.array_equal(got, np.rint(want * unit) / unit), (x, y)
