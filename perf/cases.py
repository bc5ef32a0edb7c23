"""The calls that users of the solver make, at the sizes they make them.

listed() names the cases, draw() gives others of the same ranges, prepare() builds what a program has
in hand before the call, run() makes the call, work() says what the call cannot do without, and
exact() gives the same outputs from a plain torch float64 implementation of the method (_Reference,
which uses none of the package's code).

Sizes are grid levels: `levels` L means N = 2^L cells per side (h = 1/N); L = 5 .. 11 is h = 1/32 ..
1/2048, the range of the package's workloads.
"""
import math

import torch

from paper_1502_04070_gb300.autograd import mass_half_norm2, stokes_solve
from paper_1502_04070_gb300.solver import BatchSolver, Solver
from paper_1502_04070_gb300.timestep import ImplicitEuler

MAX_CYCLES = 300


def listed():
    return [
        # one float64 cycle from zero on a small grid: the preconditioner of a caller's own Krylov loop
        dict(name="cycle_fp64_h32", kind="cycle", levels=5, beta=1.0, precision="fp64", smoother="uzawa", gamma=1, nu=3,
             state="zero"),
        # the same application with float32 cycles on an ordinary grid
        dict(name="cycle_mixed_h256", kind="cycle", levels=8, beta=1e2, precision="mixed", smoother="uzawa", gamma=1, nu=3,
             state="zero"),
        # one float64 cycle on a caller's state, largest grid (the float64 path where arithmetic limits it)
        dict(name="cycle_fp64_h2048", kind="cycle", levels=11, beta=1e4, precision="fp64", smoother="uzawa", gamma=1, nu=3,
             state="given"),
        # the plain float64 solve of a small problem to 1e-10
        dict(name="solve_fp64_h32", kind="solve", levels=5, beta=1.0, precision="fp64", gamma=1, coarse=0, inner=1,
             tol=1e-10, data="random", domain="square"),
        # the largest solve, smooth data, with the options a program tunes for it
        dict(name="solve_mixed_h2048", kind="solve", levels=11, beta=1e4, precision="mixed", gamma=1, coarse=3, inner=2,
             tol=1e-8, data="smooth", domain="square"),
        # W-cycles (the paper's cycle) on a stationary problem
        dict(name="solve_w_mixed_h512", kind="solve", levels=9, beta=0.0, precision="mixed", gamma=2, coarse=3, inner=1,
             tol=1e-8, data="random", domain="square"),
        # the non-convex domain
        dict(name="solve_lshape_mixed_h512", kind="solve", levels=9, beta=1e2, precision="mixed", gamma=1, coarse=1,
             inner=1, tol=1e-8, data="random", domain="lshape"),
        # one right-hand side for several step lengths at once (robustness sweep)
        dict(name="batch_sweep_h512", kind="batch", levels="9,9,9,9,9,9", betas="0,1,1e2,1e4,1e6,1e8", tol=1e-8),
        # many independent solves of uneven size in one launch
        dict(name="batch_uneven", kind="batch", levels="5,9,7,6,8,5,7,9,6,5,8,7,6,9,8,5,7,6,8,9,5,6,7,8",
             betas="3e-2,2e4,5e6,1e1,4e2,9e7,7e-1,6e5,3e3,2e1,8e7,1e4,5e-2,3e7,6e1,1e6,2e3,7e5,4e-1,9e3,1e2,5e7,8e0,2e5",
             tol=1e-8),
        # one step of a parameter fit: solve, loss, gradients of f, g and beta by the adjoint solve
        dict(name="adjoint_h1024", kind="adjoint", levels=10, beta=1e3, tol=1e-8),
        # implicit time steps with changing data, each warm-started from the last
        dict(name="euler_h512", kind="euler", levels=9, dt=1e-3, steps=3, tol=1e-8),
        # set-up of a right-hand side from nodal data and the true residual of a state, largest grid
        dict(name="data_h2048", kind="data", levels=11, beta=1e4),
    ]


def draw(rng):
    def log_beta(lo, hi):
        return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    kind = rng.choice(["cycle", "cycle", "cycle", "solve", "solve", "solve", "batch", "adjoint", "euler", "data"])
    if kind == "cycle":
        prec = rng.choice(["fp64", "mixed"])
        smoother = rng.choice(["uzawa", "uzawa", "normal"])
        return dict(kind=kind, levels=rng.randint(3, 11), beta=log_beta(1e-2, 1e8), precision=prec, smoother=smoother,
                    gamma=rng.choice([1, 1, 2]) if prec == "mixed" else 1, nu=rng.randint(1, 4), state=rng.choice(["zero", "given"]))
    if kind == "solve":
        shape = rng.choice(["square", "square", "square", "lshape"])
        prec = rng.choice(["fp64", "mixed", "mixed", "mixed"])
        beta = log_beta(1e-2, 1e8)
        top = 7 if prec == "fp64" else 9 if (beta < 1e4 or shape == "lshape") else 11
        gamma = rng.choice([1, 1, 2]) if prec == "mixed" and shape == "square" else 1
        if gamma == 2:
            top = min(top, 9)
        return dict(kind=kind, levels=rng.randint(4, top), beta=beta, precision=prec, gamma=gamma,
                    coarse=1 if shape == "lshape" else 3 if gamma == 2 else rng.choice([0, 0, 2, 3]),
                    inner=rng.choice([1, 1, 2]) if prec == "mixed" else 1, tol=1e-8,
                    data=rng.choice(["random", "smooth"]) if shape == "square" else "random", domain=shape)
    if kind == "batch":
        n = rng.randint(2, 24)
        return dict(kind=kind, levels=",".join(str(rng.randint(4, 9)) for _ in range(n)),
                    betas=",".join("%g" % log_beta(1e-2, 1e8) for _ in range(n)), tol=1e-8)
    if kind == "adjoint":
        return dict(kind=kind, levels=rng.randint(4, 10), beta=log_beta(1e2, 1e6), tol=1e-8)
    if kind == "euler":
        return dict(kind=kind, levels=rng.randint(4, 9), dt=log_beta(1e-6, 1e-2), steps=rng.randint(1, 3), tol=1e-8)
    return dict(kind=kind, levels=rng.randint(2, 11), beta=log_beta(1e-2, 1e8))


# ---------------------------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


class _Data:
    """Seeded inputs of a case, in the order they are asked for."""

    def __init__(self, seed):
        self.dev = _device()
        self.gen = torch.Generator(device=self.dev)
        self.gen.manual_seed(1000003 * int(seed) + 17)

    def uniform(self, *shape):
        return 2.0 * torch.rand(*shape, dtype=torch.float64, device=self.dev, generator=self.gen) - 1.0

    def velocity(self, levels, domain="square"):
        """Uniform [-1, 1] values at the velocity unknowns."""
        n = 2 ** levels
        u = self.uniform(2, 2 * n + 1, 2 * n + 1)
        u[:, 0], u[:, -1], u[:, :, 0], u[:, :, -1] = 0.0, 0.0, 0.0, 0.0
        if domain == "lshape":
            u[:, n:, n:] = 0.0
        return u

    def pressure(self, levels, domain="square"):
        n = 2 ** levels
        p = self.uniform(n + 1, n + 1)
        if domain == "lshape":
            p[n // 2 + 1:, n // 2 + 1:] = 0.0
        return p

    def smooth(self, levels, beta):
        """Nodal values of f for u = a curl(sin^2(pi x) sin^2(pi y)), p = a cos(pi x) cos(pi y), a from the seed."""
        n, pi = 2 ** levels, math.pi
        a = 1.0 + 0.5 * self.uniform(1)
        t = torch.arange(2 * n + 1, dtype=torch.float64, device=self.dev) / (2.0 * n)
        x, y = t[None, :], t[:, None]
        sx, sy = torch.sin(pi * x) ** 2, torch.sin(pi * y) ** 2
        s2x, s2y, c2x, c2y = torch.sin(2 * pi * x), torch.sin(2 * pi * y), torch.cos(2 * pi * x), torch.cos(2 * pi * y)
        fx = -2 * pi ** 3 * (c2x - 2 * sx) * s2y + beta * pi * sx * s2y - pi * torch.sin(pi * x) * torch.cos(pi * y)
        fy = 2 * pi ** 3 * s2x * (c2y - 2 * sy) - beta * pi * s2x * sy - pi * torch.cos(pi * x) * torch.sin(pi * y)
        return a * torch.stack([fx, fy])

    def right_hand_side(self, levels, domain="square"):
        """Load vectors of the size that nodal data of order one has, g summing to zero."""
        n = 2 ** levels
        f, g = self.velocity(levels, domain) / n ** 2, self.pressure(levels, domain) / n ** 2
        live = torch.ones_like(g)
        if domain == "lshape":
            live[n // 2 + 1:, n // 2 + 1:] = 0.0
        return f, g - live * (g.sum() / live.sum())

    def solve_data(self, case):
        """(nodal f, nodal g) on the square, load vectors on the L."""
        lv = case["levels"]
        if case["domain"] == "lshape":
            return self.right_hand_side(lv, "lshape")
        if case["data"] == "smooth":
            f = self.smooth(lv, case["beta"])
            return f, torch.zeros(2 ** lv + 1, 2 ** lv + 1, dtype=torch.float64, device=self.dev)
        return self.velocity(lv), self.pressure(lv)


def _batch(case):
    return [int(v) for v in case["levels"].split(",")], [float(b) for b in case["betas"].split(",")]


def prepare(case, seed):
    d, kind, lv = _Data(seed), case["kind"], case["levels"]
    st = dict(case=case)
    if kind == "cycle":
        st["S"] = Solver(lv, case["beta"], precision=case["precision"], smoother=case["smoother"], gamma=case["gamma"],
                         nu_pre=case["nu"], nu_post=case["nu"])
        st["f"], st["g"] = d.right_hand_side(lv)
        if case["state"] == "given":
            st["u"], st["p"] = d.velocity(lv), d.pressure(lv)
    elif kind == "solve":
        S = Solver(lv, case["beta"], precision=case["precision"], gamma=case["gamma"], coarse_level=case["coarse"],
                   inner_cycles=case["inner"], domain=case["domain"])
        S.autotune()
        f, g = d.solve_data(case)
        if case["domain"] == "square":
            f, g = S.load_vectors(f, g, project_g=True)
        st.update(S=S, f=f, g=g)
    elif kind == "batch":
        levels, betas = _batch(case)
        st["B"] = BatchSolver(levels, betas, precision="mixed")
        rhs = [d.right_hand_side(l) for l in levels]
        st["fs"], st["gs"] = [f for f, _ in rhs], [g for _, g in rhs]
    elif kind == "adjoint":
        st["S"] = Solver(lv, case["beta"], precision="mixed")
        st["S"].autotune()
        f, g = d.right_hand_side(lv)
        st["f"], st["g"] = f.requires_grad_(), g.requires_grad_()
        st["beta"] = torch.tensor(case["beta"], dtype=torch.float64, device=d.dev, requires_grad=True)
        st["target"] = d.velocity(lv)
    elif kind == "euler":
        st["E"] = ImplicitEuler(lv, case["dt"], precision="mixed", tol=case["tol"], max_cycles=MAX_CYCLES)
        st["E"].solver.autotune()
        st["u"], st["p"] = d.velocity(lv), torch.zeros(2 ** lv + 1, 2 ** lv + 1, dtype=torch.float64, device=d.dev)
        st["forcing"] = [(d.velocity(lv), d.pressure(lv)) for _ in range(case["steps"])]
    else:
        st["S"] = Solver(lv, case["beta"])
        st["f"], st["g"] = d.velocity(lv), d.pressure(lv)
        st["u"], st["p"] = d.velocity(lv), d.pressure(lv)
    return st


# ------------------------------------------------------------------------------------------- run
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "cycle":
        S = st["S"]
        u, p = (st["u"].clone(), st["p"].clone()) if case["state"] == "given" else (S.zeros_u(), S.zeros_p())
        return S.cycle(u, p, st["f"], st["g"])
    if kind == "solve":
        u, p, _ = st["S"].solve(st["f"], st["g"], tol=case["tol"], max_cycles=MAX_CYCLES)
        return u, p
    if kind == "batch":
        us, ps, _, _, _ = st["B"].solve(st["fs"], st["gs"], tol=case["tol"], max_cycles=MAX_CYCLES)
        return us + ps
    if kind == "adjoint":
        S = st["S"]
        u, p = stokes_solve(st["f"], st["g"], st["beta"], S, tol=case["tol"], max_cycles=MAX_CYCLES)
        loss = mass_half_norm2(u - st["target"], S)
        grads = torch.autograd.grad(loss, (st["f"], st["g"], st["beta"]))
        return (loss.detach(), u.detach(), p.detach()) + tuple(grads)
    if kind == "euler":
        u, p = st["u"].clone(), st["p"].clone()
        for f, g in st["forcing"]:
            st["E"].step(u, p, f, g)
        return u, p
    f, g = st["S"].load_vectors(st["f"], st["g"], project_g=True)
    ru, rp = st["S"].residual(st["u"], st["p"], f, g)
    return f, g, ru, rp


# ------------------------------------------------------------------------------------------ work
def _unknowns(levels, domain="square"):
    n = 2 ** levels
    return 9 * n * n * (0.75 if domain == "lshape" else 1.0)


def work(case):
    """Bytes and operations of one pass.  A smoothing step on a level reads the state, the right-hand
    side and the inverse Schur diagonal and writes the state once (28 values per cell) and takes about
    340 operations per cell; a cycle has 2 nu + 2 such passes (the defect and the transfers count as
    two), the coarser levels add a third (V) or as much again (W).  The iteration counts are those of a
    contraction by 0.35 per cycle (about what the method reaches)."""
    kind, lv = case["kind"], case["levels"]

    def cycles(l, count, width, gamma=1, nu=3, domain="square"):
        cells = _unknowns(l, domain) / 9
        levels_sum = 4.0 / 3.0 if gamma == 1 else 2.0
        return count * (2 * nu + 2) * levels_sum * 28 * cells * width, count * (2 * nu + 2) * levels_sum * 340 * cells

    def to_tol(tol):
        return math.ceil(math.log(tol) / math.log(0.35))

    if kind == "data":   # two vectors in, two out, twice
        return dict(bytes=6 * 8 * _unknowns(lv), flops=2 * 340 * _unknowns(lv) / 9)
    if kind == "cycle":
        b, f = cycles(lv, 1, 4 if case["precision"] == "mixed" else 8, case["gamma"], case["nu"])
        return dict(bytes=b, flops=f)
    if kind == "solve":
        b, f = cycles(lv, to_tol(case["tol"]), 4 if case["precision"] == "mixed" else 8, case["gamma"], 3, case["domain"])
        return dict(bytes=b, flops=f)
    if kind == "batch":
        w = [cycles(l, to_tol(case["tol"]), 4) for l in _batch(case)[0]]
        return dict(bytes=sum(x for x, _ in w), flops=sum(y for _, y in w))
    solves = 2 if kind == "adjoint" else case["steps"]
    b, f = cycles(lv, solves * to_tol(case["tol"]), 4)
    return dict(bytes=b, flops=f)


# ----------------------------------------------------------------------------------------- exact
def _triangles(o):
    """The two triangles of a square of side 2 (lattice units) of orientation o: 0 is cut from (0, 0) to
    (2, 2), 1 from (2, 0) to (0, 2)."""
    if o == 0:
        return [[(0, 0), (2, 0), (2, 2)], [(0, 0), (2, 2), (0, 2)]]
    return [[(0, 0), (2, 0), (0, 2)], [(2, 0), (2, 2), (0, 2)]]


def _bary(tri, x, y):
    (x0, y0), (x1, y1), (x2, y2) = tri
    det = (x1 - x0) * (y2 - y0) - (x2 - x0) * (y1 - y0)
    l1 = ((x - x0) * (y2 - y0) - (x2 - x0) * (y - y0)) / det
    l2 = ((x1 - x0) * (y - y0) - (x - x0) * (y1 - y0)) / det
    g1, g2 = ((y2 - y0) / det, -(x2 - x0) / det), (-(y1 - y0) / det, (x1 - x0) / det)
    g0 = (-g1[0] - g2[0], -g1[1] - g2[1])
    return (1.0 - l1 - l2, l1, l2), (g0, g1, g2), abs(det) / 2.0


def _p2(tri, x, y):
    """{square-local node: (value, d/dx, d/dy)} of the triangle's six quadratic basis functions at (x, y)."""
    l, g, _ = _bary(tri, x, y)
    out = {}
    for i in range(3):
        px, py = tri[i]
        out[3 * py + px] = (l[i] * (2 * l[i] - 1),) + tuple((4 * l[i] - 1) * g[i][c] for c in (0, 1))
        j, k = (i + 1) % 3, (i + 2) % 3
        mx, my = (tri[j][0] + tri[k][0]) // 2, (tri[j][1] + tri[k][1]) // 2
        out[3 * my + mx] = (4 * l[j] * l[k],) + tuple(4 * (l[j] * g[k][c] + l[k] * g[j][c]) for c in (0, 1))
    return out


def _p1(tri, x, y):
    l, _, _ = _bary(tri, x, y)
    return {(tri[i][1] // 2) * 2 + tri[i][0] // 2: l[i] for i in range(3)}


def _rule():
    """Degree-4 rule on a triangle: barycentric points and weights (sum 1)."""
    out = []
    for a, w in ((0.44594849091596488632, 0.22338158967801146570), (0.09157621350977074346, 0.10995174365532186764)):
        b = 1.0 - 2.0 * a
        out += [((a, a, b), w), ((a, b, a), w), ((b, a, a), w)]
    return out


def _square_matrices(o):
    """Stiffness, mass (9 x 9), divergence (x over y, 4 x 9 each) and pressure mass (4 x 4) of the unit square."""
    K, M = torch.zeros(9, 9, dtype=torch.float64), torch.zeros(9, 9, dtype=torch.float64)
    B, MP = torch.zeros(2, 4, 9, dtype=torch.float64), torch.zeros(4, 4, dtype=torch.float64)
    for tri in _triangles(o):
        for bc, w in _rule():
            x = sum(bc[i] * tri[i][0] for i in range(3))
            y = sum(bc[i] * tri[i][1] for i in range(3))
            w = w * 0.5                    # area of a triangle of the unit square
            v, q = _p2(tri, x, y), _p1(tri, x, y)
            for a, (va, ax, ay) in v.items():
                for b, (vb, bx, by) in v.items():
                    K[a, b] += w * 4.0 * (ax * bx + ay * by)   # lattice unit = half the side
                    M[a, b] += w * va * vb
                for r, s in q.items():
                    B[0, r, a] += w * 2.0 * ax * s
                    B[1, r, a] += w * 2.0 * ay * s
            for r, s in q.items():
                for t, z in q.items():
                    MP[r, t] += w * s * z
    return K, M, B.reshape(8, 9), MP


def _embedding(o):
    """Coarse basis of a square at the 5 x 5 fine lattice points (25 x 9) and the 3 x 3 fine vertices (9 x 4)."""
    W2, W1 = torch.zeros(25, 9, dtype=torch.float64), torch.zeros(9, 4, dtype=torch.float64)

    def home(x, y):
        return next(t for t in _triangles(o) if min(_bary(t, x, y)[0]) >= -1e-12)

    for b in range(5):
        for a in range(5):
            x, y = a / 2.0, b / 2.0
            for m, v in _p2(home(x, y), x, y).items():
                W2[5 * b + a, m] = v[0]
            if a % 2 == 0 and b % 2 == 0:
                for r, s in _p1(home(x, y), x, y).items():
                    W1[3 * (b // 2) + a // 2, r] = s
    return W2, W1


class _Level:
    """One grid level: operator, diagonals and transfers to the level above, square by square."""

    def __init__(self, n, beta, lshape, dev, tables):
        self.n, self.dev, self.lshape = n, dev, lshape
        h, hf = 1.0 / n, n // 2
        left = torch.arange(n, device=dev) < hf
        self.other = left[:, None] != left[None, :]                  # squares of orientation 1
        self.kept = ~(~left[:, None] & ~left[None, :]) if lshape else None   # squares of the domain
        K, M, B, MP, W2, W1 = [torch.cat([a, b]).to(dev) for a, b in zip(*tables)]   # both orientations, stacked
        self.A, self.M, self.MP, self.W2, self.W1 = K + beta * h * h * M, h * h * M, h * h * MP, W2, W1
        self.B = [h * torch.cat([B[4 * c:4 * c + 4], B[8 + 4 * c:12 + 4 * c]]) for c in (0, 1)]   # x, y divergence
        self.BT = torch.cat([h * torch.cat([b[:4].t(), b[4:].t()]) for b in (B[:8], B[8:])])
        self.W2T, self.W1T = [torch.cat([w[:len(w) // 2].t(), w[len(w) // 2:].t()]) for w in (W2, W1)]
        self.mu = torch.zeros(2 * n + 1, 2 * n + 1, dtype=torch.float64, device=dev)
        self.mu[1:-1, 1:-1] = 1.0
        self.mp = torch.ones(n + 1, n + 1, dtype=torch.float64, device=dev)
        if lshape:
            self.mu[n:, n:] = 0.0
            self.mp[hf + 1:, hf + 1:] = 0.0
        diag = torch.cat([torch.diagonal(self.A[:9]), torch.diagonal(self.A[9:])]).reshape(18, 1)
        d = self._put(self._pick(diag.expand(18, n * n)), 2, 3)[0]
        self.dinv = torch.where(self.mu > 0, 1.0 / d.clamp_min(1e-300), torch.zeros_like(d))
        # diag(B Ahat^-1 B^T): the patches of vertices three cells apart do not meet
        s = torch.zeros_like(self.mp)
        for a in range(3):
            for b in range(3):
                e = torch.zeros_like(self.mp)
                e[b::3, a::3] = 1.0
                s += e * self.b(self.dinv * self.bt(e * self.mp))
        self.sinv = torch.where(self.mp > 0, 1.0 / s.clamp_min(1e-300), torch.zeros_like(s))
        self.w = self.mass_p(torch.ones_like(self.mp)) * self.mp

    # square-local values: entry k of a square is at offset (k // m, k % m) from `step` times its corner
    @staticmethod
    def _get(x, step, m):
        return torch.nn.functional.unfold(x[None, None], m, stride=step)[0]

    def _put(self, v, step, m):
        size = step * (self.n - 1) + m
        return torch.nn.functional.fold(v[None], (size, size), m, stride=step)[0]

    def _pick(self, v):
        """Of the products with both orientations' matrices, each square's own."""
        k = v.shape[0] // 2
        v = torch.where(self.other.reshape(1, -1), v[k:], v[:k])
        return v if self.kept is None else v * self.kept.reshape(1, -1)

    def _rows(self, u, mats):
        return torch.cat([self._put(self._pick(mats @ self._get(c, 2, 3)), 2, 3) for c in u])

    def a(self, u):
        return self._rows(u * self.mu, self.A) * self.mu

    def mass_u(self, u):
        return self._rows(u, self.M) * self.mu

    def mass_p(self, p):
        return self._put(self._pick(self.MP @ self._get(p, 1, 2)), 1, 2)[0]

    def b(self, u):
        u = u * self.mu
        v = self.B[0] @ self._get(u[0], 2, 3) + self.B[1] @ self._get(u[1], 2, 3)
        return self._put(self._pick(v), 1, 2)[0] * self.mp

    def bt(self, p):
        return self._put(self._pick(self.BT @ self._get(p * self.mp, 1, 2)), 2, 3) * self.mu

    def dense(self):
        """A and the two divergence blocks as matrices over all lattice nodes and vertices."""
        def ids(x, m, step):
            k = torch.arange(x.numel(), dtype=torch.float64, device=self.dev).reshape(x.shape)
            return self._get(k, step, m).long()

        def matrix(rows, cols, size, mats):
            h = mats.shape[0] // 2
            v = torch.where(self.other.reshape(1, 1, -1), mats[h:, :, None], mats[:h, :, None])
            v = v if self.kept is None else v * self.kept.reshape(1, 1, -1)
            out = torch.zeros(size, dtype=torch.float64, device=self.dev)
            r, c = torch.broadcast_tensors(rows[:, None], cols[None])
            return out.index_put((r, c), v, accumulate=True)

        nu, np_ = ids(self.mu, 3, 2), ids(self.mp, 2, 1)
        size_u, size_p = self.mu.numel(), self.mp.numel()
        return (matrix(nu, nu, (size_u, size_u), self.A),) + tuple(matrix(np_, nu, (size_p, size_u), b) for b in self.B)

    def residual(self, u, p, f, g):
        return f * self.mu - self.a(u) - self.bt(p), (g - self.b(u)) * self.mp

    def uzawa(self, u, p, f, g, tau=0.8, sigma=0.8):
        uh = u + tau * self.dinv * (f * self.mu - self.a(u) - self.bt(p))
        dp = sigma * self.sinv * (self.b(uh) - g)
        return uh - tau * self.dinv * self.bt(dp), p + dp

    def normal(self, u, p, f, g, tau=0.35):
        ru, rp = self.residual(u, p, f, g)
        zu, zp = ru * self.dinv, rp * self.sinv
        return u + tau * self.dinv * (self.a(zu) + self.bt(zp)), p + tau * self.sinv * self.b(zu)

    def centre(self, p):
        return p - self.mp * ((self.w * p).sum() / self.w.sum())

    # canonical embedding of this (coarse) level into the next and its transpose
    def _counts(self):
        if not hasattr(self, "_cnt"):
            one = torch.ones(50, self.n ** 2, dtype=torch.float64, device=self.dev)
            self._cnt = tuple(1.0 / self._put(self._pick(one[:2 * m * m]), s, m)[0].clamp_min(1.0) for s, m in ((4, 5), (2, 3)))
        return self._cnt

    def prolong(self, u, p):
        cu, cp = self._counts()
        fu = torch.cat([self._put(self._pick(self.W2 @ self._get(c, 2, 3)), 4, 5) for c in u])
        return fu * cu, self._put(self._pick(self.W1 @ self._get(p, 1, 2)), 2, 3)[0] * cp

    def restrict(self, fu, fp):
        cu, cp = self._counts()
        u = torch.cat([self._put(self._pick(self.W2T @ self._get(c * cu, 4, 5)), 2, 3) for c in fu])
        p = self._put(self._pick(self.W1T @ self._get(fp * cp, 2, 3)), 1, 2)[0]
        return u * self.mu, p * self.mp


class _Reference:
    """The coupled multigrid method in plain float64; the exact coarsest solve is on level `low`."""

    def __init__(self, levels, beta, domain="square", smoother="uzawa", gamma=1, nu=3, low=None):
        dev, lshape = _device(), domain == "lshape"
        tables = [_square_matrices(o) + _embedding(o) for o in (0, 1)]
        self.low = min(3, levels - 1) if low is None else low
        self.L = [_Level(2 ** (k + 1), beta, lshape, dev, tables) if k >= self.low else None for k in range(levels)]
        self.step = "normal" if smoother == "normal" else "uzawa"
        self.gamma, self.nu = gamma, nu
        Z = self.L[self.low]
        iu, ip = [torch.nonzero(m.reshape(-1)).reshape(-1) for m in (Z.mu, Z.mp)]
        iu = torch.cat([iu, iu + Z.mu.numel()])
        nu_, np_ = len(iu), len(ip)
        A, Bx, By = Z.dense()
        zero = torch.zeros_like(A)
        mat = torch.zeros(nu_ + np_ + 1, nu_ + np_ + 1, dtype=torch.float64, device=dev)
        mat[:nu_, :nu_] = torch.cat([torch.cat([A, zero], 1), torch.cat([zero, A], 1)])[iu][:, iu]
        mat[nu_:-1, :nu_] = torch.cat([Bx, By], 1)[ip][:, iu]
        mat[:nu_, nu_:-1] = mat[nu_:-1, :nu_].t()
        mat[nu_:-1, -1] = mat[-1, nu_:-1] = Z.w.reshape(-1)[ip]
        self.inv, self.iu, self.ip = torch.linalg.inv(mat), iu, ip

    def _coarse(self, f, g):
        Z = self.L[self.low]
        rhs = torch.cat([f.reshape(-1)[self.iu], g.reshape(-1)[self.ip], torch.zeros(1, dtype=f.dtype, device=f.device)])
        x = self.inv @ rhs
        u, p = torch.zeros_like(f).reshape(-1), torch.zeros_like(g).reshape(-1)
        u[self.iu], p[self.ip] = x[:len(self.iu)], x[len(self.iu):-1]
        return u.reshape((2,) + Z.mu.shape), p.reshape(Z.mp.shape)

    def _visit(self, k, u, p, f, g):
        if k == self.low:
            return self._coarse(f, g)
        V, C = self.L[k], self.L[k - 1]
        for _ in range(self.nu):
            u, p = getattr(V, self.step)(u, p, f, g)
        fc, gc = C.restrict(*V.residual(u, p, f, g))
        uc, pc = torch.zeros_like(fc), torch.zeros_like(gc)
        for _ in range(self.gamma):
            uc, pc = self._visit(k - 1, uc, pc, fc, gc)
        du, dp = C.prolong(uc, pc)
        u, p = u + du * V.mu, p + dp * V.mp
        for _ in range(self.nu):
            u, p = getattr(V, self.step)(u, p, f, g)
        return u, p

    def cycle(self, u, p, f, g):
        top = self.L[-1]
        u, p = self._visit(len(self.L) - 1, u, p, f, g)
        return u, top.centre(p)

    def load(self, f, g):
        top = self.L[-1]
        g = g - (top.w * g).sum() / top.w.sum()
        return top.mass_u(f), top.mass_p(g)

    def _norm(self, u, p):
        return float(torch.sqrt((u * u).sum() + (p * p).sum()))

    def solve(self, f, g):
        """To the accuracy of the arithmetic: cycles from zero, each combined with the earlier ones by least
        squares on the residual (GCR), then, where these stall above 1e-13, cycles on the residual alone."""
        top = self.L[-1]
        u, p = torch.zeros_like(f), torch.zeros_like(g)
        goal = 1e-13 * self._norm(f, g)
        for combine, patience in ((True, 6), (False, 5)):
            best, since, past = math.inf, 0, []
            for _ in range(200):
                ru, rp = top.residual(u, p, f, g)
                r = self._norm(ru, rp)
                best, since = (r, 0) if r < 0.5 * best else (best, since + 1)
                if r <= goal or since >= patience:
                    break
                zu, zp = self.cycle(torch.zeros_like(u), torch.zeros_like(p), ru, rp)
                c = 1.0
                if combine:
                    qu, qp = top.a(zu) + top.bt(zp), top.b(zu)
                    for yu, yp, su, sp in past:
                        c = (qu * su).sum() + (qp * sp).sum()
                        zu, zp, qu, qp = zu - c * yu, zp - c * yp, qu - c * su, qp - c * sp
                    q = 1.0 / torch.sqrt((qu * qu).sum() + (qp * qp).sum())
                    zu, zp, qu, qp = q * zu, q * zp, q * qu, q * qp
                    past = past[-19:] + [(zu, zp, qu, qp)]
                    c = (ru * qu).sum() + (rp * qp).sum()
                u, p = u + c * zu, top.centre(p + c * zp)
        return u, p


def exact(case, seed):
    d, kind, lv = _Data(seed), case["kind"], case["levels"]
    if kind == "cycle":
        R = _Reference(lv, case["beta"], "square", case["smoother"], case["gamma"], case["nu"], low=0)
        f, g = d.right_hand_side(lv)
        x = (d.velocity(lv), d.pressure(lv)) if case["state"] == "given" else (torch.zeros_like(f), torch.zeros_like(g))
        return R.cycle(*x, f, g)
    if kind == "solve":
        R = _Reference(lv, case["beta"], case["domain"])
        f, g = d.solve_data(case)
        return R.solve(*(R.load(f, g) if case["domain"] == "square" else (f, g)))
    if kind == "batch":
        levels, betas = _batch(case)
        rhs = [d.right_hand_side(l) for l in levels]
        sols = [_Reference(l, b).solve(f, g) for l, b, (f, g) in zip(levels, betas, rhs)]
        return [u for u, _ in sols] + [p for _, p in sols]
    if kind == "adjoint":
        R = _Reference(lv, case["beta"])
        f, g = d.right_hand_side(lv)
        target = d.velocity(lv)
        top = R.L[-1]
        u, p = R.solve(f, g)
        m = top.mass_u(u - target)
        loss = 0.5 * ((u - target) * m).sum()
        lu, lp = R.solve(m, torch.zeros_like(g))
        return loss, u, p, lu, lp, -(lu * top.mass_u(u)).sum()
    if kind == "euler":
        beta = 1.0 / case["dt"]
        R = _Reference(lv, beta)
        u = d.velocity(lv)
        p = None
        for f, g in [(d.velocity(lv), d.pressure(lv)) for _ in range(case["steps"])]:
            u, p = R.solve(*R.load(f + beta * u, g))
        return u, p
    R = _Reference(lv, case["beta"])
    f, g = R.load(d.velocity(lv), d.pressure(lv))
    return (f, g) + R.L[-1].residual(d.velocity(lv), d.pressure(lv), f, g)
