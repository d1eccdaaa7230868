"""Performance cases of the library's public entry points.

Every case is one call (or one solve) as a user's program makes it through
``paper_2510_00998_gb300.dgmg``: the operator, residual and smoothing calls, the V-cycle
as a preconditioner, whole solves in FP64 and mixed precision, and a batch of
independent solves. Sizes are those of the repository's workloads: the 2D meshes
9^2 .. 243^2 and 729^2 of the paper's tables, the 32^3 p = 3 and 64^3 p = 4
workloads, batches with n in 8..24 and p in 2..4, requests with n in 8..48 and p
in 2..5, with unequal and odd axes.

``exact`` restates the discretisation (SIPG on tensor-product Lagrange elements, the
block-Jacobi smoother, the hp V-cycle, conjugate gradients) in plain torch FP64.
"""
import math

import numpy as np
import torch

from paper_2510_00998_gb300 import dgmg

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64

# every key a case may carry, with its default
DEFAULTS = dict(n2=0, kappa="one", mixed=0, basis=0, interior=0, gradual=0, coarsening=2, nu=2, steps=0,
                mgmult=0, rtol=1e-10, autotune=0, count=0)


def _case(name, op, n, p, **kw):
    c = dict(name=name, op=op, n0=n[0], n1=n[1], p=p)
    if len(n) == 3:
        c["n2"] = n[2]
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: the V-cycle of the 16^2, p = 2 workload as a preconditioner of
        # somebody's own Krylov loop; launches and latency count
        _case("vcycle_2d_16_p2", "vcycle", (16, 16), 2),
        # the paper's Tables 3-4: MGMult cycles to 1e-7 on a factor-3 hierarchy, nu = 4
        _case("mgmult_2d_81_p4", "solve", (81, 81), 4, mgmult=1, coarsening=3, nu=4, rtol=1e-7),
        # the paper's Table 6: block-Jacobi smoothing steps on the 729^2 mesh
        _case("smooth_2d_729_p4", "smooth", (729, 729), 4, steps=4),
        # a residual check at the highest degree, Gauss-Legendre basis, odd axes
        _case("residual_2d_243_p6_gl", "residual", (243, 241), 6, basis=1, kappa="lognormal"),
        # a preconditioner call on a middling ragged 3D mesh of low degree
        _case("vcycle_3d_23_p2", "vcycle", (23, 17, 20), 2, kappa="lognormal"),
        # smoothing steps alone at the degree of the main workload, ragged mesh
        _case("smooth_3d_32_p3", "smooth", (33, 31, 32), 3, kappa="lognormal", steps=4),
        # the FP64 operator on the large mesh: a user's own outer iteration
        _case("apply_3d_64_p4", "apply", (64, 60, 57), 4, kappa="lognormal"),
        # the same operator in FP32 (mixed-precision contexts)
        _case("apply_f32_3d_64_p4", "apply_f32", (63, 64, 61), 4, kappa="lognormal", mixed=1),
        # the main workload: FP64 conjugate gradients with the V-cycle, 32^3, p = 3
        _case("solve_3d_32_p3", "solve", (32, 32, 32), 3, autotune=1),
        # the large workload: mixed-precision solve with a rough coefficient
        _case("solve_mixed_3d_64_p4", "solve", (64, 64, 64), 4, kappa="lognormal", mixed=1, autotune=1),
        # a request of the serving range at its highest degree, gradual p-hierarchy
        _case("solve_3d_17_p5_gradual", "solve", (17, 18, 16), 5, kappa="two-phase", gradual=1),
        # independent solves of unequal size sharing launches (mixed precision)
        _case("batch_mixed_24", "batch", (0, 0), 0, mixed=1, kappa="lognormal", count=24, autotune=1),
    ]


def _ndof(c):
    n = [c["n0"], c["n1"]] + ([c["n2"]] if c["n2"] else [])
    return int(np.prod(n)) * (c["p"] + 1) ** len(n)


def _around(rng, lo, hi, d, spread=0.15):
    m = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return [max(lo, min(hi, round(m * math.exp(rng.uniform(-spread, spread))))) for _ in range(d)]


def draw(rng):
    op = rng.choice(["vcycle", "smooth", "apply", "residual", "apply_f32", "solve", "solve", "solve_mixed", "batch"])
    kappa = rng.choice(["one", "lognormal", "two-phase"])
    if op == "batch":
        mixed = rng.choice([0, 1, 1])
        return dict(op="batch", n0=0, n1=0, p=0, mixed=mixed, kappa="lognormal",
                    count=rng.randint(3, 16 if mixed else 6), autotune=rng.choice([0, 1]), salt=rng.randint(0, 999))
    dim = rng.choice([2, 3, 3]) if op in ("vcycle", "smooth", "apply", "residual", "solve") else 3
    # unknowns of the largest mesh of each kind (the listed ones' range)
    most = {"solve": 1.5e6, "solve_mixed": 1.5e7, "vcycle": 8e6}.get(op, 3.0e7)
    while True:
        if dim == 2:
            c = dict(op=op, p=rng.randint(1, 6))
            c["n0"], c["n1"] = _around(rng, 9, 243 if op == "solve" else 729, 2)
        else:
            c = dict(op=op, p=rng.randint(1, 5))
            c["n0"], c["n1"], c["n2"] = _around(rng, 8, 64, 3)
        if _ndof({**DEFAULTS, **c}) <= most:
            break
    c["kappa"] = kappa
    if op in ("solve_mixed", "apply_f32"):
        c["mixed"] = 1
    if op == "solve_mixed":
        c["op"] = "solve"
    if op == "smooth":
        c["steps"] = rng.randint(1, 6)
    if op in ("apply", "residual", "smooth", "apply_f32") and rng.random() < 0.2:
        c["basis"] = 1
    if op == "solve":
        if dim == 2 and rng.random() < 0.4:
            c.update(mgmult=1, coarsening=3, nu=4, rtol=1e-7, p=min(c["p"], 4), kappa="one")
        elif rng.random() < 0.2:
            c["gradual"] = 1
        c["autotune"] = rng.choice([0, 1])
    return c


# ------------------------------------------------------------------- inputs
def _full(case):
    c = {**DEFAULTS, **case}
    c["n"] = (c["n0"], c["n1"]) + ((c["n2"],) if c["n2"] else ())
    return c


def _kappa(kind, n, rng):
    """One coefficient per cell, x fastest: 1, lognormal(0, 1), or 1 / 100 on the two
    sides of a plane."""
    if kind == "one":
        return None
    if kind == "lognormal":
        return np.exp(rng.normal(size=int(np.prod(n))))
    g = np.meshgrid(*[(np.arange(v) + 0.5) / v - 0.5 for v in n[::-1]], indexing="ij")
    w = rng.normal(size=len(n))
    s = sum(a * b for a, b in zip(w / np.linalg.norm(w), g)) + rng.uniform(-0.2, 0.2)
    return np.where(s.reshape(-1) > 0, 100.0, 1.0)


def _modes(rng, d):
    return rng.normal(size=8), rng.integers(1, 5, size=(8, d))


def _separable(parts):
    """sum_m of the outer products of parts[a][m, cell * node] (axis a), as a vector
    [cell][node], x fastest in both."""
    d = len(parts)
    n = [p.shape[1] for p in parts]
    q = [p.shape[2] for p in parts]
    flat = [p.reshape(p.shape[0], -1) for p in parts]
    if d == 2:
        t = torch.einsum("my,mx->yx", flat[1], flat[0]).view(n[1], q[1], n[0], q[0]).permute(0, 2, 1, 3)
    else:
        t = torch.einsum("mz,my,mx->zyx", flat[2], flat[1], flat[0])
        t = t.view(n[2], q[2], n[1], q[1], n[0], q[0]).permute(0, 2, 4, 1, 3, 5)
    return t.reshape(-1).contiguous()


def _field(E, coeffs, waves, dev):
    """sum_m a_m prod_a sin(k pi x_a) at the nodes."""
    parts = []
    for a, n in enumerate(E.n):
        x = (np.arange(n)[:, None] + (E.nodes[None, :] + 1) / 2) / n
        s = np.sin(np.pi * waves[:, a, None, None] * x[None])
        parts.append(torch.tensor(s * coeffs[:, None, None] if a == 0 else s, dtype=F64, device=dev))
    return _separable(parts)


def _load(E, coeffs, waves, dev):
    """b_i = (f, phi_i), f = sum_m a_m prod_a sin(k pi x_a), by (p+2)-point Gauss."""
    xg, wg = np.polynomial.legendre.leggauss(E.q + 1)
    V = _lagrange(E.nodes, xg)[0]                                  # [point, node]
    parts = []
    for a, n in enumerate(E.n):
        x = (np.arange(n)[:, None] + (xg[None, :] + 1) / 2) / n
        s = np.sin(np.pi * waves[:, a, None, None] * x[None]) @ (V * (wg * 0.5 / n)[:, None])
        parts.append(torch.tensor(s * coeffs[:, None, None] if a == 0 else s, dtype=F64, device=dev))
    return _separable(parts)


def _problem(c, seed, dev=DEV):
    """The inputs of one mesh from the seed: element data, kappa, and u / b as the call needs them."""
    rng = np.random.default_rng(seed)
    kappa = _kappa(c["kappa"], c["n"], rng)
    E = Element(c["n"], c["p"], c["basis"])
    b = _load(E, *_modes(rng, len(c["n"])), dev)
    u = None
    if c["op"] in ("smooth", "apply", "residual", "apply_f32"):
        u = _field(E, *_modes(rng, len(c["n"])), dev)              # a smooth iterate with a rough error
        g = torch.Generator(device=dev).manual_seed(seed)
        u = u + 0.1 * torch.randn(u.shape, dtype=F64, device=dev, generator=g)
        if c["op"] == "apply_f32":
            u = u.float()
    return E, kappa, b, u


def _batch_problems(c, seed):
    rng = np.random.default_rng(seed)
    size = np.random.default_rng(c.get("salt", 0) + 4)             # sizes belong to the case
    out = []
    for _ in range(c["count"]):
        n, p = int(size.integers(8, 25)), int(size.integers(2, 5))
        kappa = _kappa(c["kappa"], (n, n, n), rng)
        out.append((Element((n, n, n), p, 0), kappa, _modes(rng, 3)))
    return out


def _opts(c):
    o = dict(precision=c["mixed"], basis=c["basis"], block_inverse=c["interior"], p_coarsening=c["gradual"],
             coarsening=c["coarsening"], nu_pre=c["nu"], nu_post=c["nu"], rtol=c["rtol"], autotune=c["autotune"],
             maxit=400)
    if c["mgmult"]:
        o["outer"] = dgmg.DGMG_OUTER_MGMULT
    return o


def prepare(case, seed):
    c = _full(case)
    if c["op"] == "batch":
        probs = _batch_problems(c, seed)
        batch = dgmg.Batch([(E.n, E.p, k) for E, k, _ in probs], **{k: _opts(c)[k] for k in
                                                                    ("precision", "autotune", "rtol", "maxit")})
        bs = [_load(E, *m, DEV) for E, _, m in probs]
        return dict(op="batch", batch=batch, b=bs, x=[torch.zeros_like(b) for b in bs])
    E, kappa, b, u = _problem(c, seed)
    ctx = dgmg.Context(c["n"], c["p"], kappa, **_opts(c))
    return dict(op=c["op"], ctx=ctx, b=b, u=u, out=torch.empty_like(b if u is None else u), steps=c["steps"])


def run(s):
    op = s["op"]
    if op == "batch":
        for x in s["x"]:
            x.zero_()
        s["batch"].solve(s["b"], s["x"])
        return s["x"]
    ctx, out = s["ctx"], s["out"]
    if op == "vcycle":
        ctx.vcycle(s["b"], out)
    elif op == "smooth":
        ctx.smooth(s["u"], s["b"], s["steps"])
        return s["u"]
    elif op == "apply":
        ctx.apply(s["u"], out)
    elif op == "residual":
        ctx.residual(s["u"], s["b"], out)
    elif op == "apply_f32":
        ctx.apply_f32(s["u"], out)
    else:
        out.zero_()
        ctx.solve(s["b"], out)
    return out


def work(case):
    """Inputs read once, outputs written once; 10 d (p + 1) operations per unknown for one
    sum-factorised application of the operator or one smoothing step, five of them in a
    V(2,2) cycle and six in an iteration of a solve, whose number is taken as 6 p (direct
    coarsening to Q1) or 5 + 3 p (gradual)."""
    c = _full(case)
    if c["op"] == "batch":
        each = [_work(_full(dict(op="solve", n0=E.n[0], n1=E.n[1], n2=E.n[2], p=E.p))) for E, _, _ in
                _batch_problems(c, 0)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    return _work(c)


def _work(c):
    d, q, nd = len(c["n"]), c["p"] + 1, _ndof(c)
    cells = nd // q ** d
    one = 10.0 * d * q * nd
    item = 4 if c["op"] == "apply_f32" else 8
    vectors = {"smooth": 3, "residual": 3}.get(c["op"], 2)
    times = {"smooth": c["steps"], "vcycle": 2 * c["nu"] + 1,
             "solve": (2 * c["nu"] + 2) * ((5 + 3 * c["p"]) if c["gradual"] else 6 * c["p"])}.get(c["op"], 1)
    return {"bytes": float(item * (vectors * nd + cells)), "flops": one * times}


# -------------------------------------------------- the method in plain FP64
def _lagrange(nodes, x):
    """Values and derivatives [point, node] of the Lagrange basis on `nodes` at x."""
    q = len(nodes)
    v, dv = np.ones((len(x), q)), np.zeros((len(x), q))
    for j in range(q):
        others = [m for m in range(q) if m != j]
        for m in others:
            v[:, j] *= (x - nodes[m]) / (nodes[j] - nodes[m])
        for m in others:
            t = np.full(len(x), 1.0 / (nodes[j] - nodes[m]))
            for k in others:
                if k != m:
                    t *= (x - nodes[k]) / (nodes[j] - nodes[k])
            dv[:, j] += t
    return v, dv


class Element:
    """1D data on a mesh of n cells per axis, degree p: GLL (0) or Gauss (1) nodes."""

    def __init__(self, n, p, basis):
        self.n, self.p, self.q = tuple(n), p, p + 1
        xg, wg = np.polynomial.legendre.leggauss(p + 1)
        inner = np.polynomial.legendre.Legendre.basis(p).deriv().roots() if p > 1 else np.zeros(0)
        self.nodes = xg if basis else np.concatenate([[-1.0], np.sort(np.real(inner)), [1.0]])
        v, dv = _lagrange(self.nodes, xg)
        self.M, self.K = (v.T * wg) @ v, (dv.T * wg) @ dv
        ends, dends = _lagrange(self.nodes, np.array([-1.0, 1.0]))
        self.e, self.de = ends, dends                              # [low / high, node]


def _along(A, U, ax):
    return torch.movedim(torch.tensordot(U, A, dims=([ax], [1])), -1, ax)


class Sipg:
    """-div(kappa grad u), symmetric interior penalty 2 p (p + 1) / h, facet terms scaled
    by the harmonic mean of kappa; vectors as [cells z, y, x][nodes z, y, x]."""

    def __init__(self, E, kappa, dev, omega=0.8, interior=0):
        self.E, self.d, self.dev, self.omega = E, len(E.n), dev, omega
        d, n = self.d, E.n
        self.shape = tuple(n[::-1]) + (E.q,) * d
        t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=F64, device=dev)
        self.h = [1.0 / v for v in n]
        self.M = [t(E.M * h / 2) for h in self.h]
        self.K = [t(E.K * 2 / h) for h in self.h]
        self.e = t(E.e)
        self.de = [t(E.de * 2 / h) for h in self.h]
        self.gamma = [2.0 * E.p * (E.p + 1) / h for h in self.h]
        k = torch.ones(n[::-1], dtype=F64, device=dev) if kappa is None else t(kappa).view(n[::-1])
        self.kappa = k.view(tuple(n[::-1]) + (1,) * d)
        self.kf = []                                               # per axis: interior facets
        for a in range(d):
            lo, hi = self._cells(self.kappa, a, 0, -1), self._cells(self.kappa, a, 1, None)
            self.kf.append(2 * lo * hi / (lo + hi))
        self.fd = None

    def _cells(self, U, a, lo, hi):
        ix = [slice(None)] * U.dim()
        ix[self.d - 1 - a] = slice(lo, hi)
        return U[tuple(ix)]

    def _vec(self, v, a):
        s = [1] * (2 * self.d)
        s[2 * self.d - 1 - a] = self.E.q
        return v.view(s)

    def apply(self, U):
        d, out = self.d, torch.zeros_like(U)
        for a in range(d):
            na = 2 * d - 1 - a
            V = self.kappa * _along(self.K[a], U, na)
            e, de = [self._vec(self.e[s], a) for s in (0, 1)], [self._vec(self.de[a][s], a) for s in (0, 1)]
            val, der = [(U * v).sum(na, keepdim=True) for v in e], [(U * v).sum(na, keepdim=True) for v in de]
            g = self.gamma[a]
            if self.E.n[a] > 1:
                m, p = (0, -1), (1, None)                          # the facet's two cells
                jump = self._cells(val[1], a, *m) - self._cells(val[0], a, *p)
                mean = (self._cells(der[1], a, *m) + self._cells(der[0], a, *p)) / 2
                flux = self.kf[a] * (g * jump - mean)
                half = self.kf[a] * jump / 2
                self._cells(V, a, *m).add_(flux * e[1] - half * de[1])
                self._cells(V, a, *p).sub_(flux * e[0] + half * de[0])
            for s, ends, sign in ((0, (0, 1), -1.0), (1, (-1, None), 1.0)):   # the boundary
                k, v, w = (self._cells(x, a, *ends) for x in (self.kappa, val[s], der[s]))
                self._cells(V, a, *ends).add_(k * ((g * v - sign * w) * e[s] - sign * v * de[s]))
            for b in range(d):
                if b != a:
                    V = _along(self.M[b], V, 2 * d - 1 - b)
            out += V
        return out

    def factor(self):
        """Fast diagonalisation of the diagonal blocks: S per cell and axis, and the sums."""
        d, n, q = self.d, self.E.n, self.E.q
        self.fd, lams = [], []
        for a in range(d):
            k = self.kappa.reshape(n[::-1])
            c = self.d - 1 - a
            kl, kr, wl, wr = k.clone(), k.clone(), torch.ones_like(k), torch.ones_like(k)
            kf = self.kf[a].reshape([s for i, s in enumerate(self.kf[a].shape) if i < d])
            kl.narrow(c, 1, n[a] - 1).copy_(kf)
            wl.narrow(c, 1, n[a] - 1).fill_(0.5)
            kr.narrow(c, 0, n[a] - 1).copy_(kf)
            wr.narrow(c, 0, n[a] - 1).fill_(0.5)
            o = lambda x, y: torch.outer(x, y)
            e0, ep, d0, dp = self.e[0], self.e[1], self.de[a][0], self.de[a][1]
            f = lambda x: x.reshape(-1, 1, 1)
            Kt = (f(k) * self.K[a] + f(kl * wl) * (o(e0, d0) + o(d0, e0)) + f(kl) * self.gamma[a] * o(e0, e0)
                  - f(kr * wr) * (o(ep, dp) + o(dp, ep)) + f(kr) * self.gamma[a] * o(ep, ep))
            Li = torch.linalg.inv(torch.linalg.cholesky(self.M[a]))
            B = Li @ Kt @ Li.T
            rows, back = torch.unique(B.reshape(len(B), -1), dim=0, return_inverse=True)
            pairs = [torch.linalg.eigh(x.view(-1, q, q)) for x in rows.split(16384)]
            lam, vec = (torch.cat(x) for x in zip(*pairs))
            self.fd.append((Li.T @ vec)[back])
            lams.append(lam[back])
        sh = [len(lams[0])] + [1] * d
        self.sums = 0
        for a in range(d):
            s = list(sh)
            s[d - a] = q
            self.sums = self.sums + lams[a].view(s)

    def _block(self, R):
        d, q = self.d, self.E.q
        X = R.reshape(-1, *([q] * d))
        for trans in (True, False):
            for a in range(d):
                S = self.fd[a].transpose(1, 2) if trans else self.fd[a]
                X = torch.movedim(X, d - a, 1).reshape(len(X), q, -1)
                X = torch.movedim(torch.bmm(S, X).reshape(-1, *([q] * d)), 1, d - a)
            if trans:
                X = X / self.sums
        return X.reshape(self.shape)

    def smooth(self, U, B, steps):
        if self.fd is None:
            self.factor()
        for _ in range(steps):
            U = U + self.omega * self._block(B - self.apply(U))
        return U


class Cycle:
    """One hp V(nu, nu) cycle: block Jacobi, P^T, the Q1 levels with point Jacobi, P."""

    def __init__(self, A, nu, f, omega=0.8):
        self.A, self.nu, self.omega = A, nu, omega
        E, d, dev = A.E, A.d, A.dev
        t = lambda a: torch.tensor(a, dtype=F64, device=dev)
        hats = lambda x: np.stack([(1 - x) / 2, (1 + x) / 2], 1)
        self.P = [t(self._to_cells(n, hats(E.nodes))) for n in E.n]
        self.C = [t(self._to_cells(n, np.eye(2))) for n in E.n]     # vertices -> cell corners
        self.T, n = [], list(E.n)
        while any(v > f for v in n):
            Ts = []
            for a in range(d):
                pos = list(range(0, n[a], f)) + [n[a]] if n[a] > f else list(range(n[a] + 1))
                I = np.zeros((n[a] + 1, len(pos)))
                for j in range(len(pos) - 1):
                    for i in range(pos[j], pos[j + 1] + 1):
                        w = (i - pos[j]) / (pos[j + 1] - pos[j])
                        I[i, j], I[i, j + 1] = 1 - w, w
                Ts.append(t(I[1:-1, 1:-1]))
                n[a] = len(pos) - 1
            self.T.append(Ts)
        self.diag, self.m = [], [tuple(v - 1 for v in E.n[::-1])]
        for Ts in self.T:
            self.m.append(tuple(Ts[a].shape[1] for a in reversed(range(d))))
        for l in range(len(self.m) - 1):                            # diagonals by probing 3^d colours
            D = torch.zeros(self.m[l], dtype=F64, device=dev)
            for c in range(3 ** d):
                x = torch.zeros_like(D)
                ix = tuple(slice((c // 3 ** i) % 3, None, 3) for i in range(d))
                x[ix] = 1
                D[ix] = self.q1(x, l)[ix]
            self.diag.append(D)
        m = int(np.prod(self.m[-1]))
        eye = torch.eye(m, dtype=F64, device=dev)
        self.coarse = torch.stack([self.q1(v.view(self.m[-1]), len(self.m) - 1).reshape(-1) for v in eye])

    @staticmethod
    def _to_cells(n, H):
        """[n * points, interior vertices]: hat values at every cell's points."""
        k = H.shape[0]
        out = np.zeros((n, k, n + 1))
        for c in range(n):
            out[c, :, c], out[c, :, c + 1] = H[:, 0], H[:, 1]
        return out.reshape(n * k, n + 1)[:, 1:-1]

    def tensor(self, mats, x, trans=False):
        d = self.A.d
        for a in range(d):
            x = _along(mats[a].T if trans else mats[a], x, d - 1 - a)
        return x

    def prolong(self, e):
        E, d = self.A.E, self.A.d
        x = self.tensor(self.P, e).view([v for n in E.n[::-1] for v in (n, E.q)])
        return x.permute([2 * i for i in range(d)] + [2 * i + 1 for i in range(d)])

    def restrict(self, R):
        E, d = self.A.E, self.A.d
        x = R.permute([i // 2 + (i % 2) * d for i in range(2 * d)]).reshape([n * E.q for n in E.n[::-1]])
        return self.tensor(self.P, x, True)

    def q1(self, v, l):
        if l > 0:
            return self.tensor(self.T[l - 1], self.q1(self.tensor(self.T[l - 1], v), l - 1), True)
        A, d = self.A, self.A.d
        n = A.E.n
        x = self.tensor(self.C, v).view([s for k in n[::-1] for s in (k, 2)])
        k = A.kappa.reshape([s for m in n[::-1] for s in (m, 1)])
        out = 0
        for a in range(d):
            y = x
            for b in range(d):
                h = A.h[b]
                m = np.array([[1, -1], [-1, 1]]) / h if a == b else np.array([[2, 1], [1, 2]]) * h / 6
                y = _along(torch.tensor(m, dtype=F64, device=A.dev), y, 2 * (d - 1 - b) + 1)
            out = out + k * y
        return self.tensor(self.C, out.reshape([2 * m for m in n[::-1]]), True)

    def levels(self, b, l):
        if l == len(self.T):
            return torch.linalg.solve(self.coarse, b.reshape(-1)).view(self.m[l])
        u = torch.zeros_like(b)
        for _ in range(self.nu):
            u = u + self.omega * (b - self.q1(u, l)) / self.diag[l]
        u = u + self.tensor(self.T[l], self.levels(self.tensor(self.T[l], b - self.q1(u, l), True), l + 1))
        for _ in range(self.nu):
            u = u + self.omega * (b - self.q1(u, l)) / self.diag[l]
        return u

    def __call__(self, B):
        A = self.A
        U = A.smooth(torch.zeros_like(B), B, self.nu)
        U = U + self.prolong(self.levels(self.restrict(B - A.apply(U)), 0))
        return A.smooth(U, B, self.nu)


def _solve(A, B, tol=3e-14, most=80):
    V = Cycle(A, 2, 2)
    X, R = torch.zeros_like(B), B.clone()
    Z = V(R)
    P, rz = Z.clone(), torch.sum(R * Z)
    stop = tol * torch.linalg.norm(B).item()
    for _ in range(most):
        Q = A.apply(P)
        al = rz / torch.sum(P * Q)
        X += al * P
        R -= al * Q
        if torch.linalg.norm(R).item() <= stop:
            break
        Z = V(R)
        new = torch.sum(R * Z)
        P = Z + (new / rz) * P
        rz = new
    return X


def exact(case, seed):
    c = _full(case)
    if c["op"] == "batch":                                          # the first few problems
        out = []
        for i, (E, kappa, m) in enumerate(_batch_problems(c, seed)):
            A = Sipg(E, kappa, DEV)
            out.append(_solve(A, _load(E, *m, DEV).view(A.shape)).reshape(-1) if i < 4 else None)
        return out
    if c["op"] in ("vcycle", "smooth", "solve") and c["kappa"] == "lognormal" and math.prod(c["n"]) > 300000:
        return None                                                 # too many different blocks
    E, kappa, b, u = _problem(c, seed)
    A = Sipg(E, kappa, DEV)
    B = b.view(A.shape)
    if c["op"] == "apply":
        return A.apply(u.view(A.shape)).reshape(-1)
    if c["op"] == "apply_f32":
        return A.apply(u.double().view(A.shape)).reshape(-1)
    if c["op"] == "residual":
        return (B - A.apply(u.view(A.shape))).reshape(-1)
    if c["op"] == "smooth":
        return A.smooth(u.view(A.shape), B, c["steps"]).reshape(-1)
    if c["op"] == "vcycle":
        return Cycle(A, c["nu"], c["coarsening"])(B).reshape(-1)
    return _solve(A, B).reshape(-1)
