"""How exact the FP64 kernels in block fixed-point arithmetic are, cell by cell, against
extended precision: coefficients that jump, stretched meshes, values of a wide range
inside a cell. A cell's error is taken of that cell's largest value."""
import numpy as np
import pytest

from ref_long import L, Reference

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def dgmg():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2510_00998_gb300 import dgmg as m
    return m


def _t(x):
    return torch.tensor(np.asarray(x, dtype=np.float64), device=DEV)


def _kappa(kind, n, rng):
    nc = int(np.prod(n))
    return 10.0 ** rng.uniform(-kind / 2, kind / 2, size=nc) if kind else np.exp(rng.normal(size=nc))


def _cell_error(got, ref):
    e = np.abs(got.cpu().numpy().astype(L).reshape(ref.shape) - ref).max(1)
    return float((e / np.abs(ref).max(1)).max())


@pytest.mark.parametrize("n,p,jumps", [((5, 4, 3), 3, 0), ((5, 4, 3), 3, 6), ((5, 4, 3), 3, 12), ((4, 3, 3), 5, 0),
                                       ((4, 3, 3), 5, 6), ((9, 8), 4, 0), ((2, 2, 60), 4, 0)])
@pytest.mark.parametrize("near", [0, 1])
def test_smoothing_step_per_cell(dgmg, n, p, jumps, near):
    """One step from a random right-hand side, and (near) from b = A u, where the step
    has to give u back. The step is 3 d passes of q products, each as good as a sum in FP64
    with a rounding per product, from eigenvectors and eigenvalues that carry as much."""
    rng = np.random.default_rng(5)
    kap = _kappa(jumps, n, rng)
    ref, ctx = Reference(n, p, kap), dgmg.Context(n, p, kap)
    u, b = rng.normal(size=(2, ctx.ndof))
    if near:
        b = ref.apply(u).reshape(-1).astype(np.float64)
    v = _t(u)
    ctx.smooth(v, _t(b), 1)
    assert _cell_error(v, ref.step(u, b, 0.8)) <= 2 * 3 * len(n) * (p + 1) * EPS


@pytest.mark.parametrize("seed", [0, 3])
def test_smoothing_step_on_stretched_cells(dgmg, seed):
    """The same where one axis' terms are hundreds of times the others'."""
    n, p = (40, 2, 2), 3
    rng = np.random.default_rng(seed)
    kap = _kappa(0, n, rng)
    ref, ctx = Reference(n, p, kap), dgmg.Context(n, p, kap)
    u, b = rng.normal(size=(2, ctx.ndof))
    v = _t(u)
    ctx.smooth(v, _t(b), 1)
    assert _cell_error(v, ref.step(u, b, 0.8)) <= 2 * 3 * len(n) * (p + 1) * EPS


def _wide(rng, n):
    """Values over 60 binary orders in every cell."""
    return rng.normal(size=n) * 2.0 ** -rng.uniform(0, 60, size=n)


MESHES = [((5, 4), 3, 0), ((5, 4, 3), 2, 0), ((5, 4, 3), 2, 1), ((4, 3, 3), 5, 0), ((3, 4), 6, 1)]


@pytest.mark.parametrize("n,p,basis", MESHES)
def test_residual_keeps_the_bits_of_b(dgmg, n, p, basis):
    """r = b - A u node by node: where A u is zero, r is b."""
    rng = np.random.default_rng(p)
    ctx = dgmg.Context(n, p, _kappa(0, n, rng), basis=basis)
    b, nl = _t(_wide(rng, ctx.ndof)), (p + 1) ** len(n)
    u, r = torch.zeros_like(b), torch.empty_like(b)
    ctx.residual(u, b, r)
    assert torch.equal(r, b)
    tr, rc = torch.zeros(ctx.trace_size(), dtype=torch.float64, device=DEV), _t(np.empty(int(ctx.info.nvert0)))
    for corners in (None, rc):
        r.zero_()
        ctx.residual_restrict(u, b, tr, r, corners)
        assert torch.equal(r, b)
    u[:nl] = 1.0                                     # the first cell: its neighbours see it, the rest does not
    ctx.residual(u, b, r)
    far = torch.ones(ctx.ndof // nl, dtype=torch.bool, device=DEV)
    far[[0, 1, n[0]] + ([n[0] * n[1]] if len(n) == 3 else [])] = False
    assert torch.equal(r.view(-1, nl)[far], b.view(-1, nl)[far])


@pytest.mark.parametrize("n,p,basis", MESHES)
def test_projection_keeps_the_bits_of_u(dgmg, n, p, basis):
    """u + P e node by node: a correction that is zero leaves u as it is, one that is zero
    at a node leaves that node; the value traces of the Lobatto basis are u's end nodes."""
    rng = np.random.default_rng(p)
    d, q = len(n), p + 1
    ctx = dgmg.Context(n, p, _kappa(0, n, rng), basis=basis)
    u = _t(_wide(rng, ctx.ndof))
    tr, e = torch.empty(ctx.trace_size(), dtype=torch.float64, device=DEV), torch.zeros(int(ctx.info.nvert0), dtype=torch.float64, device=DEV)
    v = u.clone()
    ctx.project(v, e, tr)
    assert torch.equal(v, u)
    e[0] = 3.0                                       # the vertex (1, 1[, 1]): the cells around it
    ctx.project(v, e, tr)
    w, x = v.view(n[::-1] + (q,) * d), u.view(n[::-1] + (q,) * d)
    near = torch.zeros(n[::-1], dtype=torch.bool, device=DEV)
    near[(slice(0, 2),) * d] = True
    assert torch.equal(w[~near], x[~near]) and not torch.equal(w[near], x[near])
    if basis == 0:
        assert torch.equal(w[(0,) * d][..., 0], x[(0,) * d][..., 0])     # the hat is zero on x = 0
        faces = tr.view(ctx.ndof // q ** d, 2 * d, 2, -1)
        vals = w.reshape(-1, *(q,) * d)
        assert torch.equal(faces[:, 0, 0], vals[..., 0].reshape(len(faces), -1))
        assert torch.equal(faces[:, 1, 0], vals[..., q - 1].reshape(len(faces), -1))
        last = vals[:, 0].reshape(len(faces), -1)    # the first slab: the last axis' low face
        assert torch.equal(faces[:, 2 * d - 2, 0], last)


@pytest.mark.parametrize("n,p,basis", MESHES)
@pytest.mark.parametrize("steps", [1, 3])
def test_smoothing_keeps_the_bits_of_u(dgmg, n, p, basis, steps):
    """u <- (1 - omega) u + omega D^-1 (b - N u) node by node: where b and the neighbours
    are zero, every step multiplies, whatever range the cell's values have."""
    rng = np.random.default_rng(p)
    ctx, nl = dgmg.Context(n, p, _kappa(0, n, rng), basis=basis, omega_dg=0.75), (p + 1) ** len(n)
    u = torch.zeros(ctx.ndof, dtype=torch.float64, device=DEV)
    last = slice(ctx.ndof - nl, None)                # the last cell
    u[last] = _t(_wide(rng, nl))
    v = u.clone()
    ctx.smooth(v, torch.zeros_like(u), 1)
    assert torch.equal(v[last], 0.25 * u[last])
    if steps > 1:
        w = u.clone()
        ctx.smooth(w, torch.zeros_like(u), steps)
        x = v
        for _ in range(steps - 1):
            ctx.smooth(x, torch.zeros_like(u), 1)
        # traces from the step and from the projection of its result: the same block
        assert torch.equal(w, x)


@pytest.mark.parametrize("n,p,basis", MESHES)
@pytest.mark.parametrize("scale", [-1015, -1020, -1030, -1050])
def test_values_below_the_normal_range(dgmg, n, p, basis, scale):
    """Residual, step and projection of values around and below 2^-1022: the relative bounds
    of the normal range (the residual: sums of 4 d + 2 terms per pass, d + 1 passes of q
    products) and the spacing of subnormal numbers, once per result and once per trace value
    that the caller reads and hands on."""
    rng = np.random.default_rng(p)
    d, q = len(n), p + 1
    kap = _kappa(0, n, rng)
    ref, ctx = Reference(n, p, kap, basis), dgmg.Context(n, p, kap, basis=basis)
    tiny = float(np.finfo(np.float64).smallest_subnormal)
    u, b = rng.normal(size=(2, ctx.ndof)) * 2.0 ** scale
    r = torch.empty(ctx.ndof, dtype=torch.float64, device=DEV)
    ctx.residual(_t(u), _t(b), r)
    exact = ref.residual(u, b)
    size = float(np.abs(exact).max())

    def err(x, y):
        return float(np.abs(x.cpu().numpy().astype(L).reshape(y.shape) - y).max())

    assert err(r, exact) <= 2 * (d + 1) * q * EPS * size + tiny
    v = _t(u)
    ctx.smooth(v, _t(b), 1)
    exact = ref.step(u, b, 0.8)
    assert err(v, exact) <= 2 * 3 * d * q * EPS * float(np.abs(exact).max()) + tiny
    e = torch.zeros(int(ctx.info.nvert0), dtype=torch.float64, device=DEV)
    e[0] = 2.0 ** scale
    w, tr = _t(0 * u), torch.empty(ctx.trace_size(), dtype=torch.float64, device=DEV)
    ctx.project(w, e, tr)
    assert abs(float(w.max()) / tiny - 2.0 ** (scale + 1074)) <= (0 if basis == 0 else 2.0 ** (scale + 1074))
    z = torch.zeros_like(w)
    ctx.residual_restrict(z, z, tr, r, None)         # the traces alone: - A w without the cells' own blocks
    full = -(ref.apply(w.cpu().numpy()) - ref.apply(w.cpu().numpy(), own=True))
    gain = float(np.abs(ref.apply(np.ones(ctx.ndof))).max()) * 4 * d * q
    assert err(r, full) <= 2 * (d + 1) * q * EPS * float(np.abs(full).max()) + (1 + gain) * tiny


@pytest.mark.parametrize("n,p", [((4, 3), 2), ((4, 3, 2), 1), ((3, 3, 3), 4)])
def test_factors_that_are_not_finite(dgmg, n, p):
    """Coefficients whose blocks overflow leave no numbers that look like a result."""
    ctx = dgmg.Context(n, p, np.full(int(np.prod(n)), 1e300))
    b = torch.randn(ctx.ndof, dtype=torch.float64, device=DEV, generator=torch.Generator(DEV).manual_seed(1))
    for u in (b.clone(), torch.zeros_like(b)):
        ctx.smooth(u, b, 1)
        assert torch.isnan(u).all()
    e = torch.zeros_like(b)
    ctx.vcycle(b, e)
    assert torch.isnan(e).all()
