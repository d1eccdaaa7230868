"""The FP64 kernels in block fixed-point arithmetic: every degree at meshes that end
inside a warp and inside a CTA, against the oracle; results scale exactly with powers
of two (the exponents carry the scale, the integers do not change); a value that is
not finite reaches its cell and the face neighbours as NaN and no other cell."""
import numpy as np
import pytest

from oracle import sipg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.fixture(scope="module")
def dgmg():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2510_00998_gb300 import dgmg as m
    return m


def _t(x):
    return torch.tensor(np.asarray(x, dtype=np.float64), device=DEV)


def _rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


MESHES = [((2, 2), 1), ((17, 3), 3), ((5, 9), 6), ((2, 3, 2), 1), ((11, 2, 3), 2), ((3, 5, 3), 3), ((7, 2, 2), 4),
          ((2, 3, 4), 5), ((3, 2, 3), 6)]


@pytest.mark.parametrize("n,p", MESHES)
@pytest.mark.parametrize("interior", [0, 1])
def test_smooth_and_residual_every_degree(dgmg, n, p, interior):
    rng = np.random.default_rng(p)
    kap = np.exp(rng.normal(size=int(np.prod(n))))
    mesh = sipg.Mesh(n, p)
    ctx = dgmg.Context(n, p, kap, block_inverse=interior)
    u, b = rng.normal(size=mesh.ndof), rng.normal(size=mesh.ndof)
    r = torch.empty(mesh.ndof, dtype=torch.float64, device=DEV)
    ctx.residual(_t(u), _t(b), r)
    assert _rel(r.cpu().numpy(), sipg.residual(mesh, u, b, kap)) <= 1e-12
    ut = _t(u)
    ctx.smooth(ut, _t(b), 2)
    ref = sipg.BlockJacobi(mesh, kap, interior_only=bool(interior)).step_alg2(u, b, 0.8, 2)
    assert _rel(ut.cpu().numpy(), ref) <= 1e-11


@pytest.mark.parametrize("n,p", [((5, 4), 3), ((4, 3, 3), 2), ((3, 3, 2), 4)])
def test_results_scale_with_powers_of_two(dgmg, n, p):
    ctx = dgmg.Context(n, p, np.exp(np.random.default_rng(1).normal(size=int(np.prod(n)))))
    u, b = torch.randn(2, ctx.ndof, dtype=torch.float64, device=DEV, generator=torch.Generator(DEV).manual_seed(2))
    out = []
    for s in (1.0, 2.0 ** 400, 2.0 ** -400):
        r, e, v = torch.empty_like(u), torch.empty_like(u), (u * s).clone()
        ctx.residual(u * s, b * s, r)
        ctx.vcycle(b * s, e)
        ctx.smooth(v, b * s, 3)
        out.append([w / s for w in (r, v)])
    for w in out[1:]:
        assert all(torch.equal(x, y) for x, y in zip(w, out[0]))


def test_a_nan_stays_in_its_cell_and_its_neighbours(dgmg):
    n, p = (5, 4, 3), 2
    ctx = dgmg.Context(n, p)
    u = torch.randn(ctx.ndof, dtype=torch.float64, device=DEV, generator=torch.Generator(DEV).manual_seed(3))
    y0, y1 = torch.empty_like(u), torch.empty_like(u)
    ctx.apply(u, y0)
    cell = 2 + 5 * (1 + 4 * 1)
    for bad in (float("nan"), float("inf")):
        v = u.clone()
        v[cell * 27 + 13] = bad                     # an inner node: on no face, but in every derivative trace
        ctx.apply(v, y1)
        hit = {cell} | {cell + s * d for s in (1, 5, 20) for d in (1, -1)}
        for c in range(60):
            blk0, blk1 = y0[c * 27:(c + 1) * 27], y1[c * 27:(c + 1) * 27]
            if c in hit:
                assert not torch.isfinite(blk1).all()
            else:
                assert torch.equal(blk0, blk1)


@pytest.mark.parametrize("n,p", MESHES)
@pytest.mark.parametrize("basis", [0, 1])
def test_callers_traces_and_own_traces_agree(dgmg, n, p, basis):
    """The residual from FP64 traces that the caller holds and the one whose traces stay
    integers inside: the same sums up to the rounding of the traces to 53 bits, a few
    1e-16 of terms a few hundred times the residual."""
    rng = np.random.default_rng(20 + p)
    ctx = dgmg.Context(n, p, np.exp(rng.normal(size=int(np.prod(n)))), basis=basis)
    u, b = _t(rng.normal(size=ctx.ndof)), _t(rng.normal(size=ctx.ndof))
    tr = torch.empty(ctx.trace_size(), dtype=torch.float64, device=DEV)
    own, user = torch.empty_like(u), torch.empty_like(u)
    ctx.residual(u, b, own)
    ctx.project(u, None, tr)
    ctx.residual_restrict(u, b, tr, user, None)
    assert _rel(user.cpu().numpy(), own.cpu().numpy()) <= 1e-13


@pytest.mark.parametrize("n,p", [((13, 13, 14), 4), ((14, 14, 13), 4), ((12, 12, 10), 5), ((12, 12, 11), 5),
                                 ((13, 13, 14), 6), ((14, 14, 13), 6)])
def test_residual_on_both_sides_of_the_split(dgmg, n, p):
    """3D, p >= 4: meshes just below and just above the size from which a slab has one
    lane instead of several."""
    rng = np.random.default_rng(p)
    kap = np.exp(rng.normal(size=int(np.prod(n))))
    mesh = sipg.Mesh(n, p)
    ctx = dgmg.Context(n, p, kap)
    u, b = rng.normal(size=mesh.ndof), rng.normal(size=mesh.ndof)
    r = torch.empty(mesh.ndof, dtype=torch.float64, device=DEV)
    ctx.residual(_t(u), _t(b), r)
    assert _rel(r.cpu().numpy(), sipg.residual(mesh, u, b, kap)) <= 1e-12
