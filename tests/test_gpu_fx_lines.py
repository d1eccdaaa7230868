"""The FP64 kernels beside what test_gpu_fx.py looks at: the whole V-cycle scales exactly
with powers of two, and on both sides of the line between one lane per slab and several the
smoothing steps (both block forms) and the projection with a correction agree with the
oracle, too."""
import numpy as np
import pytest

from oracle import hpmg, sipg

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


@pytest.mark.parametrize("n,p,opts", [((5, 4), 3, {}), ((4, 3, 3), 2, {}), ((40, 30), 1, {}), ((3, 3, 2), 4, {"p_coarsening": 1}),
                                      ((6, 5), 2, {"basis": 1, "nu_pre": 0})])
def test_vcycle_scales_with_powers_of_two(dgmg, n, p, opts):
    ctx = dgmg.Context(n, p, np.exp(np.random.default_rng(1).normal(size=int(np.prod(n)))), **opts)
    b = torch.randn(ctx.ndof, dtype=torch.float64, device=DEV, generator=torch.Generator(DEV).manual_seed(2))
    out = []
    for s in (1.0, 2.0 ** 400, 2.0 ** -400):
        e = torch.empty_like(b)
        ctx.vcycle(b * s, e)
        out.append(e / s)
    assert torch.equal(out[1], out[0]) and torch.equal(out[2], out[0])


@pytest.mark.parametrize("n,p", [((13, 13, 14), 4), ((14, 14, 13), 4), ((12, 12, 10), 5), ((12, 12, 11), 5)])
@pytest.mark.parametrize("interior", [0, 1])
def test_steps_and_projection_on_both_sides_of_the_split(dgmg, n, p, interior):
    rng = np.random.default_rng(p)
    kap = np.exp(rng.normal(size=int(np.prod(n))))
    mesh = sipg.Mesh(n, p)
    ctx = dgmg.Context(n, p, kap, block_inverse=interior)
    u, b = rng.normal(size=mesh.ndof), rng.normal(size=mesh.ndof)
    v = _t(u)
    ctx.smooth(v, _t(b), 2)
    ref = sipg.BlockJacobi(mesh, kap, interior_only=bool(interior)).step_alg2(u, b, 0.8, 2)
    assert _rel(v.cpu().numpy(), ref) <= 1e-11
    e = rng.normal(size=int(ctx.info.nvert0))
    w, tr = _t(u), torch.empty(ctx.trace_size(), dtype=torch.float64, device=DEV)
    ctx.project(w, _t(e), tr)
    assert _rel(w.cpu().numpy(), u + hpmg.p_prolongation(mesh) @ e) <= 1e-13
    r = torch.empty_like(w)
    ctx.residual_restrict(w, _t(b), tr, r, None)     # from those traces the residual of the new u
    assert _rel(r.cpu().numpy(), sipg.residual(mesh, w.cpu().numpy(), b, kap)) <= 1e-12
