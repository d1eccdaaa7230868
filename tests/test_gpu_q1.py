"""The one-launch Q1 cycle: its small levels as one product with the matrix of the cycle
on them, the larger ones on the whole grid, against the oracle's V-cycle. Meshes whose
finest Q1 level is the dense one (also a single level), whose dense level is at the
limit of its size or just above it, and with one to three levels on the grid; thin
meshes; both coarsening factors; steps before and after from 0 up; and a new kappa,
for which weights and matrix are computed again. The tolerances are those of the
V-cycle of each precision."""
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


def _check(ctx, mesh, kap, opts, tol):
    r = np.random.default_rng(3).normal(size=mesh.ndof)
    e = torch.empty(mesh.ndof, dtype=torch.float64, device=DEV)
    ctx.vcycle(_t(r), e)
    ref = hpmg.Hierarchy(mesh, kap, **opts).vcycle(r)
    assert np.abs(e.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("n,p,opts", [
    ((2, 2), 2, {}), ((2, 2, 2), 1, {}), ((16, 16), 2, {}), ((5, 3, 4), 2, {}),
    ((34, 34), 1, {}), ((35, 34), 1, {}),     # 1089 vertices: dense from the finest level; 1122: the first on the grid
    ((11, 12, 11), 1, {}), ((12, 12, 11), 1, {}),
    ((300, 3), 1, {}), ((2, 70, 3), 1, {}), ((90, 3, 40), 1, {}),
    ((40, 30), 1, {"nu_pre": 0, "nu_post": 1}), ((60, 50), 1, {"nu_pre": 0, "nu_post": 2}),
    ((60, 50), 1, {"nu_pre": 2, "nu_post": 0}), ((22, 21, 20), 1, {"nu_pre": 1, "nu_post": 0}),
    ((60, 50), 1, {"nu_pre": 3, "nu_post": 2}), ((24, 20, 28), 1, {"factor": 3}), ((80, 81), 1, {"factor": 3})])
@pytest.mark.parametrize("prec", [0, 1])
def test_cycle_of_any_hierarchy(dgmg, n, p, opts, prec):
    kap = np.exp(np.random.default_rng(p).normal(size=int(np.prod(n))))
    mesh = sipg.Mesh(n, p)
    copts = {("coarsening" if k == "factor" else k): v for k, v in opts.items()}
    ctx = dgmg.Context(n, p, kap, precision=prec, **copts)
    _check(ctx, mesh, kap, opts, 2e-5 if prec else 1e-11)
    kap2 = np.exp(np.random.default_rng(p + 7).normal(size=int(np.prod(n))))
    ctx.update_kappa(kap2)
    _check(ctx, mesh, kap2, opts, 2e-5 if prec else 1e-11)
    assert dgmg.wait_timeouts() == 0


@pytest.mark.parametrize("prec", [0, 1])
def test_cycle_under_capture(dgmg, prec):
    """Both launch forms replay from a graph with the same result."""
    for n in ((16, 16), (60, 50)):
        ctx = dgmg.Context(n, 1, None, precision=prec)
        r = torch.randn(ctx.ndof, dtype=torch.float64, device=DEV, generator=torch.Generator(DEV).manual_seed(1))
        e = torch.empty_like(r)
        ctx.vcycle(r, e)
        ref = e.clone()
        torch.cuda.synchronize()
        g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(g, stream=s):
            ctx.vcycle(r, e, stream=s)
        e.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(e, ref)
