"""The vector kernels of the solvers (dot products whose last block finishes the sum,
fused updates): lengths below one block, odd lengths (no whole 16-byte packs) and
lengths of many blocks, with vectors at 16-byte boundaries and one element off them.
The residual that the kernels report is the one of the returned solution, and a
solution does not depend on where its vectors lie: the dots of two runs differ by the
order of their sums only, 1e-13 of ||b|| in a solution converged to 1e-10."""
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


def _off(t, off):
    buf = torch.empty(t.numel() + 2, dtype=t.dtype, device=DEV)
    assert buf.data_ptr() % 16 == 0
    v = buf[off:off + t.numel()]
    v.copy_(t)
    return v


@pytest.mark.parametrize("n,p", [((2, 2), 2), ((3, 3), 2), ((5, 5), 4), ((3, 3, 3), 2), ((41, 37), 2), ((9, 11, 7), 4)])
@pytest.mark.parametrize("opts", [{}, {"nu_pre": 2, "nu_post": 1}, {"precision": 1}, {"outer": 2}])
def test_solution_of_any_length_and_alignment(dgmg, n, p, opts):
    opts = dict(opts)
    mesh = sipg.Mesh(n, p)
    rng = np.random.default_rng(mesh.ndof)
    kap = np.exp(0.5 * rng.normal(size=int(np.prod(n))))
    b = torch.tensor(rng.normal(size=mesh.ndof), device=DEV)
    if opts.pop("outer", None):
        opts["outer"] = dgmg.DGMG_OUTER_MGMULT
    ctx = dgmg.Context(n, p, kap, **opts)
    sol = []
    for off in (0, 1):
        x = _off(torch.zeros_like(b), off)
        st, _ = ctx.solve(_off(b, off), x, allow_notconverged=True)   # the stationary cycle may need more
        sol.append(x.cpu().numpy())
        res = np.linalg.norm(b.cpu().numpy() - sipg.apply(mesh, sol[-1], kap)) / np.linalg.norm(b.cpu().numpy())
        assert abs(st.rel_residual - res) <= 1e-3 * res + 1e-14
    assert np.abs(sol[0] - sol[1]).max() <= 1e-10 * np.abs(sol[0]).max()


@pytest.mark.parametrize("prec", [0, 1])
def test_batch_of_any_lengths_and_alignment(dgmg, prec):
    spec = [((2, 2), 2), ((3, 3), 2), ((5, 5), 4), ((41, 37), 2), ((2, 3), 1)]
    rng = np.random.default_rng(5)
    meshes = [sipg.Mesh(n, p) for n, p in spec]
    bs = [torch.tensor(rng.normal(size=m.ndof), device=DEV) for m in meshes]
    batch = dgmg.Batch([(n, p, None) for n, p in spec], precision=prec)
    sol = []
    for off in (0, 1):
        xs = [_off(torch.zeros_like(b), off) for b in bs]
        stats, _ = batch.solve([_off(b, off) for b in bs], xs)
        for m, b, x, st in zip(meshes, bs, xs, stats):
            bn = b.cpu().numpy()
            res = np.linalg.norm(bn - sipg.apply(m, x.cpu().numpy())) / np.linalg.norm(bn)
            assert res <= 1.05e-10 and abs(st.rel_residual - res) <= 1e-3 * res + 1e-14
        sol.append(xs)
    for x, y in zip(*sol):
        assert (x - y).abs().max().item() <= 1e-10 * x.abs().max().item()
