"""Batched FP64 solves of small problems of high degree: as single solves, they take
several lanes per slab while the problems of a degree have few cells together, and one
beyond; the map of the work items has to follow. Batches below, at and above the line
against single solves, whose kernels take the line by their own cells."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
DEV = "cuda:0"


@pytest.mark.parametrize("problems", [
    [((3, 4, 3), 5), ((2, 3, 5), 5)], [((4, 4, 4), 4), ((5, 3, 3), 4), ((3, 3, 3), 2)], [((3, 3, 4), 6)],
    [((8, 10, 19), 5)], [((8, 10, 19), 5), ((2, 2, 2), 5)], [((16, 8, 19), 4)], [((13, 11, 17), 4), ((2, 2, 3), 4)]])
def test_batch_agrees_with_single_solves(problems):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2510_00998_gb300 import dgmg
    rng = np.random.default_rng(1)
    probs = [(n, p, np.exp(0.3 * rng.normal(size=int(np.prod(n))))) for n, p in problems]
    bs = [torch.tensor(rng.normal(size=int(np.prod(n)) * (p + 1) ** 3), device=DEV) for n, p, _ in probs]
    xs = [torch.zeros_like(b) for b in bs]
    batch = dgmg.Batch(probs, rtol=1e-12)
    sts, _ = batch.solve(bs, xs)
    info = batch.info()
    for k in range(info.groups):
        q = info.group_q[k]
        cells = sum(int(np.prod(n)) for n, p, _ in probs if p + 1 == q)
        if q >= 5:
            assert list(info.group_tiles[k]) == ([4] * 3 if cells <= (1520 if q == 6 else 2432) else [{5: 24, 6: 20, 7: 16}[q]] * 3)
    for (n, p, kap), b, x, st in zip(probs, bs, xs, sts):
        y = torch.zeros_like(b)
        one = dgmg.Context(n, p, kap, rtol=1e-12)
        one.solve(b, y)
        assert st.rel_residual <= 1e-12
        assert float((x - y).norm() / y.norm()) <= 1e-8      # two solutions to 1e-12, conditions up to 1e4
