"""opts.recompute_block computes the factors of every DG level before every smoothing step,
also on the finest level of a new context: the launches are counted."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FACTOR_KERNELS = {0: 4, 1: 1}      # FP64: eigenvectors, the table's exponents, the table, the limbs; FP32: one


@pytest.mark.parametrize("n,p,opts", [((6, 5, 4), 2, {}), ((9, 7), 3, {}), ((4, 3, 5), 3, {"p_coarsening": 1})])
@pytest.mark.parametrize("precision", [0, 1])
def test_factors_are_computed_before_every_step(n, p, opts, precision):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2510_00998_gb300 import dgmg
    kappa = np.exp(np.random.default_rng(2).normal(size=int(np.prod(n))))
    count = {}
    for rb in (0, 1):
        ctx = dgmg.Context(n, p, kappa, precision=precision, recompute_block=rb, **opts)
        b = torch.randn(ctx.ndof, dtype=torch.float64, device="cuda:0", generator=torch.Generator("cuda:0").manual_seed(3))
        e, u = torch.zeros_like(b), torch.zeros_like(b)
        at = [dgmg.kernel_launches()]
        ctx.smooth(u, b, 3)
        at.append(dgmg.kernel_launches())
        ctx.vcycle(b, e)
        at.append(dgmg.kernel_launches())
        torch.cuda.synchronize()
        count[rb] = np.diff(at)
        ctx.close()
    levels = p if opts else 1
    assert count[1][0] - count[0][0] == 3 * FACTOR_KERNELS[0]                    # dgmg_smooth: FP64
    assert count[1][1] - count[0][1] == 4 * levels * FACTOR_KERNELS[precision]   # nu_pre + nu_post = 4
