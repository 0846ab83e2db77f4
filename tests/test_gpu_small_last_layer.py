"""Small models: the last layer of a step in one pass (up to 32 classes: 4, 8, 16 or 32 lanes of a warp to a row), and the
round's mean loss as the meta-update's launch leaves it, alone and beside other handles."""
import numpy as np
import pytest

from tests.util import l2_rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("dims,B,P", [
    ([20, 30, 2], 9, 3), ([7, 4], 5, 2), ([33, 17, 5], 31, 2), ([12, 40, 8], 4, 40), ([24, 9, 17], 37, 3),
    ([16, 50, 32], 8, 2), ([16, 50, 33], 8, 2)])
def test_round_and_its_mean_loss(oracle, mode, dims, B, P):
    import paper_2110_00625_b200 as m
    rng = np.random.default_rng(B)
    x = rng.standard_normal((50 * P, dims[0]), dtype=np.float32)
    y = rng.integers(0, dims[-1], size=len(x)).astype(np.int32)
    w1 = m.workloads.mlp_init(dims)
    kw = dict(P=P, K=3, mu=0.9, B=B, seed=7, dims=dims, x=x, y=y)
    g = [m.Mavg(w1, local_lr=0.01, objective=m.OBJ_MLP, gemm_bf16=mode, defer_broadcast=bool(i), **kw) for i in (0, 1)]
    o = oracle.Mavg(w1, gamma=0.01, objective=oracle.OBJ_MLP, bf16=mode != 0, stride=g[0].stride, **kw)
    tol = 2e-6 if mode == 0 else 2e-3        # a few steps' sums in another order, operands that round the other way
    for r in range(3):
        got = [h.round(want_loss=r != 1) for h in g]
        losses, _ = o.local_steps()
        o.meta_update()
        for h, mean in zip(g, got):
            own = h.get_losses()
            assert l2_rel(own, losses) <= 10 * (r + 1) * tol
            if r != 1:                       # the mean in fp32, over P x K losses
                assert abs(mean - own.astype(np.float64).mean()) <= 1e-6 * abs(mean)
            assert l2_rel(h.w.cpu().numpy(), o.w) <= (r + 1) * tol
    for h in g:
        h.close()
