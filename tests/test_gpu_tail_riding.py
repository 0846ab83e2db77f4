"""The fused last layer in steps whose weight-gradient launches carry the next step's forward products:
the launch of the layer below adds the bias that the fused last layer's side branch steps."""
import numpy as np
import pytest

from tests.util import l2_rel

pytestmark = pytest.mark.gpu


def _run(dims, P, profiled, schedule, beta=0.0):
    import paper_2110_00625_b200 as m
    B, K = 16, 5                     # (up to four steps may be rebuilt, where nothing rides)
    rng = np.random.default_rng(5)
    x = rng.standard_normal((1024, dims[0]), dtype=np.float32)
    y = rng.integers(0, dims[-1], size=1024).astype(np.int32)
    g = m.Mavg(m.workloads.mlp_init(dims), P=P, K=K, local_lr=0.01, mu=0.9, B=B, seed=3,
               objective=m.OBJ_MLP, dims=dims, gemm_bf16=1, x=x, y=y, x_bf16=True,
               defer_broadcast=True, learner_momentum=beta)
    assert g.get_step_plan()["fwd_with_wgrad"] == len(dims) - 2 and not g.rebuilt()
    g.set_schedule(schedule)
    g.set_profiling(profiled)
    losses = [g.round(want_loss=True) for _ in range(2)]
    g.sync()
    out = [g.w.cpu().numpy(), g.v.cpu().numpy(), g.replicas[:, :g.n].cpu().numpy()]
    g.close()
    return losses, out


@pytest.mark.parametrize("dims,P", [([8192, 512, 10], 18), ([3072, 512, 10], 48),
                                    ([3072, 512, 256, 10], 56)])
@pytest.mark.parametrize("beta", [0.0, 0.9])
def test_graph_equals_launch_by_launch(dims, P, beta):
    # the launch-by-launch form has no side branch: the same bits mean that the branch is joined in time
    la, a = _run(dims, P, False, 0, beta)
    lb, b = _run(dims, P, True, 0, beta)
    assert la == lb
    for x, y in zip(a, b):
        assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
    # and the plain tensor-core launches, which differ in summation order (per-round drift bound 5e-2)
    lc, c = _run(dims, P, False, 2, beta)
    assert np.allclose(la, lc, rtol=2e-2)
    assert l2_rel(a[1], c[1]) <= 5e-2
