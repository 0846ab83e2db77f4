"""Where the fused last layer and the side launch of the last two layers' weight gradients are taken: both
sides of every line of the rule."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
K = 2

# dims, P, B, fused last layer, side launch (a GPU of 148 SMs)
CASES = [
    ([128, 128, 128, 10], 74, 32, True, True),         # half a wave of the data gradient's tiles
    ([128, 128, 128, 10], 75, 32, True, False),        # more: few weights, less than a wave of learners
    ([128, 128, 128, 10], 148, 32, True, False),
    ([128, 128, 128, 10], 149, 32, False, False),      # more than a wave of learners
    ([64, 800, 800, 16], 10, 32, True, True),          # 70 tiles
    ([64, 800, 800, 16], 16, 32, True, False),         # 112
    ([64, 800, 800, 16], 15, 32, False, False),        # 105 tiles: below three quarters of a wave
    ([64, 520, 520, 32], 24, 16, False, False),        # more than 16 K weights
    ([64, 128, 32], 128, 64, True, False),             # rows x weights: 32 M
    ([64, 128, 32], 128, 80, False, False),
    ([64, 512, 32], 48, 64, True, False),              # 48 M, four row tiles
    ([64, 512, 32], 52, 64, False, False),
    ([64, 64, 4], 128, 256, True, False),              # 32 K rows
    ([64, 64, 4], 129, 256, False, False),
]


@pytest.mark.parametrize("dims,P,B,fused,beside", CASES)
def test_both_sides_of_the_rule(dims, P, B, fused, beside):
    import paper_2110_00625_b200 as m
    x = np.random.default_rng(1).standard_normal((512, dims[0]), dtype=np.float32)
    y = np.zeros(512, dtype=np.int32)
    g = m.Mavg(m.workloads.mlp_init(dims), P=P, K=K, local_lr=0.01, mu=0.9, B=B, seed=3,
               objective=m.OBJ_MLP, dims=dims, gemm_bf16=1, x=x, y=y)
    assert g.get_step_plan()["wgrad_merged"]
    g.set_profiling(True)                # launch by launch: one launch takes all weight gradients
    g.round()
    prof = g.get_profile()
    g.set_profiling(False)
    before = g.launch_count()
    g.local_steps()                      # the graph, after the launch that sets its round
    replayed = g.launch_count() - before - 1
    serial = sum(n for _, n in prof.values()) - prof["meta_update"][1] - prof["broadcast"][1] - prof["aux"][1]
    g.close()
    assert prof["loss"][1] == (2 * K if fused else 0)
    assert replayed - serial == (K if beside else 0)
