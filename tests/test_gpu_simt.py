"""CUDA-core learner steps at the edges of their tiles and of the rules that choose between their
launches, against the oracle, in the two forms (all steps of a small model in one launch, and a launch per
product, there from a graph and launch by launch in profiled rounds): two local steps from identical
replicas with learner momentum, whose buffers hold the gradients without the cancellation of a weight
difference."""
import numpy as np
import pytest

from tests.util import l2_rel, mlp_layout

pytestmark = pytest.mark.gpu
SEED = 0x211000625

# dims, B, P: what it reaches
SMALL = [                                  # one launch for both steps
    ([5, 3], 1, 1),                        # one layer, one sample, everything smaller than a tile
    ([64, 64, 64, 10], 64, 3),             # whole groups of rows
    ([65, 129, 33, 7], 63, 2),             # rows that do not start on 16 bytes, ragged everywhere
    ([9, 1, 7], 3, 1),                     # a width of one, fewer samples than a group of rows
    ([32, 64, 10], 32, 4),                 # eight blocks a learner, one group of rows each
    ([33, 40, 40, 12], 29, 5),             # uneven rows and columns per block, padded rows
    ([32, 64, 10], 50, 150),               # more learners than SMs: one block each
    ([24, 30, 40], 70, 40),                # two blocks a learner, more than 32 classes
    ([80, 128, 112, 16], 32, 3),           # the largest of its kind: four rows of W share a task
]
PRODUCTS = [                               # a launch per product
    ([5000, 3], 1, 1),                     # one layer, one sample
    ([3072, 10], 65, 2),                   # one layer, last row block of one sample
    ([64, 64, 64, 64, 64, 10], 64, 3),     # whole tiles, contraction of one slab group
    ([65, 129, 63, 7], 65, 2),             # rows that do not start on 16 bytes, ragged everywhere
    ([260, 132, 100], 100, 2),             # 16-byte rows, ragged tiles; 100 classes in one launch
    ([1000, 333, 100], 50, 2),             # the last layer's weights start off 16 bytes
    ([1024, 512, 100], 40, 1),             # last layer just above what one launch holds: 4 launches
    ([96, 256, 600], 33, 2),               # many classes
    ([3072, 64, 10], 16, 1),               # contraction split over eight blocks
    ([130, 72, 40, 24, 16, 6], 9, 2),      # five layers
    ([1500, 1, 1500], 3, 1),               # a width of one
    ([80, 128, 128, 16], 32, 3),           # just past the largest small model
]


@pytest.mark.parametrize("profiled", [False, True])
@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("dims,B,P", SMALL + PRODUCTS)
def test_two_steps_against_the_oracle(oracle, mode, dims, B, P, profiled):
    import paper_2110_00625_b200 as m
    S = 40 * P + 3
    rng = np.random.default_rng(len(dims) * 1000 + B)
    x = rng.standard_normal((S, dims[0]), dtype=np.float32)
    y = rng.integers(0, dims[-1], size=S).astype(np.int32)
    w1 = m.workloads.mlp_init(dims)
    kw = dict(P=P, K=2, mu=0.9, B=B, seed=SEED, dims=dims, x=x, y=y)
    g = m.Mavg(w1, local_lr=0.01, objective=m.OBJ_MLP, gemm_bf16=mode, learner_momentum=0.5,
               x_bf16=mode == 2, defer_broadcast=B % 2 == 0, **kw)
    kw["x"] = g.x.float().cpu().numpy()
    o = oracle.Mavg(w1, gamma=0.01, objective=oracle.OBJ_MLP, bf16=mode != 0, beta=0.5,
                    stride=g.stride, **kw)
    g.set_profiling(profiled)
    before = g.launch_count()
    g.local_steps()
    assert (g.launch_count() - before == 1) == ((dims, B, P) in SMALL)
    losses, _ = o.local_steps()
    g.sync()
    # fp32: sums of at most 3072 terms in another order, a few 1e-7 each; bf16 operands: a sum that
    # rounds to the other neighbour moves an operand by 4e-3 of itself (2e-2 per step is the gate of
    # the whole-step comparisons)
    tol = 2e-5 if mode == 0 else 2e-2
    assert np.abs(g.get_losses() - losses).max() <= tol * np.abs(losses).max()
    u, rep = g.u.cpu().numpy(), g.replicas.cpu().numpy()
    # every weight matrix and every bias on its own: an operand that rounds to the other neighbour moves by
    # 2^-8 of itself, so a gradient does not move by more even where all its operands do
    part = 2e-5 if mode == 0 else 4e-3
    for j in range(P):
        for w_off, rows, cols, b_off in mlp_layout(dims):
            for at, size in ((w_off, rows * cols), (b_off, rows)):
                assert l2_rel(u[j, at:at + size], o.u[j, at:at + size]) <= part
        assert l2_rel(u[j, :g.n], o.u[j, :g.n]) <= tol
        assert l2_rel(rep[j, :g.n], o.replicas[j, :g.n]) <= 0.1 * tol
    g.close()
