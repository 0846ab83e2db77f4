"""Products of fp32 models and of bf16 operands in any shape (csrc/split_gemm.cuh) where their kernels change form: two
batch tiles, batches beyond one accumulator of a weight gradient, tiles of 64 and of 128 outputs, rows that are no whole
pairs, a last layer of several launches; and infinite weights."""
import numpy as np
import pytest

from tests.util import l2_rel, mlp_layout

pytestmark = pytest.mark.gpu

SHAPES = [                                  # dims, B, P
    ([700, 140, 7], 129, 2),                # two batch tiles, the second of one sample's group
    ([301, 131, 66, 5], 257, 2),            # just beyond one accumulator, odd rows
    ([300, 260, 9], 256, 1),                # the largest batch of one
    ([640, 1100, 70], 40, 4),               # tiles of 128 outputs, 70 of the last layer's
    ([1024, 512, 130], 24, 1),              # last layer of several launches, two tiles of classes
    ([129, 65, 200, 3], 530, 1),            # many slabs, five batch tiles
]


def _pair(oracle, mode, dims, B, P, beta, w1=None, x=None, K=2):
    import paper_2110_00625_b200 as m
    rng = np.random.default_rng(B)
    S = 60 * P + 7
    x = rng.standard_normal((S, dims[0]), dtype=np.float32) if x is None else x
    y = rng.integers(0, dims[-1], size=len(x)).astype(np.int32)
    w1 = m.workloads.mlp_init(dims) if w1 is None else w1
    kw = dict(P=P, K=K, mu=0.9, B=B, seed=11, dims=dims, x=x, y=y)
    g = m.Mavg(w1, local_lr=0.01, objective=m.OBJ_MLP, gemm_bf16=mode, learner_momentum=beta, defer_broadcast=P == 1, **kw)
    o = oracle.Mavg(w1, gamma=0.01, objective=oracle.OBJ_MLP, bf16=mode != 0, beta=beta, stride=g.stride, **kw)
    return g, o


@pytest.mark.parametrize("beta", [0.0, 0.5])
@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("dims,B,P", SHAPES)
def test_two_steps(oracle, mode, dims, B, P, beta):
    g, o = _pair(oracle, mode, dims, B, P, beta)
    start = o.replicas[:, :g.n].astype(np.float64)
    g.local_steps()
    losses, _ = o.local_steps()
    g.sync()
    assert l2_rel(g.get_losses(), losses) <= (1e-6 if mode == 0 else 2e-3)
    # The steps themselves, every weight matrix and bias on its own.  fp32: a sum of n like terms in fp32 is off by at
    # most sqrt(n) 2^-24 of itself, here n <= 1100 and three products in a row; the oracle's and the learners' weights are
    # rounded to 2^-24 of themselves, which is the larger part of a step's difference without the momentum buffer.  bf16
    # operands: one that rounds to the other neighbour moves by 2^-8 of itself.
    got = g.u.cpu().numpy() if beta else g.replicas.cpu().numpy()
    want = o.u if beta else o.replicas
    for j in range(P):
        for w_off, rows, cols, b_off in mlp_layout(dims):
            for at, size in ((w_off, rows * cols), (b_off, rows)):
                base = np.zeros(size) if beta else start[j, at:at + size]
                a, b = got[j, at:at + size] - base, want[j, at:at + size] - base
                noise = 0.0 if beta else 2 ** -23 * np.linalg.norm(base) / np.linalg.norm(b)
                assert l2_rel(a, b) <= (6e-6 if mode == 0 else 4e-3) + noise
    g.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, 3.4e38])
@pytest.mark.parametrize("dims,B,P", [([300, 200, 10], 32, 2), ([301, 200, 70, 10], 300, 1)])
def test_infinite_weights_reach_no_more_than_their_own_unit(oracle, dims, B, P, value):
    # a unit of layer 1 whose pre-activation is -inf for every sample is dead; what its weight's smaller parts would add
    # to the sum is NaN
    import paper_2110_00625_b200 as m
    x = np.random.default_rng(3).standard_normal((100, dims[0])).astype(np.float32)
    x[:, 5] = -np.sign(value) * (2.0 + np.abs(x[:, 5]))
    w1 = m.workloads.mlp_init(dims)
    w1[7 * dims[0] + 5] = value
    g, o = _pair(oracle, 0, dims, B, P, 0.0, w1, x)
    g.local_steps()
    losses, _ = o.local_steps()
    g.sync()
    assert np.isfinite(losses).all() and l2_rel(g.get_losses(), losses) <= 1e-6
    rep, want = g.replicas[:, :g.n].cpu().numpy(), o.replicas[:, :g.n]
    at = 7 * dims[0] + 5
    assert (rep[:, at] == np.float32(value)).all() and (want[:, at] == np.float32(value)).all()
    rep[:, at] = 0.0
    want = want.copy()
    want[:, at] = 0.0
    assert l2_rel(rep, want) <= 1e-6
    g.close()


@pytest.mark.parametrize("value", [3.4e38, -3.4e38, np.finfo(np.float32).max])
@pytest.mark.parametrize("dims,B,P", [([300, 200, 70, 10], 32, 2), ([301, 200, 70, 10], 300, 1)])
def test_the_largest_fp32_values_are_finite_ones(oracle, dims, B, P, value):
    # above 3.39e38 a value rounds to a bf16 infinity, whose product with a zero is NaN: weights of layers 1 and 2 whose
    # inputs are zero (where they are not, the unit is dead), and inputs whose weights are
    import paper_2110_00625_b200 as m
    x = np.random.default_rng(3).standard_normal((100, dims[0])).astype(np.float32)
    x[0::2, 5] = 0.0
    x[1::2, 5] = -1e-30 * np.sign(value)
    x[0::3, 9] = value
    w1 = m.workloads.mlp_init(dims)
    W1, b1 = w1[:dims[1] * dims[0]].reshape(dims[1], dims[0]), w1[dims[1] * dims[0]:][:dims[1]]
    W2 = w1[dims[1] * (dims[0] + 1):][:dims[2] * dims[1]].reshape(dims[2], dims[1])
    W1[7, 5] = W2[3, 11] = value
    W1[:, 9] = 0.0
    b1[11] = -1e9                                # unit 11 is dead
    g, o = _pair(oracle, 0, dims, B, P, 0.0, w1, x, K=1)
    g.local_steps()
    losses, _ = o.local_steps()
    g.sync()
    assert np.isfinite(losses).all() and l2_rel(g.get_losses(), losses) <= 1e-6
    rep, want = g.replicas[:, :g.n].cpu().numpy(), o.replicas[:, :g.n].copy()
    large = [np.flatnonzero(w1 == np.float32(value)), np.arange(dims[1]) * dims[0] + 9]
    assert (rep[:, large[0]] == np.float32(value)).all() and (want[:, large[0]] == np.float32(value)).all()
    assert np.abs(want[:, large[1]]).max() > 1e30 and l2_rel(rep[:, large[1]], want[:, large[1]]) <= 6e-6   # a step, as above
    for at in large + [np.array([dims[1] * dims[0] + 11])]:
        rep[:, at] = want[:, at] = 0.0
    assert l2_rel(rep, want) <= 1e-6
    g.close()
