"""Whole rounds on the CUDA cores, both forms of the learner level (all steps in one launch, and a launch
per product replayed from a graph), against the oracle: where the learners start from, and local steps
called twice in a row."""
import numpy as np
import pytest
import torch

from tests.util import l2_rel

pytestmark = pytest.mark.gpu

# small: at most 4096 parameters, all K steps are one launch; large: a graph of launches per product
SMALL, LARGE = [64, 48, 10], [300, 200, 10]


def _pair(oracle, mode, dims, P=3, K=3, B=16, beta=0.0, **kw):
    import paper_2110_00625_b200 as m
    rng = np.random.default_rng(17)
    x = rng.standard_normal((1000, dims[0]), dtype=np.float32)
    y = rng.integers(0, dims[-1], size=1000).astype(np.int32)
    w1 = m.workloads.mlp_init(dims)
    common = dict(P=P, K=K, mu=0.9, B=B, seed=5, dims=dims, x=x, y=y)
    g = m.Mavg(w1, local_lr=0.01, objective=m.OBJ_MLP, gemm_bf16=mode, learner_momentum=beta, **common, **kw)
    o = oracle.Mavg(w1, gamma=0.01, objective=oracle.OBJ_MLP, bf16=mode != 0, beta=beta, stride=g.stride,
                    **common)
    return g, o


def _tol(mode):
    # a few steps of fp32 sums in another order / of bf16 operands that round to the other neighbour:
    # the drift of the weights themselves stays a tenth of the 2e-5 / 2e-2 a step's gradient may have
    return 2e-6 if mode == 0 else 2e-3


def _steps_launches(g):
    before = g.launch_count()
    g.local_steps()
    return g.launch_count() - before


@pytest.mark.parametrize("defer", [False, True])
@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("mode", [0, 2])
def test_rows_edited_between_rounds_are_where_the_learners_start(oracle, mode, dims, defer):
    # a program that perturbs the learners' copies of w~ at a round boundary (written on request where
    # the re-broadcast is deferred): in the first round, in a replayed one, and not after it
    g, o = _pair(oracle, mode, dims, defer_broadcast=defer)
    rng = np.random.default_rng(23)
    for r in range(4):
        if r != 2:
            if defer:
                g.materialize_replicas()
            noise = 0.1 * rng.standard_normal((3, g.n), dtype=np.float32)
            g.replicas[:, :g.n] += torch.from_numpy(noise).to(g.device)
            o.replicas[:, :g.n] += noise
        launches = _steps_launches(g)
        assert (launches == 1) == (dims is SMALL)
        losses, _ = o.local_steps()
        g.sync()
        rep = g.replicas[:, :g.n].cpu().numpy()
        for j in range(3):
            assert l2_rel(rep[j], o.replicas[j, :g.n]) <= (r + 1) * _tol(mode)
        assert l2_rel(g.get_losses(), losses) <= 10 * (r + 1) * _tol(mode)
        g.meta_update()
        o.meta_update()
        g.sync()
        assert l2_rel(g.w.cpu().numpy(), o.w) <= (r + 1) * _tol(mode)
    g.close()


@pytest.mark.parametrize("beta", [0.0, 0.9])
@pytest.mark.parametrize("defer", [False, True])
@pytest.mark.parametrize("dims", [SMALL, LARGE])
@pytest.mark.parametrize("mode", [0, 2])
def test_local_steps_twice_in_a_row(oracle, mode, dims, defer, beta):
    # the second call goes on from the learners' own models and momentum; two such rounds
    g, o = _pair(oracle, mode, dims, beta=beta, defer_broadcast=defer)
    for r in range(2):
        for _ in range(2):
            assert (_steps_launches(g) == 1) == (dims is SMALL)
            losses, _ = o.local_steps()
            g.sync()
            assert l2_rel(g.get_losses(), losses) <= 10 * (r + 1) * _tol(mode)
        rep = g.replicas[:, :g.n].cpu().numpy()
        for j in range(3):
            assert l2_rel(rep[j], o.replicas[j, :g.n]) <= (r + 1) * _tol(mode)
            if beta:
                # the buffers hold the gradients themselves
                assert l2_rel(g.u[j, :g.n].cpu().numpy(), o.u[j, :g.n]) <= 10 * (r + 1) * _tol(mode)
        g.meta_update()
        o.meta_update()
        g.sync()
        assert l2_rel(g.w.cpu().numpy(), o.w) <= (r + 1) * _tol(mode)
        assert l2_rel(g.v.cpu().numpy(), o.v) <= 10 * (r + 1) * _tol(mode)
    g.close()


@pytest.mark.parametrize("mode", [0, 2])
def test_rows_beyond_the_batch_take_no_part(oracle, mode):
    # Hidden unit 0 is dead for every sample but would be alive for a row of zeros, and an infinite weight
    # hangs on it: 0 x inf is no number, ReLU makes it zero, and everything stays finite.  The batch of 5
    # leaves 3 rows of the last group of four that must not bring the infinity in.
    import paper_2110_00625_b200 as m
    dims, P, B = [4, 2, 2, 3], 2, 5
    rng = np.random.default_rng(2)
    x = np.abs(rng.standard_normal((40, 4), dtype=np.float32)) + 0.1
    y = rng.integers(0, 3, size=40).astype(np.int32)
    w1 = (0.3 * rng.standard_normal(10 + 6 + 9)).astype(np.float32)
    w1[0:4] = -100.0                     # W_1's first row
    w1[8] = 1.0                          # its bias
    w1[10] = np.inf                      # W_2[0, 0]
    kw = dict(P=P, K=2, mu=0.9, B=B, seed=4, dims=dims, x=x, y=y)
    g = m.Mavg(w1, local_lr=0.01, objective=m.OBJ_MLP, gemm_bf16=mode, **kw)
    o = oracle.Mavg(w1, gamma=0.01, objective=oracle.OBJ_MLP, bf16=mode != 0, stride=g.stride, **kw)
    assert _steps_launches(g) == 1
    losses, _ = o.local_steps()
    g.sync()
    assert np.isfinite(losses).all() and l2_rel(g.get_losses(), losses) <= 10 * _tol(mode)
    rep, want = g.replicas[:, :g.n].cpu().numpy(), o.replicas[:, :g.n]
    finite = np.isfinite(want)
    assert np.array_equal(np.isfinite(rep), finite) and finite.sum() == P * (g.n - 1)
    assert l2_rel(rep[finite], want[finite]) <= _tol(mode)
    g.close()
