"""Rebuilt local steps (weights formed anew each step from w~, u and the steps' rows) against the plain form, which steps
each learner's weights in place: one and several row and column tiles, ragged ones, batches of whole and part slabs, one
accumulator buffer and two, u zero, reset and carried over."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _pair(dims, P, K, B, beta, reset, defer, calls, seed=0):
    import paper_2110_00625_b200 as m
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(4000, dims[0], generator=gen, device="cuda")
    y = torch.randint(0, dims[-1], (4000,), generator=gen, device="cuda").int()
    w1 = m.workloads.mlp_init(dims, seed=seed)
    out = []
    for schedule in (0, 2):
        g = m.Mavg(w1, P=P, K=K, local_lr=0.002, mu=0.9, B=B, seed=3, objective=m.OBJ_MLP, dims=dims, gemm_bf16=1, x=x, y=y,
                   x_bf16=True, defer_broadcast=defer, learner_momentum=beta, learner_momentum_reset=reset)
        g.set_schedule(schedule)
        assert g.rebuilt() == (schedule == 0)
        calls(g)
        g.sync()
        out.append((g.v.clone(), g.w.clone(), g.replicas[:, :g.n].clone(),
                    g.u[:, :g.n].clone() if beta else g.v.clone(), torch.from_numpy(g.get_losses().copy())))
        g.close()
    return [((a.double() - b.double()).norm() / b.double().norm()).item() for a, b in zip(*out)]


def _rounds(g):
    g.round()
    g.round()


def _steps_from_own_weights(g):                   # the second call does not start from w~
    g.round()
    g.local_steps()
    g.local_steps()


@pytest.mark.parametrize("dims,P,K,B,beta,reset,defer,calls", [
    ([520, 264, 136, 10], 118, 3, 16, 0.9, False, True, _rounds),
    ([520, 264, 136, 10], 170, 2, 16, 0.9, True, False, _rounds),
    ([520, 264, 136, 10], 167, 4, 80, 0.5, False, False, _rounds),
    ([1000, 520, 32], 55, 2, 48, 0.9, False, True, _steps_from_own_weights),
    ([784, 128, 3], 281, 2, 256, 0.9, False, False, _rounds),
    ([2048, 2048, 2048, 10], 13, 2, 144, 0.9, False, False, _rounds),
    ([3072, 2048, 2048, 2048, 10], 8, 4, 64, 0.9, False, True, _rounds),
])
def test_with_momentum_the_steps_are_the_plain_ones(dims, P, K, B, beta, reset, defer, calls):
    # The same fp32 steps in the same order, from sums whose terms are the same: the order of a sum's parts differs in a
    # few places (1e-7 of a gradient), and where that moves a weight across a bf16 rounding boundary (1 in 2^15 of them, a
    # 2^-9 of the weight) the next step's gradient moves by 2^-9 2^-7.5 = 1e-5 at most.
    assert max(_pair(dims, P, K, B, beta, reset, defer, calls)) < 1e-5


@pytest.mark.parametrize("dims,P,K,B", [([2056, 512, 264, 10], 41, 6, 32), ([2056, 1000, 32], 24, 2, 160),
                                        ([3072, 1000, 520, 10], 14, 4, 128), ([3072, 2048, 2048, 2048, 10], 8, 3, 64)])
def test_without_momentum_one_step_from_the_sum_of_the_gradients(dims, P, K, B):
    # One fp32 rounding of the weights instead of K; v (the mean displacement) differs where a weight rounds to the other
    # bf16 neighbour: the two forms' spread is that of any other order of sums, 2^-8 of v at these sizes, and twice that.
    assert max(_pair(dims, P, K, B, 0.0, False, True, lambda g: g.round())) < 2 ** -7


def test_by_the_momentum_and_steps_of_now():
    import paper_2110_00625_b200 as m
    dims, P, B = [3072, 1024, 512, 10], 10, 64       # 37 M hidden weights: with momentum only
    x = torch.randn(2000, dims[0], device="cuda")
    y = torch.randint(0, dims[-1], (2000,), device="cuda").int()
    w1 = m.workloads.mlp_init(dims)
    kw = dict(P=P, local_lr=0.002, mu=0.9, B=B, seed=3, objective=m.OBJ_MLP, dims=dims, gemm_bf16=1, x=x, y=y, x_bf16=True,
              with_learner_u=True)
    g = m.Mavg(w1, K=4, learner_momentum=0.9, **kw)
    rebuilt = [g.rebuilt()]
    for beta, K in ((0.9, 3), (0.0, 4), (0.5, 4), (0.0, 2), (0.5, 1), (0.5, 6), (0.5, 2)):
        g.set_learner_momentum(beta)
        g.set_hparams(K, 0.002, 1.0, 0.9)
        rebuilt.append(g.rebuilt())
        w = g.w.clone()
        g.set_round(0)
        g.v.zero_()
        g.u.zero_()
        g.round()
        h = m.Mavg(w, K=K, learner_momentum=beta, **kw)
        h.round()
        for a, b in zip((g.w, g.v, g.replicas[:, :g.n], g.u[:, :g.n]), (h.w, h.v, h.replicas[:, :h.n], h.u[:, :h.n])):
            assert torch.equal(a, b)
        h.close()
    assert rebuilt == [True, True, False, True, False, False, False, True]
    g.close()
