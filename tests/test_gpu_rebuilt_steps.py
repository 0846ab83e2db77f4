"""Rebuilt local steps (weights formed anew each step from w~, u and the steps' rows) are the plain form's, which steps each
learner's weights in place, to the bit: one and several row and column tiles, ragged ones, batches of whole and part slabs, u
zero, reset and carried over, more steps than accumulators; first steps of all learners at once, products split over a
cluster or over blocks, forward products that ride on the plain form's weight gradients, the fused last layer."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(dims, P, K, B, beta, reset, defer, calls, rebuilt, how, odd=(), with_u=False):
    """The state after `calls`.  The plain form of the same settings: a handle made for one step (how == "steps"), without
    the momentum that would make it one for rebuilt steps ("momentum"), or the plain tiles where these sum alike ("tiles")."""
    import paper_2110_00625_b200 as m
    gen = torch.Generator(device="cuda").manual_seed(0)
    x = torch.randn(4000, dims[0], generator=gen, device="cuda")
    y = torch.randint(0, dims[-1], (4000,), generator=gen, device="cuda").int()
    w1 = m.workloads.mlp_init(dims)
    for at, value in odd:
        w1[at] = value
    late_momentum, late_steps = not rebuilt and how == "momentum", not rebuilt and how == "steps"
    g = m.Mavg(w1, P=P, K=1 if late_steps else K, local_lr=0.002, mu=0.9, B=B, seed=3,
               objective=m.OBJ_MLP, dims=dims, gemm_bf16=1, x=x, y=y, x_bf16=True, defer_broadcast=defer,
               learner_momentum=0.0 if late_momentum else beta, learner_momentum_reset=reset, with_learner_u=with_u or beta != 0)
    if late_steps:
        g.set_hparams(K, 0.002, 1.0, 0.9)
    if late_momentum:
        g.set_learner_momentum(beta, reset)
    if not rebuilt and how == "tiles":
        g.set_schedule(2)
    assert g.rebuilt() == rebuilt and not g.factored()
    calls(g)
    g.sync()
    out = [g.v.clone(), g.w.clone(), g.replicas[:, :g.n].clone(), torch.from_numpy(g.get_losses().copy())]
    if beta:
        out.append(g.u[:, :g.n].clone())
    g.close()
    return out


def _rounds(g):
    g.round()
    g.round()


def _steps_from_own_weights(g):                   # the second call does not start from w~
    g.round()
    g.local_steps()
    g.local_steps()


@pytest.mark.parametrize("dims,P,K,B,beta,reset,defer,calls,how", [
    ([520, 264, 136, 10], 118, 3, 16, 0.9, False, True, _rounds, "momentum"),
    ([520, 264, 136, 10], 170, 2, 16, 0.9, True, False, _rounds, "momentum"),
    ([520, 264, 136, 10], 167, 4, 80, 0.5, False, False, _rounds, "momentum"),
    ([1000, 520, 32], 55, 2, 48, 0.9, False, True, _steps_from_own_weights, "momentum"),
    ([784, 128, 3], 281, 2, 256, 0.9, False, False, _rounds, "momentum"),
    ([3072, 1024, 512, 10], 10, 4, 64, 0.9, False, True, _rounds, "momentum"),
    ([2424, 776, 32], 18, 3, 48, 0.9, False, True, _rounds, "momentum"),
    ([2048, 2048, 2048, 10], 13, 2, 144, 0.9, False, False, _rounds, "steps"),
    ([3072, 2048, 2048, 2048, 10], 8, 4, 64, 0.9, False, True, _rounds, "steps"),
    ([2056, 1000, 32], 24, 2, 160, 0.0, False, True, _rounds, "tiles"),
    ([1120, 1304, 1304, 1304, 10], 10, 6, 16, 0.0, False, True, _rounds, "steps"),
    ([1352, 1984, 1984, 1984, 10], 9, 6, 48, 0.0, False, False, _rounds, "steps"),
    ([1416, 1800, 1800, 1800, 32], 7, 2, 48, 0.0, False, True, _steps_from_own_weights, "steps"),
    ([3072, 2048, 2048, 2048, 10], 8, 3, 64, 0.0, False, True, _rounds, "steps"),
    ([2488, 608, 608, 32], 27, 2, 48, 0.0, False, False, _rounds, "steps"),
    ([3072, 1024, 512, 10], 14, 4, 16, 0.0, False, True, _rounds, "steps"),          # riding products in partial sums
    ([2816, 1184, 1184, 1184, 10], 24, 2, 96, 0.0, False, False, _rounds, "steps"),
    ([3072, 2048, 10], 13, 4, 16, 0.9, False, True, _rounds, "steps"),                # some rows whole, the others not
    ([3048, 1000, 504, 264, 10], 13, 3, 32, 0.9, False, True, _rounds, "steps"),      # ragged
    ([1632, 1024, 512, 10], 24, 2, 32, 0.9, False, True, _rounds, "steps"),           # runs of an odd number of tiles
])
def test_the_steps_are_the_plain_ones(dims, P, K, B, beta, reset, defer, calls, how):
    got, want = (_run(dims, P, K, B, beta, reset, defer, calls, rebuilt, how) for rebuilt in (True, False))
    for a, b in zip(got, want):
        assert torch.equal(a, b)


def _profiled(g):
    g.set_profiling(True)
    _rounds(g)


@pytest.mark.parametrize("dims,P,K,B,beta,how", [([3072, 1024, 512, 10], 10, 4, 64, 0.9, "momentum"),
                                                 ([1120, 1304, 1304, 1304, 10], 10, 6, 16, 0.0, "steps")])
def test_launch_by_launch_and_with_a_buffer_for_momentum(dims, P, K, B, beta, how):
    want = _run(dims, P, K, B, beta, False, True, _rounds, False, how)
    for calls, with_u in ((_profiled, False), (_rounds, True)):
        for a, b in zip(_run(dims, P, K, B, beta, False, True, calls, True, how, with_u=with_u), want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("dims,P,K,B,beta,how", [([3072, 1024, 512, 10], 10, 3, 64, 0.9, "momentum"),
                                                 ([1416, 1800, 1800, 1800, 32], 7, 2, 48, 0.0, "steps")])
@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan"), 3.4e38])
def test_what_is_not_finite_spreads_as_in_the_plain_form(dims, P, K, B, beta, how, value):
    odd = [(7 * dims[0] + 5, value), (dims[1] * (dims[0] + 1) + 11 * dims[1] + 3, value)]   # in W_1 and W_2
    got, want = (_run(dims, P, K, B, beta, False, True, lambda g: g.round(), rebuilt, how, odd) for rebuilt in (True, False))
    assert not all(torch.isfinite(t).all() for t in want)
    for a, b in zip(got, want):
        assert torch.equal(a.isnan(), b.isnan()) and torch.equal(a.nan_to_num(nan=0.0), b.nan_to_num(nan=0.0))


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
