"""The one-launch pseudo-gradient round against its two halves called one after the other: the same
bits in w~, v, the replicas and the learner momentum."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
SMS = 148


def _handle(n, P, K, **kw):
    import paper_2110_00625_b200 as m
    return m.Mavg(m.workloads.global_model(n), P=P, K=K, local_lr=0.05, block_lr=0.7, seed=11,
                  objective=m.OBJ_PSEUDOGRAD, sigma=0.1, **kw)


def _state(g):
    g.sync()
    out = [g.w, g.v, g.replicas[:, :g.n]] + ([g.u[:, :g.n]] if g.u is not None else [])
    return [t.cpu().numpy().view(np.uint32) for t in out]


# (n, K): both sides of the size rule for few and for many steps, blocks of 64 and of 256 threads,
# every remainder of n by 4, a last block of one quad
@pytest.mark.parametrize("n,K", [(512 * SMS - 1, 1), (512 * SMS, 4), (512 * SMS + 1, 1),
                                 (4096 * SMS - 2, 5), (4096 * SMS + 3, 5), (8192 * SMS + 2, 1),
                                 (8192 * SMS + 1028, 3)])
@pytest.mark.parametrize("kw", [dict(mu=0.9), dict(mu=0.0, defer_broadcast=True),
                                dict(mu=0.9, defer_broadcast=True, learner_momentum=0.9),
                                dict(mu=0.5, learner_momentum=0.5, learner_momentum_reset=True)])
def test_round_is_local_steps_then_meta_update(n, K, kw):
    a, b = _handle(n, 5, K, **kw), _handle(n, 5, K, **kw)
    for r in range(3):
        if r == 2:                       # a round that starts from diverged replicas
            a.local_steps(); b.local_steps()
        a.round()
        b.local_steps(); b.meta_update()
        assert a.get_round() == b.get_round()
        for x, y in zip(_state(a), _state(b)):
            assert np.array_equal(x, y)
    a.close(); b.close()


def test_more_step_keys_than_the_fused_round_holds():
    # P K = 4095, 4096 and 4100: the last takes the two launches
    for P, K in ((63, 65), (64, 64), (41, 100)):
        a, b = _handle(8192 * SMS + 1, P, K, mu=0.9), _handle(8192 * SMS + 1, P, K, mu=0.9)
        before = a.launch_count()
        a.round()
        assert a.launch_count() - before == (1 if P * K <= 4096 else 2)
        b.local_steps(); b.meta_update()
        for x, y in zip(_state(a), _state(b)):
            assert np.array_equal(x, y)
        a.close(); b.close()
        torch.cuda.empty_cache()


# both sides of every line of the rule: n, P, K, learner momentum, launches
@pytest.mark.parametrize("n,P,K,beta,launches", [
    (512 * SMS - 1, 3, 1, 0.0, 2), (512 * SMS, 3, 1, 0.0, 1), (512 * SMS, 300, 1, 0.0, 1),
    (512 * SMS, 32, 2, 0.0, 1), (640 * SMS - 1, 33, 2, 0.0, 2), (640 * SMS, 33, 2, 0.0, 1),
    (512 * SMS, 16, 4, 0.0, 1), (512 * SMS, 17, 4, 0.0, 2), (1024 * SMS - 1, 17, 4, 0.0, 2),
    (1024 * SMS, 17, 4, 0.0, 1), (1024 * SMS, 512, 4, 0.0, 1), (1024 * SMS, 513, 4, 0.0, 2),
    (1024 * SMS, 1001, 3, 0.0, 1),
    (4096 * SMS - 1, 2, 5, 0.0, 2), (4096 * SMS, 2, 24, 0.0, 1), (4096 * SMS, 2, 25, 0.0, 2),
    (6144 * SMS - 1, 2, 25, 0.0, 2), (6144 * SMS, 2, 25, 0.0, 1),
    (6144 * SMS, 32, 64, 0.0, 1), (6144 * SMS, 33, 64, 0.0, 2), (8192 * SMS, 33, 64, 0.0, 1),
    (512 * SMS, 48, 1, 0.9, 1), (512 * SMS, 49, 1, 0.9, 2), (512 * SMS, 16, 3, 0.9, 1), (512 * SMS, 17, 3, 0.9, 2),
    (512 * SMS, 8, 4, 0.9, 1), (512 * SMS, 9, 4, 0.9, 2), (1024 * SMS, 16, 4, 0.9, 1),
    (1024 * SMS, 17, 4, 0.9, 2), (2048 * SMS - 1, 17, 4, 0.9, 2), (2048 * SMS, 17, 4, 0.9, 1),
    (4096 * SMS, 2, 5, 0.9, 1)])
def test_where_a_round_is_one_launch(n, P, K, beta, launches):
    g = _handle(n, P, K, mu=0.9, defer_broadcast=True, learner_momentum=beta)
    before = g.launch_count()
    g.round()
    assert g.launch_count() - before == launches
    g.close()
    torch.cuda.empty_cache()
