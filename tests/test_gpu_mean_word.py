"""The pinned words that rounds leave their mean loss in: a handle gives its own back without waiting for the stream, and one
that finds none free has the mean copied back."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DIMS = [8, 4]


def _handles(n, **kw):
    import paper_2110_00625_b200 as m
    x, y = torch.randn(64, DIMS[0], device="cuda"), torch.randint(0, DIMS[1], (64,), device="cuda").int()
    w1 = m.workloads.mlp_init(DIMS)
    return [m.Mavg(w1, P=2, K=2, local_lr=0.1, mu=0.9, B=4, seed=i, objective=m.OBJ_MLP, dims=DIMS, x=x, y=y, **kw)
            for i in range(n)]


def test_destroying_a_handle_does_not_wait_for_its_stream():
    s = torch.cuda.Stream()
    g, = _handles(1, stream=s)
    g.round(want_loss=True)
    done = torch.cuda.Event()
    with torch.cuda.stream(s):
        torch.cuda._sleep(400_000_000)            # about 0.2 s
        done.record()
    g.close()
    assert not done.query()
    s.synchronize()


def test_more_handles_than_words():
    handles = _handles(1030)
    for _ in range(2):
        for g in handles:
            mean = g.round(want_loss=True)
            assert abs(mean - g.get_losses().astype(np.float64).mean()) <= 1e-6 * abs(mean)
    for g in handles:
        g.close()
    g, = _handles(1)                              # and the words are there again
    mean = g.round(want_loss=True)
    assert abs(mean - g.get_losses().astype(np.float64).mean()) <= 1e-6 * abs(mean)
    g.close()
