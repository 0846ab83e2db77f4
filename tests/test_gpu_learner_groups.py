"""fp32 and odd-shaped models with less scratch than all learners' weight operands take: the learners take their local steps in
groups, with the same bits."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(monkeypatch, dims, mode, P, K, B, beta, defer, share):
    """share: of the way from the least scratch to all of it."""
    import paper_2110_00625_b200 as m
    lib = m.load_library()
    full, least = lib.mavg_workspace_bytes, lib.mavg_workspace_least_bytes

    def some(cfg, out):
        a, b = C.c_size_t(), C.c_size_t()
        assert full(cfg, C.byref(a)) == 0 and least(cfg, C.byref(b)) == 0
        assert b.value < a.value
        out._obj.value = b.value + int(share * (a.value - b.value))
        return 0

    monkeypatch.setattr(lib, "mavg_workspace_bytes", some)
    rng = np.random.default_rng(B)
    x = rng.standard_normal((40 * P, dims[0]), dtype=np.float32)
    y = rng.integers(0, dims[-1], size=len(x)).astype(np.int32)
    g = m.Mavg(m.workloads.mlp_init(dims), P=P, K=K, local_lr=0.01, mu=0.9, B=B, seed=5, objective=m.OBJ_MLP, dims=dims,
               gemm_bf16=mode, x=x, y=y, learner_momentum=beta, defer_broadcast=defer)
    monkeypatch.undo()
    before = g.launch_count()
    g.round()
    loss = g.round(want_loss=True)
    g.local_steps()
    g.local_steps()                                # the second does not start from w~
    g.sync()
    out = [g.w.clone(), g.v.clone(), g.replicas[:, :g.n].clone(), torch.from_numpy(g.get_losses().copy()), torch.tensor(loss)]
    if beta:
        out.append(g.u[:, :g.n].clone())
    launches = g.launch_count() - before
    g.close()
    return out, launches


@pytest.mark.parametrize("dims,mode,P,K,B,beta,defer", [
    ([301, 131, 66, 5], 0, 5, 3, 33, 0.5, True),
    ([300, 260, 90], 2, 5, 2, 150, 0.0, False),
    ([1024, 512, 130], 0, 3, 2, 24, 0.0, True),      # last layer of several launches
    ([333, 100], 2, 4, 2, 40, 0.9, False),
    ([80, 128, 16], 0, 16, 2, 48, 0.0, True),        # beyond the small-model kernel's line
])
def test_the_same_bits_in_groups(monkeypatch, dims, mode, P, K, B, beta, defer):
    want, most = _run(monkeypatch, dims, mode, P, K, B, beta, defer, 1.0)
    for share in (0.0, 0.3, 0.6):
        got, launches = _run(monkeypatch, dims, mode, P, K, B, beta, defer, share)
        assert launches > most
        for a, b in zip(got, want):
            assert torch.equal(a, b)
