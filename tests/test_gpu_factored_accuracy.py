"""Rounds in factored form are no further from 64 bits than rounds that step each learner's own weights: both
forms round their operands to bf16, but the first rounds the weights once for all steps, learners and samples,
so nothing of that rounding averages out.  Centred inputs, inputs in [0, 1] and non-negative ones."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
LR, SEEDS = 0.002, 6


def _inputs(dims, kind, seed):
    import paper_2110_00625_b200 as m
    rng = np.random.default_rng(100 + seed)
    x = torch.from_numpy(rng.standard_normal((4096, dims[0]), dtype=np.float32))
    y = (x @ torch.from_numpy(rng.standard_normal((dims[0], dims[-1]), dtype=np.float32))).argmax(1)
    x = {"centred": x, "unit": torch.sigmoid(1.5 * x), "positive": torch.relu(x)}[kind].bfloat16()
    return m.workloads.mlp_init(dims, seed=seed), x, y.to(torch.int32)


def _exact(dims, P, K, w1, g):
    """v (the mean displacement) and the mean loss in float64."""
    L, x, y = len(dims) - 1, g.x.double(), g.y.long()
    w1 = torch.from_numpy(w1).cuda().double()
    total, losses = torch.zeros_like(w1), []
    for j in range(P):
        w = w1.clone()
        for k in range(1, K + 1):
            i = torch.from_numpy(g.get_batch_indices(1, j, k).astype(np.int64)).cuda()
            leaf = w.clone().requires_grad_(True)
            a, off = x[i], 0
            for l in range(L):
                W = leaf[off:off + dims[l + 1] * dims[l]].view(dims[l + 1], dims[l])
                off += W.numel()
                a = a @ W.T + leaf[off:off + dims[l + 1]]
                off += dims[l + 1]
                if l < L - 1:
                    a = torch.relu(a)
            loss = torch.nn.functional.cross_entropy(a, y[i])
            loss.backward()
            losses.append(loss.item())
            w = w - LR * leaf.grad
        total += w - w1
    return total / P, float(np.mean(losses))


@pytest.mark.parametrize("dims,P,K,B", [([1000, 312, 10], 40, 4, 80), ([520, 200, 136, 12], 20, 9, 48),
                                        ([1032, 1000, 520, 264, 10], 26, 5, 64)])
@pytest.mark.parametrize("kind", ["centred", "unit", "positive"])
def test_no_further_from_64_bits_than_the_plain_form(dims, P, K, B, kind):
    import paper_2110_00625_b200 as m
    err = {0: [], 2: []}
    for seed in range(SEEDS):
        w1, x, y = _inputs(dims, kind, seed)
        want = None
        for schedule in err:
            g = m.Mavg(w1, P=P, K=K, local_lr=LR, mu=0.9, B=B, seed=seed, objective=m.OBJ_MLP, dims=dims, gemm_bf16=1,
                       x=x, y=y, x_bf16=True)
            g.set_schedule(schedule)
            assert g.factored() == (schedule == 0)
            if want is None:
                want = _exact(dims, P, K, w1, g)
            loss = g.round(want_loss=True)
            err[schedule].append(((g.v.double() - want[0]).norm().item() / want[0].norm().item(), loss - want[1]))
            g.close()
    fac, plain = (np.sqrt(np.mean(np.square(err[s]), axis=0)) for s in (0, 2))
    # root mean square over the seeds: v and the mean loss
    assert (fac <= plain).all(), (fac, plain)
