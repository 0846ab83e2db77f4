"""Products of the CUDA-core path with bf16 operands form long sums as exactly as fp32 sums rounded to nearest.
The operands are chosen so that they are exact in bf16: all that is left is how the products are added."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _handle(dims, w1, x, y, B, mode=2):
    import paper_2110_00625_b200 as m
    g = m.Mavg(w1, P=1, K=1, local_lr=1.0, mu=0.0, B=B, seed=3, objective=m.OBJ_MLP, dims=dims, gemm_bf16=mode, x=x, y=y)
    return g, g.get_batch_indices(1, 0, 1).astype(np.int64)


def _step(g):
    g.local_steps()
    g.sync()
    row = g.replicas[0, :g.n].cpu().numpy().astype(np.float64)
    g.close()
    return row


def _check(got, want, size, adds, chained):
    # in units of 2^-24 of the sum: each of `adds` additions rounds to nearest, either way, by half a unit at most, and
    # they add up as their root.  A chain of 16 products at a time in a matrix instruction's accumulator cuts off what
    # falls behind the last place, all the same way: up to two units a link.
    rms = np.sqrt(np.mean(((got - want) / size) ** 2)) * 2 ** 24
    assert rms <= np.sqrt(adds) / 2 + 2 * chained / 16, rms


@pytest.mark.parametrize("B", [60, 512, 513, 3000, 12000])
def test_weight_gradient_over_a_long_batch(B):
    # one layer from zero weights: p = 1/8, so dZ is bf16(2^-3 / B) for the classes that no sample has
    rng = np.random.default_rng(1)
    dims = [640, 8]
    x = torch.from_numpy(rng.uniform(0.5, 1.0, (8192, 640)).astype(np.float32)).bfloat16().float().numpy()
    y = rng.integers(0, 4, 8192).astype(np.int32)
    g, i = _handle(dims, np.zeros(641 * 8, np.float32), x, y, B)
    w = -_step(g)[:640 * 8].reshape(8, 640)[4:]
    dz = float(torch.tensor(0.125 / B).bfloat16())
    want = np.broadcast_to(dz * x[i].astype(np.float64).sum(0), w.shape)
    # 32 samples to an addition beyond 512, and chains of 32; up to there one chain
    _check(w, want, want, B / 32 if B > 512 else 0, 32 if B > 512 else B)


@pytest.mark.parametrize("C", [90, 1000])
def test_data_gradient_over_many_classes(C):
    # one sample whose hidden activations are next to nothing: p = 1 / C, and the step of b_1 is -dZ_1
    rng = np.random.default_rng(2)
    dims = [32, 24, C]
    x = rng.uniform(0.5, 1.0, (64, 32)).astype(np.float32)
    y = rng.integers(0, C, 64).astype(np.int32)
    W2 = torch.from_numpy(rng.uniform(0.5, 1.0, (C, 24)).astype(np.float32)).bfloat16().float().numpy()
    tiny = 2.0 ** -40
    w1 = np.concatenate([np.zeros(32 * 24), np.full(24, tiny), W2.reshape(-1), np.zeros(C)]).astype(np.float32)
    g, i = _handle(dims, w1, x, y, 1)
    db = -_step(g)[32 * 24:33 * 24]
    label = int(y[i[0]])
    dz = torch.full((C,), 1.0 / C, dtype=torch.float64)
    dz[label] -= 1.0
    dz = dz.float().bfloat16().double().numpy()
    terms = dz[:, None] * W2.astype(np.float64)
    _check(db, terms.sum(0), np.abs(terms).sum(0), C / 64, 64)


@pytest.mark.parametrize("B", [64, 100, 128, 129, 160, 192, 193, 256, 257, 300, 1000])
def test_fp32_weight_gradient_no_further_off_than_a_chain_of_fmas(B):
    # one layer from zero weights: dZ is the same for all samples and the classes that none of them has, so the gradient is a
    # sum of like terms, whose cut-off errors all go the same way
    rng = np.random.default_rng(4)
    dims = [640, 8]
    x = rng.uniform(0.0, 1.0, (8192, 640)).astype(np.float32)
    y = rng.integers(0, 4, 8192).astype(np.int32)
    g, i = _handle(dims, np.zeros(641 * 8, np.float32), x, y, B, mode=0)
    w = -_step(g)[:640 * 8].reshape(8, 640)[4:]
    dz = float(np.float32(0.125) * (np.float32(1.0) / np.float32(B)))
    want = dz * x[i].astype(np.float64).sum(0)
    chain = np.zeros(640, np.float32)
    for row in x[i]:
        chain = (chain + dz * row.astype(np.float64)).astype(np.float32)

    def off(a):
        return np.sqrt(np.mean(((a - want) / want) ** 2))

    # What a chain of two slabs loses where a few samples more begin a second: B = 160 1.05 times as much as the chain of FMAs
    # (a rounded one is the same sum in expectation, and this is one draw of 640); 1.3 with three or four slabs to a chain.
    assert off(w) <= 1.15 * off(chain), (off(w) * 2 ** 24, off(chain) * 2 ** 24)
