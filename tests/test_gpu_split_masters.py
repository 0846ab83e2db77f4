"""Masters kept as two 16-bit halves between the steps of a call (layers whose forward product rides on
the weight-gradient launch and whose bf16 copy the data gradient reads): nothing of the fp32 value is
lost, and the round is the one that keeps fp32 masters."""
import numpy as np
import pytest

from tests.util import l2_rel

pytestmark = pytest.mark.gpu
B = 32


def _learners(dims):
    """Enough for layer 1's weight gradients to be a launch of their own (64 tiles per SM)."""
    return 13 if dims[0] > 3000 else 70


def _handle(dims, K, lr, w1=None, schedule=0, **kw):
    import paper_2110_00625_b200 as m
    rng = np.random.default_rng(7)
    x = rng.standard_normal((1024, dims[0]), dtype=np.float32)
    y = rng.integers(0, dims[-1], size=1024).astype(np.int32)
    w1 = m.workloads.mlp_init(dims) if w1 is None else w1
    # made for one step where its losses' room allows more: steps in place, not rebuilt
    late = _learners(dims) * K <= 64
    g = m.Mavg(w1, P=_learners(dims), K=1 if late else K, local_lr=lr, mu=0.9, B=B, seed=3, objective=m.OBJ_MLP, dims=dims,
               gemm_bf16=1, x=x, y=y, x_bf16=True, defer_broadcast=True, **kw)
    g.set_hparams(K, lr, 1.0, 0.9)
    assert not (late and g.rebuilt())
    g.set_schedule(schedule)
    assert g.get_step_plan()["fwd_with_wgrad"] == len(dims) - 2
    assert not g.factored()          # rounds that keep no weights between their steps
    return g


# whole tiles; ragged rows and columns in every layer, runs that end in a partial tile, and layer 2's low
# halves in layer 1's bf16 copy (in the others they take the place of the second copy of layer L-1); a
# layer 2 that finds no room and keeps fp32 masters below a split layer 3
SHAPES = [[3072, 1024, 512, 10], [3048, 1000, 504, 264, 10], [520, 1024, 1024, 512, 10]]


@pytest.mark.parametrize("dims", SHAPES)
@pytest.mark.parametrize("K", [1, 2, 5])
@pytest.mark.parametrize("beta", [0.0, 0.9])
def test_a_step_of_length_zero_keeps_every_bit(dims, K, beta):
    K = min(K, 8191 // (_learners(dims) * B))
    # local_lr = 0: w <- w + (-0) g leaves every value as it is, whatever steps it goes through;
    # values on and beside the ties of the bf16 rounding, subnormal ones and the largest below 1
    import paper_2110_00625_b200 as m
    w1 = m.workloads.mlp_init(dims)
    bits = w1.view(np.uint32).copy()
    rng = np.random.default_rng(1)
    at = rng.permutation(bits.size)[:bits.size // 4]
    low = np.array([0x8000, 0x7fff, 0x8001, 0xffff, 0, 1], dtype=np.uint32)
    bits[at] = (bits[at] & np.uint32(0xffff0000)) | low[rng.integers(0, 6, at.size)]
    bits[at[:64]] = np.uint32(0x00008000)
    bits[at[64:128]] = np.uint32(0x3f7fffff)
    bits[at[128:192]] = np.uint32(0x00000001)
    # zeros of either sign become +0: keep them out
    w1 = np.where(bits << 1 == 0, np.uint32(0x3c000000), bits).view(np.float32)
    g = _handle(dims, K, 0.0, w1=w1, learner_momentum=beta)
    for _ in range(2):               # the second call does not start from w~: its steps are in place in any case
        g.local_steps()
        g.sync()
        rep = g.replicas[:, :g.n].cpu().numpy().view(np.uint32)
        for row in rep:
            assert np.array_equal(row, w1.view(np.uint32))
    g.close()


@pytest.mark.parametrize("dims", SHAPES)
def test_same_round_as_with_fp32_masters(dims):
    # the plain schedule keeps fp32 masters throughout; the two differ in summation orders: per-round
    # drift bound of the bf16 path (5e-2), here three steps
    a, b = _handle(dims, 3, 0.002), _handle(dims, 3, 0.002, schedule=2)
    for _ in range(2):
        la, lb = a.round(want_loss=True), b.round(want_loss=True)
        assert abs(la - lb) <= 2e-2 * abs(lb)
    a.local_steps(); a.local_steps()          # the second call starts from fp32 replicas
    b.local_steps(); b.local_steps()
    a.sync(); b.sync()
    assert l2_rel(a.v.cpu().numpy(), b.v.cpu().numpy()) <= 5e-2
    n = a.n
    ra, rb = a.replicas[:, :n].cpu().numpy(), b.replicas[:, :n].cpu().numpy()
    w = a.w.cpu().numpy()
    for j in (0, -1):
        assert l2_rel(ra[j] - w, rb[j] - w) <= 5e-2
    a.close(); b.close()


def test_a_weight_that_is_not_a_number_stays_one():
    # and spreads exactly as far as it does with fp32 masters
    import paper_2110_00625_b200 as m
    dims = SHAPES[0]
    w1 = m.workloads.mlp_init(dims)
    at = dims[0] * dims[1] + dims[1] + 5 * dims[1] + 7          # in W_2
    w1[at] = np.nan
    nans = []
    for schedule in (0, 2):
        g = _handle(dims, 3, 0.002, w1=w1, schedule=schedule)
        g.round()
        g.sync()
        nans.append(np.isnan(g.w.cpu().numpy()))
        g.close()
    assert nans[0][at] and np.array_equal(nans[0], nans[1])


@pytest.mark.parametrize("dims", SHAPES)
@pytest.mark.parametrize("K", [2, 3])
def test_next_call_starts_from_a_whole_bf16_copy(dims, K):
    # the last step's launches read the low halves that lie in layer 1's bf16 copy and write that copy
    # anew; the next call without a meta-update reads it in its first forward product.  Launch by launch
    # there is no side stream: the same bits mean that the one is read before the other is written.
    out = []
    for profiled in (False, True):
        g = _handle(dims, K, 0.002)
        g.set_profiling(profiled)
        g.local_steps(); g.local_steps(); g.local_steps()      # (the first may have rebuilt steps)
        g.sync()
        out.append((g.get_losses(), g.replicas[:, :g.n].cpu().numpy().view(np.uint32)))
        g.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
