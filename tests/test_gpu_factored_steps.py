"""Local steps taken from w~ and the factors dZ, A of the earlier steps (no hidden weights per learner until
the end of the call): against the same form in torch, against the plain form, and where a call must not
depend on how it is issued."""
import numpy as np
import pytest
import torch

from tests.util import assert_tiles_close, l2_rel

pytestmark = pytest.mark.gpu
LR = 0.002

# dims, P, K, B: one, two and three hidden layers; ragged row, column and contraction tiles; batches of 16
# (16 learners to a block), 80 (three), 256 (one) and cut into column pieces; 10, 12 and 32 classes; last
# layers of one block and of eight per learner
SHAPES = [
    ([1000, 312, 10], 40, 4, 80),
    ([520, 200, 136, 12], 20, 9, 48),
    ([264, 648, 648, 10], 64, 8, 16),
    ([512, 384, 32], 16, 2, 256),
    ([1032, 1000, 520, 264, 10], 52, 5, 32),
    ([2000, 1000, 1000, 10], 32, 2, 128),
    ([3072, 512, 512, 10], 8, 8, 128),
]


def _handle(dims, P, K, B, schedule=0, **kw):
    import paper_2110_00625_b200 as m
    rng = np.random.default_rng(3)
    x = torch.from_numpy(rng.standard_normal((4096, dims[0]), dtype=np.float32)).bfloat16()
    y = (x.float().numpy() @ rng.standard_normal((dims[0], dims[-1])).astype(np.float32)).argmax(1).astype(np.int32)
    w1 = m.workloads.mlp_init(dims)
    g = m.Mavg(w1, P=P, K=K, local_lr=kw.pop("lr", LR), mu=0.9, B=B, seed=5, objective=m.OBJ_MLP, dims=dims,
               gemm_bf16=1, x=x, y=y, x_bf16=True, **kw)
    g.set_schedule(schedule)
    return g, w1


def _takes(dims, P, K, B, **kw):
    """Whether such a handle's rounds take the form; they then have one launch for all hidden weights, none per step."""
    g, _ = _handle(dims, P, K, B, **kw)
    takes = g.factored()
    g.set_profiling(True)
    g.round()
    launches = g.get_profile()["wgrad_sgd_gemm"][1]
    g.close()
    assert K == 1 or takes == (launches == 1), (takes, launches)
    return takes


def _q(t):
    return t.bfloat16().float()


def _both(t):
    return _q(t) + _q(t - _q(t))         # what the forward products read of the weights


def _reference(dims, P, K, B, w1, x, y, idx):
    """The learners' models after K steps in fp32 with the form's bf16 operands, and the losses."""
    L = len(dims) - 1
    W0, b0, off = [], [], 0
    for l in range(L):
        W0.append(w1[off:off + dims[l + 1] * dims[l]].view(dims[l + 1], dims[l]))
        off += dims[l + 1] * dims[l]
        b0.append(w1[off:off + dims[l + 1]])
        off += dims[l + 1]
    models, losses = [], []
    for j in range(P):
        W, b = [w.clone() for w in W0], [t.clone() for t in b0]
        A, D = [[] for _ in range(L)], [[] for _ in range(L)]
        for k in range(K):
            a = [x[idx[j][k]].float()]
            for l in range(L):
                ai = _q(a[l])
                w = W0[l] if l < L - 1 else W[l]
                z = ai @ _both(w).T + b[l]
                if k and l < L - 1:
                    z = z + _q(-LR * (ai @ torch.cat(A[l]).T)) @ torch.cat(D[l])
                a.append(torch.relu(z) if l < L - 1 else z)
            yy = y[idx[j][k]].long()
            losses.append(torch.nn.functional.cross_entropy(a[-1], yy).item())
            dz = torch.softmax(a[-1], 1)
            dz[torch.arange(B), yy] -= 1
            dz /= B
            for l in range(L - 1, -1, -1):
                dq, ai = _q(dz), _q(a[l])
                if l:
                    da = dq @ _q(W0[l] if l < L - 1 else W[l])
                    if k and l < L - 1:
                        da = da + _q(-LR * (dq @ torch.cat(D[l]).T)) @ torch.cat(A[l])
                A[l].append(ai)
                D[l].append(dq)
                W[l] = W[l] - LR * (dq.T @ ai)
                b[l] = b[l] - LR * dz.sum(0)
                if l:
                    dz = da * (ai > 0)
        models.append(torch.cat([torch.cat([W[l].reshape(-1), b[l]]) for l in range(L)]))
    return torch.stack(models), np.array(losses).reshape(P, K)


@pytest.mark.parametrize("dims,P,K,B", SHAPES)
def test_against_the_same_form_in_torch_and_the_plain_form(dims, P, K, B):
    assert _takes(dims, P, K, B)
    g, w1 = _handle(dims, P, K, B, defer_broadcast=True)
    idx = [[torch.from_numpy(g.get_batch_indices(1, j, k).astype(np.int64)).cuda() for k in range(1, K + 1)]
           for j in range(P)]
    g.local_steps()
    g.sync()
    w = torch.from_numpy(w1).cuda()
    want, losses = _reference(dims, P, K, B, w, g.x, g.y, idx)
    got = g.replicas[:, :g.n]
    assert np.abs(g.get_losses() - losses).max() <= 5e-3 * losses.max()
    # per learner the two differ where a rounding or a ReLU branch falls the other way (worst 4.3e-2, three
    # hidden layers); a wrong tile is off by 1.  The mean over the learners, tile by tile, averages those out.
    for j in range(P):
        assert l2_rel((got[j] - w).cpu().numpy(), (want[j] - w).cpu().numpy()) <= 8e-2, j
    assert_tiles_close((got.mean(0) - w).cpu().numpy(), (want.mean(0) - w).cpu().numpy(), dims)
    plain, _ = _handle(dims, P, K, B, schedule=2, defer_broadcast=True)
    g.meta_update()
    plain.round()
    g.sync(); plain.sync()
    assert l2_rel(g.v.cpu().numpy(), plain.v.cpu().numpy()) <= 2e-2
    g.close(); plain.close()


@pytest.mark.parametrize("dims,P,K,B", SHAPES)
def test_the_same_bits_however_it_is_issued(dims, P, K, B):
    # replayed, launch by launch, with copies written eagerly or not, in a handle made for more steps; a second
    # call without a meta-update starts from the learners' own models
    out = []
    spare = next(e for e in (3, 2, 1, 0) if _takes(dims, P, K + e, B))      # (a handle that never does has no room for it)
    for profiled, defer, more in ((False, True, 0), (True, True, 0), (False, False, 0), (False, True, spare)):
        g, _ = _handle(dims, P, K + more, B, defer_broadcast=defer)
        if more:
            g.set_hparams(K, LR, 1.0, 0.9)
        g.set_profiling(profiled)
        loss = [g.round(want_loss=True) for _ in range(2)]
        g.local_steps()
        g.sync()
        first = g.replicas[:, :g.n].cpu().numpy().view(np.uint32)
        g.local_steps(); g.meta_update()
        g.sync()
        out.append((loss, first, g.w.cpu().numpy().view(np.uint32), g.v.cpu().numpy().view(np.uint32)))
        g.close()
    for other in out[1:]:
        assert other[0] == out[0][0]
        for a, b in zip(out[0][1:], other[1:]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("dims,P,K,B", SHAPES[:3])
def test_steps_of_length_zero_keep_every_bit(dims, P, K, B):
    g, w1 = _handle(dims, P, K, B, lr=0.0)
    g.local_steps()
    g.sync()
    zero = w1 == 0.0                  # -0 * g + 0 may be either zero
    for row in g.replicas[:, :g.n].cpu().numpy():
        assert np.array_equal(row[~zero].view(np.uint32), w1[~zero].view(np.uint32)) and not row[zero].any()
    g.close()


def test_where_the_form_is_taken():
    # both sides of its lines: 8192 rows a round, two steps, momentum, a hidden layer; the added work (K) below 5.5 times
    # the weights, where they are few for a step's launches (P) only for small batches or one hidden layer
    for dims, P, K, B, kw, want in [
        ([1000, 312, 10], 32, 2, 128, {}, True), ([1000, 312, 10], 31, 2, 128, {}, False),
        ([1000, 312, 10], 64, 1, 128, {}, False), ([1000, 312, 10], 32, 2, 128, dict(learner_momentum=0.9), False),
        ([1000, 10], 32, 2, 128, {}, False),
        ([1000, 312, 10], 16, 5, 144, {}, True), ([1000, 312, 10], 16, 6, 144, {}, False),
        ([400, 400, 10], 13, 8, 128, {}, True), ([400, 400, 10], 13, 9, 128, {}, False),
        ([400, 400, 10], 12, 8, 128, {}, False), ([400, 400, 10], 13, 7, 144, {}, False),
        ([520, 200, 136, 12], 19, 9, 48, {}, True), ([520, 200, 136, 12], 19, 10, 48, {}, False),
        ([376, 136, 19], 20, 14, 32, {}, True), ([376, 136, 19], 19, 14, 32, {}, False),
        ([616, 192, 80, 80, 30], 65, 4, 96, {}, True), ([616, 192, 80, 80, 30], 64, 4, 96, {}, False),
    ]:
        assert _takes(dims, P, K, B, **kw) == want, (dims, P, K, B, kw)


def test_a_refused_allocation_leaves_the_plain_form(monkeypatch):
    # the room for the rows of all steps is not to be had: a handle in the plain form, and the same round as one
    import ctypes as C
    dims, P, K, B = SHAPES[-1]
    g, _ = _handle(dims, P, K, B)
    full, least = g.workspace.numel(), C.c_size_t()
    assert g.lib.mavg_workspace_least_bytes(C.byref(g.cfg), C.byref(least)) == 0 and least.value < full
    g.close()
    empty = torch.empty

    def refuse(size, *a, **kw):
        if size == full:
            raise torch.cuda.OutOfMemoryError("refused")
        return empty(size, *a, **kw)

    monkeypatch.setattr(torch, "empty", refuse)
    g, _ = _handle(dims, P, K, B)
    assert g.workspace.numel() == least.value and not g.factored()
    monkeypatch.setattr(torch, "empty", empty)
    plain, _ = _handle(dims, P, K, B, schedule=2)
    assert abs(g.round(want_loss=True) - plain.round(want_loss=True)) <= 1e-3
    g.sync(); plain.sync()
    assert l2_rel(g.v.cpu().numpy(), plain.v.cpu().numpy()) <= 2e-2
    g.close(); plain.close()


def test_a_workspace_of_the_plain_forms_size_keeps_that_form():
    # buffers sized before the form existed: a handle of one step has no use for more than the plain form needs
    import ctypes as C
    from paper_2110_00625_b200 import binding
    dims, P, K, B = SHAPES[-1]
    g, _ = _handle(dims, P, K, B)
    assert g.factored()
    one, plain = binding.Config.from_buffer_copy(g.cfg), C.c_size_t()
    one.K = 1
    assert g.lib.mavg_workspace_bytes(C.byref(one), C.byref(plain)) == 0
    buf = binding.Buffers.from_buffer_copy(g.buf)
    buf.workspace_bytes = plain.value + 4 * P * K + 256          # the losses of K steps
    assert buf.workspace_bytes < g.workspace.numel()
    h, used = C.c_void_p(), C.c_int32(-1)
    assert g.lib.mavg_create(C.byref(g.cfg), C.byref(buf), C.byref(h)) == 0
    assert g.lib.mavg_get_factored(h, C.byref(used)) == 0 and used.value == 0
    assert g.lib.mavg_round(h, None) == 0 and g.lib.mavg_sync(h) == 0
    assert torch.isfinite(g.w).all()
    g.lib.mavg_destroy(h)
    g.close()


@pytest.mark.parametrize("dims,P,K,B", [SHAPES[0], SHAPES[1], SHAPES[4]])
@pytest.mark.parametrize("value", [np.inf, -np.inf, 3.4e38, np.nan])
@pytest.mark.parametrize("layer", [1, -1])        # the first and the last hidden layer
def test_a_weight_that_is_not_finite_spreads_as_in_the_plain_form(dims, P, K, B, value, layer):
    # an infinite weight makes activations infinite, and those whatever they meet: the loss and every weight are
    # finite, or not, as without the form (3.4e38 rounds to infinity as bf16)
    layer = layer % (len(dims) - 1)
    out = []
    for schedule in (0, 2):
        g, w1 = _handle(dims, P, K, B, schedule=schedule)
        at = sum(dims[i] * dims[i + 1] + dims[i + 1] for i in range(layer - 1)) + 3 * dims[layer - 1] + 5
        g.w[at] = value
        g.set_round(0)
        assert g.factored() == (schedule == 0)
        out.append((np.isfinite(g.round(want_loss=True)), np.isfinite(g.w.cpu().numpy())))
        g.close()
    assert out[0][0] == out[1][0]
    assert np.array_equal(out[0][1], out[1][1]), (out[0][1].mean(), out[1][1].mean())


@pytest.mark.parametrize("dims,P,K,B,x_bf16,defer", [([1000, 312, 10], 40, 4, 80, True, True),
                                                     ([520, 200, 136, 12], 20, 9, 48, False, False),
                                                     ([1032, 1000, 520, 264, 10], 52, 5, 32, False, True)])
def test_rounds_of_either_form_on_one_handle(dims, P, K, B, x_bf16, defer):
    # The forms share scratch, and a factored round leaves the learners' bf16 copies unwritten: every call in turn
    # leaves what a handle made for it, from the same model, leaves.
    import paper_2110_00625_b200 as m
    rng = np.random.default_rng(3)
    x = torch.from_numpy(rng.standard_normal((4096, dims[0]), dtype=np.float32))
    y = rng.integers(0, dims[-1], 4096).astype(np.int32)

    def make(w1, K=K, beta=0.0, schedule=0):
        g = m.Mavg(w1, P=P, K=K, local_lr=LR, mu=0.9, B=B, seed=5, objective=m.OBJ_MLP, dims=dims, gemm_bf16=1, x=x, y=y,
                   x_bf16=x_bf16, defer_broadcast=defer, learner_momentum=beta, learner_momentum_reset=True,
                   with_learner_u=True)
        g.set_schedule(schedule)
        return g

    def steps_twice(g):
        g.local_steps(); g.local_steps(); g.meta_update()

    def host(g):
        w, v = g.w.cpu(), g.v.cpu()
        g.round_host(w, v)
        assert torch.equal(w, g.w.cpu()) and torch.equal(v, g.v.cpu())

    def run_out(g):
        g.set_wait_limit(20_000)
        g.selftest_wait()
        with pytest.raises(m.MavgError):
            g.sync()
        g.set_wait_limit(0)
        g.round()

    a = make(m.workloads.mlp_init(dims))
    turns = [(lambda: None, {}, a.round, "round"),
             (lambda: a.set_schedule(2), dict(schedule=2), a.round, "round"),
             (lambda: a.set_schedule(0), {}, a.round, "round"),
             (lambda: a.set_hparams(1, LR, 1.0, 0.9), dict(K=1), a.round, "round"),
             (lambda: a.set_hparams(K, LR, 1.0, 0.9), {}, lambda: steps_twice(a), "steps"),
             (lambda: a.set_learner_momentum(0.9, True), dict(beta=0.9), a.round, "round"),
             (lambda: a.set_learner_momentum(0.0, True), {}, lambda: host(a), "round"),
             (lambda: a.set_schedule(2), dict(schedule=2), lambda: host(a), "round"),
             (lambda: a.set_schedule(0), {}, lambda: run_out(a), "round"),
             (lambda: None, {}, lambda: host(a), "round")]
    for turn, (change, kw, call, plain_call) in enumerate(turns):
        change()
        w, v, done = a.w.clone(), a.v.clone(), a.get_round()
        b = make(w.cpu().numpy(), **kw)
        b.v.copy_(v)
        b.set_round(done)
        takes = not kw
        assert a.factored() == b.factored() == takes, turn
        call()
        b.round() if plain_call == "round" else steps_twice(b)
        a.materialize_replicas(); b.materialize_replicas()
        a.sync(); b.sync()
        assert np.array_equal(a.get_losses()[:, :b.K], b.get_losses()), turn
        for p, q in ((a.w, b.w), (a.v, b.v), (a.replicas[:, :a.n], b.replicas[:, :b.n])):
            assert torch.equal(p.view(torch.int32), q.view(torch.int32)), turn
        b.close()
    a.close()


def test_handles_on_streams_of_their_own_side_by_side():
    # launches of clusters that wait within themselves, of few and of many columns of tensor memory, and a handle in
    # the plain form, all at once: the bits of each on its own
    picks = [(SHAPES[6], 0), (SHAPES[1], 0), (([3072, 512, 512, 10], 4, 2, 64), 0), (SHAPES[5], 0), (SHAPES[1], 2)]

    def run(together):
        handles = []
        for shape, schedule in picks:
            torch.cuda.synchronize()
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                handles.append(_handle(*shape, schedule=schedule, defer_broadcast=True, stream=stream)[0])
            stream.synchronize()
        if together:
            for _ in range(10):
                for g in handles:
                    g.round()
        else:
            for g in handles:
                for _ in range(10):
                    g.round()
                g.sync()
        out = []
        for g in handles:
            g.sync()
            out.append((g.w.cpu().numpy().view(np.uint32), g.v.cpu().numpy().view(np.uint32)))
            g.close()
        return out

    for alone, beside in zip(run(False), run(True)):
        assert np.array_equal(alone[0], beside[0]) and np.array_equal(alone[1], beside[1])
