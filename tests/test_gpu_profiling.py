"""Profiled rounds run the launches of ordinary ones where a round's steps are one launch: the same bits,
the same number of launches, each of them timed."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _small(m, mode):
    dims = [64, 48, 10]
    rng = np.random.default_rng(3)
    x = rng.standard_normal((500, dims[0]), dtype=np.float32)
    y = rng.integers(0, dims[-1], size=500).astype(np.int32)
    return m.Mavg(m.workloads.mlp_init(dims), P=3, K=4, local_lr=0.05, mu=0.9, B=31, seed=9,
                  objective=m.OBJ_MLP, dims=dims, gemm_bf16=mode, x=x, y=y)


def _pseudograd(m, mode):
    return m.Mavg(m.workloads.global_model(700_001), P=3, K=4, local_lr=0.05, mu=0.9, seed=9,
                  objective=m.OBJ_PSEUDOGRAD, sigma=0.1, defer_broadcast=bool(mode))


@pytest.mark.parametrize("make,mode,want", [
    (_small, 0, dict(wgrad_sgd_gemm=1, meta_update=1)), (_small, 2, dict(wgrad_sgd_gemm=1, meta_update=1)),
    (_pseudograd, 0, dict(pseudograd_steps=1)), (_pseudograd, 1, dict(pseudograd_steps=1))])
def test_profiled_round_is_the_round(make, mode, want):
    import paper_2110_00625_b200 as m
    out = []
    for profiled in (False, True):
        g = make(m, mode)
        g.set_profiling(profiled)
        before = g.launch_count()
        for _ in range(2):
            g.round()
        launches = g.launch_count() - before
        if profiled:
            prof = g.get_profile()
            assert {k: n for k, (_, n) in prof.items() if n} == {k: 2 * n for k, n in want.items()}
            assert all(ms > 0 for ms, n in prof.values() if n)
        g.sync()
        out.append((launches, g.w.cpu().numpy().view(np.uint32), g.v.cpu().numpy().view(np.uint32),
                    g.replicas[:, :g.n].cpu().numpy().view(np.uint32)))
        g.close()
    assert out[0][0] == out[1][0] == 2 * sum(want.values())
    for a, b in zip(out[0][1:], out[1][1:]):
        assert np.array_equal(a, b)
