"""The pinned words that rounds leave their mean loss in: a handle gives its own back without waiting for the stream, and one
that finds none free has the mean copied back.  A process's first handle, which allocates them, may be made beside a capture."""
import os
import subprocess
import sys

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


FIRST = """
import ctypes as C
import torch
import paper_2110_00625_b200 as m
from paper_2110_00625_b200 import binding as b

gemm, dims, S = %d, [64, 64, 10], 256
lib, s = b.load_library(), torch.cuda.Stream()
n = sum(dims[l + 1] * (dims[l] + 1) for l in range(2))
x, y = torch.randn(S, dims[0], device="cuda"), torch.randint(0, 10, (S,), device="cuda").int()
w, v, rep = torch.randn(n, device="cuda"), torch.empty(n, device="cuda"), torch.empty(2, (n + 31) // 32 * 32, device="cuda")
cfg = b.make_config(2, 2, 0.1, 0.9, B=16, objective=m.OBJ_MLP, n=n, dims=dims, gemm_bf16=gemm, x_ptr=x.data_ptr(),
                    y_ptr=y.data_ptr(), n_samples=S, stream=s.cuda_stream)
size = C.c_size_t()
assert lib.mavg_workspace_bytes(C.byref(cfg), C.byref(size)) == 0
scratch = torch.empty(size.value, dtype=torch.uint8, device="cuda")
buf = b.Buffers(rep.data_ptr(), rep.shape[1], w.data_ptr(), v.data_ptr(), scratch.data_ptr(), size.value, None)
h, a, graph = C.c_void_p(), torch.zeros(8, device="cuda"), torch.cuda.CUDAGraph()
torch.cuda.synchronize()
with torch.cuda.graph(graph):                     # captured on another stream, in the mode that minds other streams
    a += 1
    assert lib.mavg_create(C.byref(cfg), C.byref(buf), C.byref(h)) == 0
    a += 1
loss = C.c_float()
assert lib.mavg_round(h, C.byref(loss)) == 0 and loss.value > 0
graph.replay()
assert a.tolist() == [2.0] * 8
if gemm != 1:                                     # (a handle that replays a graph of its own destroys it)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        a += 1
        assert lib.mavg_destroy(h) == 0
    graph.replay()
    assert a.tolist() == [3.0] * 8
print("done")
"""


@pytest.mark.parametrize("gemm", [0, 1, 2])
def test_the_first_handle_beside_a_capture(gemm):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    out = subprocess.run([sys.executable, "-c", FIRST % gemm], capture_output=True, text=True, cwd=root, timeout=300)
    assert out.stdout.split() == ["done"], out.stderr[-800:]
