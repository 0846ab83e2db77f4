"""Tensor memory: whatever mix of blocks an SM's shared memory admits, its 512 columns are enough for all of them, so
that no allocation ever waits.  Blocks that hold columns can be waiting for others (a cluster's for one another, a
successor's for the kernel before it), and with launches of several handles side by side an allocation without a time
limit could close a circle.  Host arithmetic and sources only."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00625_b200", "csrc")
MAIN = r'''
#include <cstdio>
#include "gemm_unit.cuh"
#include "wgrad_unit.cuh"
int main() {
  const size_t gemm = sizeof(mavg::gemm::GemmShared), wgrad = sizeof(mavg::wgrad::WgradShared);
  for (unsigned c = 32; c <= 512; c *= 2)
    for (size_t fixed : {gemm, gemm + 16, wgrad}) printf("%u %zu %zu\n", c, fixed, mavg::tc::tmem_share_bytes(c, fixed));
}
'''


def test_no_mix_of_blocks_runs_out_of_columns(tmp_path):
    from paper_2110_00625_b200 import build as B
    if not os.path.exists(B.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run([B.NVCC, *B.FLAGS, "-I", CSRC, str(src), "-o", str(exe)], check=True)
    kinds = [tuple(map(int, line.split())) for line in subprocess.run([str(exe)], capture_output=True, text=True,
                                                                      check=True).stdout.splitlines()]
    assert len(kinds) == 15

    def most_columns(room, left):              # over all mixes that fit `room` bytes of an SM's shared memory
        if not left:
            return 0
        columns, fixed, dynamic = left[0]
        held = fixed + dynamic + 1024          # 1 KB of it is reserved per block
        return max(n * columns + most_columns(room - n * held, left[1:]) for n in range(room // held + 1))

    assert most_columns(228 * 1024, kinds) <= 512
    # and the share is no more than needed: as many blocks of one kind as there are columns for do fit
    for columns, fixed, dynamic in kinds:
        assert 228 * 1024 // (fixed + dynamic + 1024) == 512 // columns
        assert fixed + dynamic <= 227 * 1024       # a block may have that much


def test_every_launch_that_takes_tensor_memory_asks_for_its_share():
    launches = {"factored.cu": 3, "fwd_dense.cu": 1, "mlp_tc.cu": 2, "wgrad_tc.cu": 2}
    for name in os.listdir(CSRC):
        text = open(os.path.join(CSRC, name)).read()
        kernels = len(re.findall(r"\btmem_alloc\(&", text))
        assert (kernels > 0) == (name in launches), name
        assert name not in launches or kernels == launches[name] == len(re.findall(r"tmem_share_bytes\(", text)), name


def test_the_next_kernel_begins_after_a_block_has_its_columns():
    # in every kernel that takes tensor memory: alloc, then the trigger, then the wait for the kernel before
    for name in ("factored.cu", "fwd_dense.cu", "mlp_tc.cu", "wgrad_tc.cu"):
        text = open(os.path.join(CSRC, name)).read()
        allocs = [m.start() for m in re.finditer(r"\btmem_alloc\(", text)]
        assert allocs, name
        for at in allocs:
            kernel = text[text.rindex("__global__", 0, at):]
            body = kernel[:kernel.index("tmem_dealloc(")]
            first = body.index("tmem_alloc(")
            early = [m.start() for m in re.finditer(r"grid_launch_dependents\(\)", body) if m.start() < first]
            # (a block that returns at once takes none)
            assert all("return;" in body[e:e + 60] for e in early), name
            assert first < body.index("grid_launch_dependents()", first) < body.index("grid_dependency_wait()"), name
