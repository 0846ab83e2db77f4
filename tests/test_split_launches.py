"""Launches of the products of fp32 and odd-shaped models: their share of an SM's shared memory for their share of its
tensor memory, what they stage and exchange fits what they ask for, and the order of their set-up.  Host arithmetic and
sources only (the rules are those of test_tensor_memory_share.py)."""
import os
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00625_b200", "csrc")
MAIN = r'''
#include <algorithm>
#include <cstdio>
#include "split_gemm.cuh"
using namespace mavg;
int main() {
  for (int np : {1, 3}) {
    for (int n = 16; n <= split::kMaxN; n += 16) {
      const split::LaunchShape s = split::product_shape(np, n);
      printf("%d %d %d %u %zu %d %zu\n", np, n, s.stages, s.tmem_cols, s.smem, split::product_stage_bytes(np, n), sizeof(split::Barriers));
    }
    const split::LaunchShape s = split::wgrad_shape(np);
    printf("%d %d %d %u %zu %d %zu\n", np, 0, s.stages, s.tmem_cols, s.smem, split::wgrad_stage_bytes(np), sizeof(split::Barriers));
  }
}
'''


def test_a_products_launch_holds_what_it_needs(tmp_path):
    from paper_2110_00625_b200 import build as B
    if not os.path.exists(B.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run([B.NVCC, *B.FLAGS, "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rows = [tuple(map(int, line.split())) for line in subprocess.run([str(exe)], capture_output=True, text=True,
                                                                     check=True).stdout.splitlines()]
    assert len(rows) == 18
    for np_, n, stages, columns, smem, stage, fixed in rows:
        assert fixed + smem + 1024 <= 228 * 1024
        assert 228 * 1024 // (fixed + smem + 1024) <= 512 // columns       # blocks of an SM / blocks its columns are for
        assert columns >= ((3 if np_ == 3 else 2) * n if n else 128 * (4 if np_ == 3 else 2))
        assert stages >= 2 and stages * stage + 1024 <= smem
        for splits in range(1, 9) if n else ():                            # the sums a block receives
            share = -(-(n // 16) // splits)
            assert splits * share * 16 * 128 * 4 + 1024 <= smem


def test_set_up_in_the_order_that_the_next_kernel_relies_on():
    text = open(os.path.join(CSRC, "split_gemm.cuh")).read()
    allocs = [m.start() for m in re.finditer(r"\btmem_alloc\(", text)]
    assert len(allocs) == 2
    for at in allocs:
        kernel = text[text.rindex("__global__", 0, at):]
        body = kernel[:kernel.index("tmem_dealloc(")]
        assert body.index("tmem_alloc(") < body.index("grid_launch_dependents()") < body.index("grid_dependency_wait()")
