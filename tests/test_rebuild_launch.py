"""The launch that forms the weights of rebuilt local steps: with its shared memory no other block that takes tensor memory
finds room on its SM, and its set-up takes its columns before the next kernel may begin.  Host arithmetic and sources only
(the rules are those of test_tensor_memory_share.py)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00625_b200", "csrc")
MAIN = r'''
#include <algorithm>
#include <cstdio>
#include "rebuild.cuh"
using namespace mavg;
int main() {
  for (bool last : {false, true})
    printf("%zu %zu %zu %zu\n", sizeof(rebuild::Shared), rebuild::launch_bytes(last), rebuild::smem_of(last), tc::tmem_share_bytes(32, 0));
}
'''


def test_its_shared_memory_is_its_share_of_an_sm(tmp_path):
    from paper_2110_00625_b200 import build as B
    if not os.path.exists(B.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run([B.NVCC, *B.FLAGS, "-I", CSRC, str(src), "-o", str(exe)], check=True)
    for line in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines():
        fixed, dynamic, used, least = map(int, line.split())
        assert fixed % 16 == 0 and fixed + dynamic <= 227 * 1024 and used <= dynamic
        # all 512 columns: beside it not even a block of the fewest columns fits
        assert fixed + dynamic + 1024 + least + 1024 > 228 * 1024


def test_it_takes_its_columns_before_the_next_kernel_may_begin():
    text = open(os.path.join(CSRC, "rebuild.cuh")).read()
    body = text[text.index("tmem_alloc("):text.index("tmem_dealloc(")]
    assert body.index("grid_launch_dependents()") < body.index("grid_dependency_wait()")
    assert text.count("tmem_alloc(") == 1
