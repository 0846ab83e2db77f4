"""The choice of the small-model kernel when the CUDA runtime refuses one of the calls it rests on: the
handle falls back to the launch per product.  Host code only: mlp_small.cu is linked with stand-ins for
the two calls, whose results the test sets."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2110_00625_b200", "csrc")

MAIN = r'''
#include <cstdio>
#include "mlp.cuh"
static cudaError_t attribute, query;
extern "C" cudaError_t __wrap_cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return attribute; }
extern "C" cudaError_t __wrap_cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 1000;
  return query;
}
int main() {
  const cudaError_t cases[3][2] = {{cudaSuccess, cudaSuccess}, {cudaSuccess, cudaErrorNotSupported},
                                   {cudaErrorInvalidValue, cudaSuccess}};
  for (auto& c : cases) {
    attribute = c[0];
    query = c[1];
    mavg_ctx h{};
    h.cfg.P = 4; h.cfg.K = 4; h.cfg.B = 32; h.cfg.n = 2762; h.cfg.n_layers = 2;
    h.cfg.dims[0] = 32; h.cfg.dims[1] = 64; h.cfg.dims[2] = 10;
    mavg::small_setup(&h);
    printf("%d ", h.small_splits);
  }
}
'''


def test_refused_calls_leave_the_launch_per_product(tmp_path):
    from paper_2110_00625_b200 import build as B
    if not os.path.exists(B.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run([B.NVCC, *B.FLAGS, "-I", CSRC, str(src), os.path.join(CSRC, "mlp_small.cu"), "-o", str(exe),
                    "-Xlinker", "--wrap=cudaFuncSetAttribute",
                    "-Xlinker", "--wrap=cudaOccupancyMaxActiveClusters"], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True)
    assert out.stdout.split() == ["8", "0", "0"]
