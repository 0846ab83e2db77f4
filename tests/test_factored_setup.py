"""Setting up factored rounds when one of the calls it rests on is refused: the handle keeps the plain form instead
of failing.  Host code only: factored.cu is linked with stand-ins for the two calls, whose results the test sets."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00625_b200", "csrc")

MAIN = r'''
#include <cstdio>
#include <vector>
#include "mlp.cuh"
#include "tc_state.cuh"
static cudaError_t attribute;
static int encodes, refuse_at;
extern "C" cudaError_t __wrap_cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return attribute; }
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return ++encodes == refuse_at ? CUDA_ERROR_INVALID_VALUE : CUDA_SUCCESS;
}
int main() {
  std::vector<char> ws(4096);
  const int cases[3][2] = {{0, 0}, {0, 7}, {1, 0}};
  for (auto& c : cases) {
    attribute = c[0] ? cudaErrorInvalidValue : cudaSuccess;
    encodes = 0;
    refuse_at = c[1];
    mavg_ctx h{};
    h.cfg.P = 8; h.cfg.K = 8; h.cfg.B = 128; h.cfg.n_layers = 3;
    h.cfg.dims[0] = 3072; h.cfg.dims[1] = h.cfg.dims[2] = 512; h.cfg.dims[3] = 10;
    h.sm_count = 148;
    h.buf.workspace = ws.data();
    h.buf.replicas = (float*)ws.data();
    h.buf.replica_stride = 1841168;
    mavg::TcState st{};
    st.encode = encode;
    mavg::fac_setup(&h, &st);
    printf("%d ", st.fac != nullptr);
    delete st.fac;
  }
}
'''


def test_refused_calls_leave_the_plain_form(tmp_path):
    from paper_2110_00625_b200 import build as B
    if not os.path.exists(B.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.run([B.NVCC, *B.FLAGS, "-I", CSRC, str(src), os.path.join(CSRC, "factored.cu"), "-o", str(exe),
                    "-Xlinker", "--wrap=cudaFuncSetAttribute"], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True)
    assert out.stdout.split() == ["1", "0", "0"]
