"""Setting up fp32 and odd-shaped models when the CUDA runtime or driver refuses one of the calls it rests on: a refused
cluster query only means that products are not split, and small models need nothing of that path.  Host code only: the files
are linked with stand-ins for the calls, whose results the test sets."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00625_b200", "csrc")
MAIN = r'''
#include <cstdio>
#include <vector>
#include "mlp.cuh"
#include "tensor_map.cuh"
static cudaError_t attribute, query;
static bool encoder;
static int small_clusters, queries, attributes;
extern "C" cudaError_t __wrap_cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { ++attributes; return attribute; }
extern "C" cudaError_t __wrap_cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* lc) {
  if (lc->blockDim.x == 384) {                     // the small-model kernel's
    *n = small_clusters;
    return small_clusters < 0 ? cudaErrorNotSupported : cudaSuccess;
  }
  ++queries;
  *n = 30;
  return query;
}
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
extern "C" cudaError_t __wrap_cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* r) {
  *fn = encoder ? (void*)encode : nullptr;
  *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
static void set_up(int d0, int d1) {
  static std::vector<char> ws(1 << 24);
  mavg_ctx h{};
  h.cfg.P = 4; h.cfg.K = 4; h.cfg.B = 32; h.cfg.n = d0 * d1 + d1 + d1 * 10 + 10; h.cfg.n_layers = 2;
  h.cfg.dims[0] = d0; h.cfg.dims[1] = d1; h.cfg.dims[2] = 10;
  h.sm_count = 148;
  h.buf.workspace = ws.data();
  queries = attributes = 0;
  const mavg_status st = mavg::mlp_setup(&h);
  printf("%d %d %d %d\n", (int)st, h.small_splits, queries, attributes);
}
int main() {
  attribute = cudaSuccess; query = cudaErrorNotSupported; encoder = false; small_clusters = 1000;
  set_up(32, 64);                                  // small: neither queries nor maps
  small_clusters = -1; encoder = true;
  set_up(32, 64);                                  // refused there: the other path, without splits
  set_up(512, 256);
  encoder = false;
  set_up(512, 256);                                // no maps: nothing left
  encoder = true; query = cudaSuccess;
  set_up(512, 256);                                // asked again, as nothing was learned
  set_up(512, 512);                                // the same shape of a product
  attribute = cudaErrorInvalidValue;
  set_up(512, 256);
}
'''


def test_refused_calls_and_what_is_asked_for(tmp_path):
    from paper_2110_00625_b200 import build as B
    if not os.path.exists(B.NVCC):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "main.cu", tmp_path / "main"
    src.write_text(MAIN)
    wrap = ["cudaFuncSetAttribute", "cudaOccupancyMaxActiveClusters", "cudaGetDriverEntryPoint"]
    subprocess.run([B.NVCC, *B.FLAGS, "-I", CSRC, str(src), *(os.path.join(CSRC, f) for f in ("mlp.cu", "mlp_simt.cu", "mlp_small.cu")),
                    "-o", str(exe), "-Xlinker", "--unresolved-symbols=ignore-all",
                    *(a for w in wrap for a in ("-Xlinker", "--wrap=" + w))], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")
    rows = [tuple(map(int, line.split())) for line in out if line]
    assert [r[0] == 0 for r in rows] == [True, True, True, False, True, True, False]
    assert rows[0][1:3] == (8, 0) and rows[0][3] == 1
    assert all(r[1] == 0 for r in rows[1:])
    assert [r[2] for r in rows[1:]] == [7, 7, 0, 7, 0, 0]
    # the forward product, one weight gradient and the fused last layer, two attributes each, and the first launch: no kernel
    # that is not launched
    assert rows[2][3] == 7
