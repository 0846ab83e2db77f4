// Tensor maps of the tiled copies (host side).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <string>

namespace mavg {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's encoder, or null with the reason.
inline EncodeTiledFn tensor_map_encoder(std::string* why) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  const cudaError_t e = cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres);
  if (e == cudaSuccess && fn && qres == cudaDriverEntryPointSuccess) return (EncodeTiledFn)fn;
  if (why) *why = "cuTensorMapEncodeTiled is not available from this driver";
  cudaGetLastError();
  return nullptr;
}

// Tensor [batch, rows, inner] with the given strides (in elements) and box inner x box_rows x box_batch.
inline bool encode_tiled(EncodeTiledFn encode, CUtensorMap* m, CUtensorMapDataType dt, int esize, void* ptr,
                int inner, int rows, int batch, int64_t row_stride, int64_t batch_stride,
                int box_inner, int box_rows, CUtensorMapSwizzle swz, std::string* why, int box_batch = 1) {
  cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)rows, (cuuint64_t)batch};
  cuuint64_t strides[2] = {(cuuint64_t)row_stride * esize, (cuuint64_t)batch_stride * esize};
  cuuint32_t box[3] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows, (cuuint32_t)box_batch};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = encode(m, dt, 3, ptr, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                      CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    if (why) *why = "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r);
    return false;
  }
  return true;
}

}  // namespace mavg
