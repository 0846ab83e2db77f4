// Minibatch side of the learner level: "randomly sample a mini-batch of size B_n"
// (Algorithm 1) as a counter-based index stream, and the gather of the sampled rows for the
// tensor-core path.
#include <mutex>

#include "mlp.cuh"

namespace mavg {
namespace {

// The B indices of one learner, a thread per slot.
__global__ void k_batch_indices(int32_t* __restrict__ idx, uint64_t seed, int64_t round, int step,
                                int P, int B, int64_t S, int j) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < B) idx[s] = sample_index(seed, round, j, step, s, P, S);
}

template <typename TIN>
__device__ __forceinline__ float to_f32(TIN v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

// Index stream and gather in one kernel, for bf16 operands: block (32, 8) handles 32 batch slots of
// learner blockIdx.z and 64 input columns; it writes the rows [P, B, d] and, through a
// shared-memory tile, their transpose [P, d, B].  Blocks of the first column chunk also write the
// indices and labels.  d is a multiple of 8, B a multiple of 16.
template <typename TIN>
__global__ void __launch_bounds__(256)
k_sample_gather(const TIN* __restrict__ x, const int32_t* __restrict__ y, uint64_t seed,
                int64_t round, const int64_t* __restrict__ round_ptr, int step, int P, int B,
                int64_t S, int d, int32_t* __restrict__ idx_out, int32_t* __restrict__ labels_out,
                __nv_bfloat16* __restrict__ out_bf, __nv_bfloat16* __restrict__ out_bft) {
  __shared__ int32_t sidx[32];
  __shared__ __nv_bfloat16 tile[32][66];
  const int p = blockIdx.z, s0 = blockIdx.x * 32, c0 = blockIdx.y * 64;
  const int tx = threadIdx.x, ty = threadIdx.y;
  if (round_ptr) round = *round_ptr;
  if (ty == 0) {
    const int s = s0 + tx;
    int32_t i = 0;
    if (s < B) {
      i = sample_index(seed, round, p, step, s, P, S);
      if (blockIdx.y == 0) {
        idx_out[p * B + s] = i;
        labels_out[p * B + s] = y[i];
      }
    }
    sidx[tx] = i;
  }
  __syncthreads();
  const int c = c0 + 2 * tx;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int sl = ty + 8 * r, s = s0 + sl;
    __nv_bfloat16 v0 = __float2bfloat16_rn(0.f), v1 = v0;
    if (s < B && c < d) {                      // d is even: c + 1 < d as well
      const TIN* src = x + (size_t)sidx[sl] * d + c;
      v0 = __float2bfloat16_rn(to_f32<TIN>(src[0]));
      v1 = __float2bfloat16_rn(to_f32<TIN>(src[1]));
      __nv_bfloat162 pr;
      pr.x = v0; pr.y = v1;
      *reinterpret_cast<__nv_bfloat162*>(out_bf + ((size_t)p * B + s) * d + c) = pr;
    }
    tile[sl][2 * tx] = v0;
    tile[sl][2 * tx + 1] = v1;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int cl = ty + 8 * r, cc = c0 + cl, s = s0 + tx;
    if (cc < d && s < B) out_bft[((size_t)p * d + cc) * B + s] = tile[tx][cl];
  }
}

}  // namespace

cudaError_t launch_batch_indices(mavg_ctx* c, int64_t round, int step, int j, int32_t* idx) {
  const int B = c->cfg.B;
  prof_begin(c, MAVG_K_BATCH);
  k_batch_indices<<<(B + 255) / 256, 256, 0, c->stream>>>(idx, c->cfg.seed, round, step, c->cfg.P, B,
                                                          c->cfg.n_samples, j);
  prof_end(c);
  return cudaGetLastError();
}

cudaError_t launch_sample_gather(mavg_ctx* c, int64_t round, int step, int32_t* idx,
                                 int32_t* labels, __nv_bfloat16* out_bf, __nv_bfloat16* out_bft) {
  const int P = c->cfg.P, B = c->cfg.B, d = c->cfg.dims[0];
  dim3 grid((B + 31) / 32, (d + 63) / 64, P), block(32, 8);
  const int64_t* rp = c->capturing ? (const int64_t*)(ws_ptr(c, c->ws.status) + 64) : nullptr;
  prof_begin(c, MAVG_K_BATCH);
  if (c->cfg.x_dtype == MAVG_X_BF16)
    k_sample_gather<__nv_bfloat16><<<grid, block, 0, c->stream>>>(
        (const __nv_bfloat16*)c->cfg.x, c->cfg.y, c->cfg.seed, round, rp, step, P, B,
        c->cfg.n_samples, d, idx, labels, out_bf, out_bft);
  else
    k_sample_gather<float><<<grid, block, 0, c->stream>>>(
        (const float*)c->cfg.x, c->cfg.y, c->cfg.seed, round, rp, step, P, B, c->cfg.n_samples, d,
        idx, labels, out_bf, out_bft);
  prof_end(c);
  return cudaGetLastError();
}

}  // namespace mavg

namespace mavg {
// ------------------------------------------------------------------------------------------------
// mavg_batch_indices_noalloc: the index stream without a handle and without any allocation.
// The B indices are staged in a fixed array that lives in the library's device image (every GPU
// that loads the library carries these 256 KB until the process exits) and are then copied to
// the caller's host buffer.
namespace {

constexpr int kNoAllocMaxB = 65536;
static __device__ __align__(256) int32_t g_noalloc_idx[kNoAllocMaxB];

constexpr int kNoAllocMaxDevices = 64;
int32_t* g_noalloc_ptr[kNoAllocMaxDevices] = {};
std::mutex g_noalloc_mutex;

// In host code the array's name is only a handle for the runtime, not a device address; the
// address on the current device is looked up once per device and remembered.
cudaError_t noalloc_scratch(int device, int32_t** out) {
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[device]) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_idx);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[device] = (int32_t*)ptr;
  }
  *out = g_noalloc_ptr[device];
  return cudaSuccess;
}

}  // namespace
}  // namespace mavg

extern "C" mavg_status mavg_batch_indices_noalloc(uint64_t seed, int64_t round, int32_t P,
                                                  int32_t learner, int32_t step,
                                                  int64_t n_samples, int32_t B, void* stream,
                                                  int32_t* out) {
  using namespace mavg;
  if (!out || round < 1 || step < 1 || P < 1 || learner < 0 || learner >= P || B < 1 ||
      n_samples < P || n_samples >= ((int64_t)1 << 31)) {
    set_thread_error("mavg_batch_indices_noalloc: bad round, P, learner, step, n_samples, B or out");
    return MAVG_ERR_INVALID_ARG;
  }
  if (B > kNoAllocMaxB) {
    set_thread_error("mavg_batch_indices_noalloc: B exceeds the built-in staging array of 65536 "
                     "indices; use mavg_get_batch_indices with a workspace instead");
    return MAVG_ERR_INVALID_ARG;
  }
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e == cudaSuccess && (device < 0 || device >= kNoAllocMaxDevices)) {
    set_thread_error("mavg_batch_indices_noalloc: device ordinal out of range");
    return MAVG_ERR_UNSUPPORTED;
  }
  int32_t* scratch = nullptr;
  if (e == cudaSuccess) e = noalloc_scratch(device, &scratch);
  cudaStream_t s = (cudaStream_t)stream;
  if (e == cudaSuccess) {
    k_batch_indices<<<(B + 255) / 256, 256, 0, s>>>(scratch, seed, round, step, P, B, n_samples,
                                                    learner);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out, scratch, (size_t)B * sizeof(int32_t), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    set_thread_error(std::string("mavg_batch_indices_noalloc: ") + cudaGetErrorString(e));
    return MAVG_ERR_CUDA;
  }
  return MAVG_OK;
}
