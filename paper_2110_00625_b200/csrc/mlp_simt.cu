// MLP learner step of models that the bf16 tensor-core path does not take: true fp32 arithmetic, and bf16 operands of
// any widths, batch size and class count; batched over the P learners.
//   forward   Z_l = A_{l-1} W_l^T + b_l,  A_l = act(Z_l)          (A_0 = gathered minibatch)
//   backward  dA_{l-1} = (dZ_l W_l) .* [A_{l-1} > 0];  dW_l = dZ_l^T A_{l-1};  db_l = colsum dZ_l
//   SGD       W_l <- W_l - gamma dW_l, b_l <- b_l - gamma db_l    (Algorithm 1's local update)
// The products run on tcgen05 with fp32 operands as three bf16 planes, or with QUANT on the operands rounded to bf16
// (nearest-even) as one, which makes this path compute the same thing as the tensor-core path (split_gemm.cuh).
// Rounds of 3072-512-512-10, P = 4, K = 4, B = 100 in fp32: 366 us, 570 with chains of FMAs on the CUDA cores (53 us for
// layer 1's forward product, 22 here; 55 for the weight gradients, 24 to 32 here); 1000-333-100, P = 6, K = 4, B = 50 with
// bf16 operands: 127 us, 170 with warp-level MMAs.  Relative error of one step's gradients against 64 bits (2-norm, weight
// matrices of layers 1, 2, .. in units of 1e-7, FMA chains / here): 3072-512-512-10, B = 100 2.8 3.2 2.8 / 1.8 1.8 2.4;
// inputs in [0, 1] 1.9 2.8 2.8 / 1.9 1.8 1.9, B = 192 2.3 2.8 2.9 / 1.6 1.5 1.6, B = 256 2.4 2.9 2.8 / 1.9 1.8 1.9, B = 300
// 2.6 3.0 3.0 / 1.7 1.6 1.6; 2900-130-800-77, B = 31 2.8 3.8 3.4 / 2.1 2.4 2.1; 1501-799-99, B = 129 2.5 2.8 / 1.9 2.0;
// 301-131-66-5, B = 256, [0, 1] 2.2 2.2 2.4 / 1.7 1.5 1.5; 700-300-10, B = 512, [0, 1] 3.1 3.3 / 1.5 1.5.  With two slabs to
// an accumulator of a forward product 2.8 3.0 3.4 where it is 1.9 1.9 2.0.
// A step is L-1 forward launches, one for the whole last layer up to its data gradient (which
// also gathers the next step's minibatch), L-2 data gradients and one for the weight gradients,
// bias gradients and SGD steps of all layers.  While a deferred re-broadcast is outstanding the first
// step of a round reads the weights from w~ and writes the results to the replicas, so its P copies
// are never needed.
#include <algorithm>
#include <array>
#include <map>
#include <mutex>

#include "mlp.cuh"
#include "split_gemm.cuh"
#include "tensor_map.cuh"

namespace mavg {
namespace {

using split::pitch_of;

__device__ __forceinline__ float qbf(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
template <bool QUANT>
__device__ __forceinline__ float operand(float v) { return QUANT ? qbf(v) : v; }
template <bool QUANT> constexpr int kPlanes = QUANT ? 1 : 3;

// ------------------------------------------------------------------------- minibatch and loss
struct GatherArgs {
  const void* x; int x_bf16;
  const int32_t* y;
  uint64_t seed; int64_t round; const int64_t* round_ptr;
  int step, P, p0, n, B, d;            // learners p0 .. p0 + n - 1 of P
  int64_t S;
  __nv_bfloat16* out; int64_t plane;   // planes [n, B, pitch_of(d)]
  int32_t* labels;                     // [n, B]
};

// One sampled row: index, label and the row itself.
template <bool QUANT>
__device__ __forceinline__ void gather_row(const GatherArgs& g, int row) {
  constexpr int NP = kPlanes<QUANT>;
  __shared__ int32_t sidx;
  if (threadIdx.x == 0) {
    const int64_t round = g.round_ptr ? *g.round_ptr : g.round;
    sidx = sample_index(g.seed, round, g.p0 + row / g.B, g.step, row % g.B, g.P, g.S);
    g.labels[row] = g.y[sidx];
  }
  __syncthreads();
  const size_t src = (size_t)sidx * g.d;
  const int pitch = pitch_of(g.d);
  __nv_bfloat16* dst = g.out + (size_t)row * pitch;
  const bool vec = g.d % 8 == 0;
  for (int c = 8 * threadIdx.x; c < pitch; c += 8 * blockDim.x) {
    uint4 pl[NP];
    if (QUANT && g.x_bf16 && vec) {
      pl[0] = *reinterpret_cast<const uint4*>((const __nv_bfloat16*)g.x + src + c);
    } else {
      float v[8];
      if (g.x_bf16) {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = c + i < g.d ? __bfloat162float(((const __nv_bfloat16*)g.x)[src + c + i]) : 0.f;
      } else if (vec) {
        const float4* x = reinterpret_cast<const float4*>((const float*)g.x + src + c);
        const float4 a = x[0], b = x[1];
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = c + i < g.d ? ((const float*)g.x)[src + c + i] : 0.f;
      }
      split::split8<NP>(v, pl);
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) *reinterpret_cast<uint4*>(dst + q * g.plane + c) = pl[q];
  }
}

// A call's first launch: its first minibatch, a block per row, and the planes of the weights it starts from, eight
// rows per block.
template <bool QUANT>
__global__ void __launch_bounds__(256)
k_simt_begin(const __grid_constant__ GatherArgs g, const __grid_constant__ split::SplitWeights w) {
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();
  if ((int)blockIdx.x < g.n * g.B) {
    gather_row<QUANT>(g, blockIdx.x);
    return;
  }
  const int row = ((int)blockIdx.x - g.n * g.B) * 8 + (int)threadIdx.x / 32;
  if (row < w.copies * w.first[w.L]) split::split_weight_row<kPlanes<QUANT>>(w, row);
}

// Softmax of one row z (C logits in shared or global memory) by a warp: writes dz and returns the loss.
template <typename Put>
__device__ __forceinline__ float softmax_row(const float* z, int C, int label, float inv_b, Put put) {
  const int lane = threadIdx.x % 32;
  if (C <= 128) {                          // four classes a lane, read once
    float v[4], m = -INFINITY, se = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = lane + 32 * q < C ? z[lane + 32 * q] : -INFINITY;
#pragma unroll
    for (int q = 0; q < 4; ++q) m = fmaxf(m, v[q]);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (lane + 32 * q < C) se += expf(v[q] - m);
    for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
    const float lse = m + logf(se);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (lane + 32 * q < C) put(lane + 32 * q, (expf(v[q] - lse) - (lane + 32 * q == label ? 1.f : 0.f)) * inv_b);
    return lse - z[label];
  }
  float m = z[lane < C ? lane : 0];
  for (int c = lane + 32; c < C; c += 32) m = fmaxf(m, z[c]);
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  float se = 0.f;
  for (int c = lane; c < C; c += 32) se += expf(z[c] - m);
  for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
  const float lse = m + logf(se);
  for (int c = lane; c < C; c += 32) put(c, (expf(z[c] - lse) - (c == label ? 1.f : 0.f)) * inv_b);
  return lse - z[label];
}

constexpr int kTailRows = 8, kTailThreads = 512;

// `count` contiguous floats into shared memory, 16 bytes per load wherever the source starts, eight loads of a
// thread in flight.
template <bool QUANT>
__device__ __forceinline__ void copy_floats(float* dst, const float* __restrict__ src, int count) {
  const int head = min(count, (int)((16 - ((uintptr_t)src & 15)) & 15) / 4), n4 = (count - head) / 4;
  const int t = threadIdx.x;
  const float4* s4 = reinterpret_cast<const float4*>(src + head);
  for (int i0 = t; i0 < n4; i0 += 8 * kTailThreads) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (i0 + u * kTailThreads < n4) v[u] = s4[i0 + u * kTailThreads];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = i0 + u * kTailThreads;
      if (i >= n4) break;
      float* d = dst + head + 4 * i;
      d[0] = operand<QUANT>(v[u].x);
      d[1] = operand<QUANT>(v[u].y);
      d[2] = operand<QUANT>(v[u].z);
      d[3] = operand<QUANT>(v[u].w);
    }
  }
  const int rest = count - head - 4 * n4;
  if (t < head) dst[t] = operand<QUANT>(src[t]);
  if (t < rest) dst[head + 4 * n4 + t] = operand<QUANT>(src[head + 4 * n4 + t]);
}

// Elements of a bf16 row in shared memory: whole groups of 16, then an odd number of 16-byte units.
__host__ __device__ constexpr int bf_pitch(int n) { return (((n + 15) / 16 * 16 >> 3) | 1) << 3; }

// The last layer of 8 batch rows of a learner: logits, loss, dZ_L and the data gradient through the
// layer, in one block of 512 threads; the remaining blocks gather the next step's minibatch.  A
// layer of few classes is latency, not work: as a forward product, a loss and a data gradient it
// takes three launches with one busy tile column (25 us for 512 x 10, P = 4, B = 100, against
// 9 here).  The layer's weights and the rows' activations are brought into shared memory at once, which exposes one
// trip to the L2.  For the logits a warp takes
// two rows and every fourth group of four classes (lanes along the input width); for the data
// gradient a thread takes two columns of the input and four rows.
// Dynamic shared memory: dZ [C][8], logits [8][C], the rows of A_{L-1} [8][in], W_L [C][in].
// With bf16 operands the two products are warp-level MMAs on the bf16 planes (mma_tail), whose rows come in by
// asynchronous copies, with the operands of four MMAs fetched together: 333 x 100, P = 6, B = 50 9 us (24 with FMAs; 14 with
// the fp32 weights rounded on their way in, 12 with a load, a wait and an MMA at a time and the planes through registers).
struct TailArgs {
  const __nv_bfloat16* a; int64_t a_plane; // A_{L-1}: planes [P, B, pitch_of(in)]
  const float* w; const float* b; int64_t w_batch;
  const int32_t* labels;
  int P, B, in, C, row_blocks;
  float* row_loss;                         // [P, B]
  float* dz;                               // [P, B, C]
  float* dzp;                              // dZ_{L-1} [P, B, in], null for a one-layer model
  __nv_bfloat16* dz_pl; int64_t dz_plane;  // both as planes of rows of pitch_of(C), pitch_of(in)
  __nv_bfloat16* dzp_pl; int64_t dzp_plane;
  bool mma;                                // bf16 operands on warp-level MMAs (mma_tail) ...
  const __nv_bfloat16* w16; int64_t w16_batch;   // ... with W_L from its plane
};

// k_simt_tail's block with bf16 operands.  Dynamic shared memory: W_L [C, to a multiple of 16][in], the rows of
// A_{L-1} [16][in] (the last eight are zero), dZ [16][C], all bf16; logits [8][C].
__device__ __forceinline__ void mma_tail(const TailArgs& t, int p, int r0, uint8_t* smem) {
  const int rows = min(kTailRows, t.B - r0), in = t.in, C = t.C;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int ip = bf_pitch(in), dp = bf_pitch(C), c16 = (C + 15) / 16 * 16, in16 = (in + 15) / 16 * 16;
  __nv_bfloat16* w = reinterpret_cast<__nv_bfloat16*>(smem);
  __nv_bfloat16* a = w + (size_t)c16 * ip;
  __nv_bfloat16* dq = a + 16 * ip;
  float* z = reinterpret_cast<float*>(dq + 16 * dp);
  const float* bias = t.b + (size_t)p * t.w_batch;
  // Rows of the planes come in as they are, 16 bytes at a time and all on their way at once: what lies behind a row's end
  // is zero there (products and gathers write it so, W_L's was cleared when the handle was made).  Zeros: the rows'
  // columns beyond the planes' pitch, rows beyond the last class and the batch rows, and dZ.
  const int pitch = pitch_of(in), units = pitch / 8, left = in16 - pitch;      // 0 or 8
  auto fill = [&](__nv_bfloat16* dst, const __nv_bfloat16* __restrict__ src, int count, int padded) {
    int r = threadIdx.x / units, k = threadIdx.x - r * units;
    const int dr = kTailThreads / units, dk = kTailThreads - dr * units;
    while (r < count) {
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(tc::smem_u32(dst + r * ip + 8 * k)),
                   "l"(src + (size_t)r * pitch + 8 * k) : "memory");
      r += dr;
      if ((k += dk) >= units) { k -= units; ++r; }
    }
    if (left)
      for (int i = threadIdx.x; i < count; i += kTailThreads) *reinterpret_cast<uint4*>(dst + i * ip + pitch) = make_uint4(0, 0, 0, 0);
    const int n = (padded - count) * ip / 8;
    for (int i = threadIdx.x; i < n; i += kTailThreads) reinterpret_cast<uint4*>(dst + count * ip)[i] = make_uint4(0, 0, 0, 0);
  };
  fill(w, t.w16 + (size_t)p * t.w16_batch, C, c16);
  fill(a, t.a + ((size_t)p * t.B + r0) * pitch, rows, 16);
  for (int i = threadIdx.x; i < 16 * dp / 8; i += kTailThreads) reinterpret_cast<uint4*>(dq)[i] = make_uint4(0, 0, 0, 0);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int i8 = lane / 8, j8 = lane % 8, qr = lane / 4, qc = 2 * (lane % 4);
  for (int nt = warp; nt < (C + 7) / 8; nt += kTailThreads / 32) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = 0; k0 < in16; k0 += 64) {            // 64 inputs' sum on its own: the MMAs cut off, see split_gemm.cuh
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t fa[4][4], fb[4][2];                     // the operands of four steps together
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k0 + 16 * u < in16) {
          tc::ldsm_x4(fa[u], a + ((i8 & 1) * 8 + j8) * ip + k0 + 16 * u + (i8 >> 1) * 8);
          tc::ldsm_x2(fb[u], w + (size_t)(nt * 8 + j8) * ip + k0 + 16 * u + (i8 & 1) * 8);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k0 + 16 * u < in16) tc::mma_bf16(d, fa[u], fb[u][0], fb[u][1]);
      s[0] += d[0];
      s[1] += d[1];
    }
    const int c = nt * 8 + qc;
    if (c < C) z[qr * C + c] = s[0] + bias[c];
    if (c + 1 < C) z[qr * C + c + 1] = s[1] + bias[c + 1];
  }
  __syncthreads();
  if (warp < rows) {
    const size_t row = (size_t)p * t.B + r0 + warp;
    const float loss = softmax_row(z + warp * C, C, t.labels[row], 1.0f / (float)t.B, [&](int c, float g) {
      t.dz[row * C + c] = g;
      dq[warp * dp + c] = __float2bfloat16_rn(g);
      t.dz_pl[row * pitch_of(C) + c] = dq[warp * dp + c];
    });
    if (lane == 0) t.row_loss[row] = loss;
  }
  if (!t.dzp) return;
  __syncthreads();
  for (int nt = warp; nt < (in + 7) / 8; nt += kTailThreads / 32) {
    float s[2] = {0.f, 0.f};
    for (int k0 = 0; k0 < c16; k0 += 64) {             // 64 classes' sum on its own, likewise
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t fa[4][4], fb[4][2];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k0 + 16 * u < c16) {
          tc::ldsm_x4(fa[u], dq + ((i8 & 1) * 8 + j8) * dp + k0 + 16 * u + (i8 >> 1) * 8);
          tc::ldsm_x2_t(fb[u], w + (size_t)(k0 + 16 * u + (i8 & 1) * 8 + j8) * ip + nt * 8);
        }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k0 + 16 * u < c16) tc::mma_bf16(d, fa[u], fb[u][0], fb[u][1]);
      s[0] += d[0];
      s[1] += d[1];
    }
    const int i = nt * 8 + qc;
    if (qr < rows && i < in) {                         // ReLU'(0) = 0
      const size_t row = (size_t)p * t.B + r0 + qr;
      const float2 act = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(a + qr * ip + i));
      const float v0 = act.x > 0.f ? s[0] : 0.f, v1 = act.y > 0.f ? s[1] : 0.f;
      t.dzp[row * in + i] = v0;
      if (i + 1 < in) t.dzp[row * in + i + 1] = v1;
      *reinterpret_cast<__nv_bfloat162*>(t.dzp_pl + row * pitch + i) = __floats2bfloat162_rn(v0, v1);   // (i + 1 == in: 0)
    }
  }
}

template <bool QUANT>
__global__ void __launch_bounds__(kTailThreads)
k_simt_tail(const __grid_constant__ TailArgs t, const __grid_constant__ GatherArgs next) {
  extern __shared__ __align__(16) float sm[];
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();
  if ((int)blockIdx.x >= t.P * t.row_blocks) {
    gather_row<QUANT>(next, blockIdx.x - t.P * t.row_blocks);
    return;
  }
  const int p = blockIdx.x / t.row_blocks, r0 = blockIdx.x % t.row_blocks * kTailRows;
  if (QUANT && t.mma) {
    mma_tail(t, p, r0, reinterpret_cast<uint8_t*>(sm));
    return;
  }
  const int rows = min(kTailRows, t.B - r0), in = t.in, C = t.C;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  float* dzq = sm;                         // [C][8], operand of the data gradient
  float* z = dzq + kTailRows * C;          // [8][C]
  float* a = z + kTailRows * C;            // [8][in]
  const float* W = t.w + (size_t)p * t.w_batch;
  const float* bias = t.b + (size_t)p * t.w_batch;
  constexpr int NP = kPlanes<QUANT>;
  const int pitch = pitch_of(in);
  const __nv_bfloat16* arow = t.a + ((size_t)p * t.B + r0) * pitch;
  float* w = a + kTailRows * in;
  copy_floats<QUANT>(w, W, C * in);
  // a value is the sum of its planes, the small ones first; four of a thread's pairs on their way at once
  const int pairs = pitch / 2;
  for (int i0 = threadIdx.x; i0 < kTailRows * pairs; i0 += 4 * kTailThreads) {
    uint32_t h[4][NP];
    int r[4], k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * kTailThreads;
      r[u] = i / pairs;
      k[u] = 2 * (i - r[u] * pairs);
#pragma unroll
      for (int q = 0; q < NP; ++q)
        h[u][q] = r[u] < rows ? *reinterpret_cast<const uint32_t*>(arow + q * t.a_plane + (size_t)r[u] * pitch + k[u]) : 0u;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (r[u] >= kTailRows) break;
      float x0 = 0.f, x1 = 0.f;
#pragma unroll
      for (int q = NP - 1; q >= 0; --q) {
        x0 += __uint_as_float(h[u][q] << 16);
        x1 += __uint_as_float(h[u][q] & 0xffff0000u);
      }
      if (k[u] < in) a[r[u] * in + k[u]] = x0;
      if (k[u] + 1 < in) a[r[u] * in + k[u] + 1] = x1;
    }
  }
  __syncthreads();
  {
    const int r = warp % 4 * 2;
    const float* x = a + r * in;
    for (int c0 = warp / 4 * 4; c0 < C; c0 += kTailThreads / 32) {
      float s[2][4] = {};
      const int last = C - 1 - c0;         // classes beyond the last repeat it
      const float* w0 = w + c0 * in;
      const float* wr[4] = {w0, w0 + min(1, last) * in, w0 + min(2, last) * in, w0 + min(3, last) * in};
#pragma unroll 4
      for (int i = lane; i < in; i += 32) {
        const float x0 = x[i], x1 = x[in + i];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float wv = wr[q][i];
          s[0][q] = fmaf(x0, wv, s[0][q]);
          s[1][q] = fmaf(x1, wv, s[1][q]);
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          for (int o = 16; o > 0; o >>= 1) s[h][q] += __shfl_xor_sync(0xffffffffu, s[h][q], o);
          if (lane == 4 * h + q && q <= last) z[(r + h) * C + c0 + q] = s[h][q] + bias[c0 + q];
        }
    }
  }
  __syncthreads();
  if (warp < rows) {
    const size_t row = (size_t)p * t.B + r0 + warp;
    const float loss = softmax_row(z + warp * C, C, t.labels[row], 1.0f / (float)t.B, [&](int c, float g) {
      t.dz[row * C + c] = g;
      split::put_planes<NP>(t.dz_pl, t.dz_plane, row * pitch_of(C) + c, g);
      dzq[c * kTailRows + warp] = operand<QUANT>(g);
    });
    if (lane == 0) t.row_loss[row] = loss;
  } else if (warp < kTailRows) {
    for (int c = lane; c < C; c += 32) dzq[c * kTailRows + warp] = 0.f;
  }
  if (!t.dzp) return;
  __syncthreads();
  constexpr int kCols = kTailThreads / 2;
  const int rh = threadIdx.x / kCols * 4;            // first of this thread's four rows
  for (int i0 = threadIdx.x % kCols; i0 < in; i0 += 2 * kCols) {
    const int i1 = i0 + kCols < in ? i0 + kCols : i0;   // i0 again: stored once
    float s[2][4] = {};
#pragma unroll 4
    for (int c = 0; c < C; ++c) {
      const float wv[2] = {w[c * in + i0], w[c * in + i1]};
      const float4 dv = *reinterpret_cast<const float4*>(dzq + c * kTailRows + rh);
      const float d[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int r = 0; r < 4; ++r) s[h][r] = fmaf(d[r], wv[h], s[h][r]);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = h ? i1 : i0;
      if (h && i1 == i0) break;
#pragma unroll
      for (int r = 0; r < 4; ++r)                // ReLU'(0) = 0
        if (rh + r < rows) {
          const size_t row = (size_t)p * t.B + r0 + rh + r;
          const float v = a[(rh + r) * in + i] > 0.f ? s[h][r] : 0.f;
          t.dzp[row * in + i] = v;
          split::put_planes<NP>(t.dzp_pl, t.dzp_plane, row * pitch + i, v);
        }
    }
  }
}

// Loss and dZ_L from the logits, for last layers too large for k_simt_tail.  Blocks 0..P-1: a learner's B
// rows, a warp per row; the remaining blocks gather the next step's minibatch.
template <bool QUANT>
__global__ void __launch_bounds__(1024)
k_simt_loss(const float* __restrict__ logits, const int32_t* __restrict__ labels, int P, int B, int C,
            float* __restrict__ row_loss, float* __restrict__ dz, __nv_bfloat16* __restrict__ dz_pl, int64_t dz_plane,
            const __grid_constant__ GatherArgs next) {
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();
  if ((int)blockIdx.x >= P) {
    gather_row<QUANT>(next, blockIdx.x - P);
    return;
  }
  const int p = blockIdx.x;
  for (int b = threadIdx.x / 32; b < B; b += 32) {
    const size_t row = (size_t)p * B + b;
    const float loss = softmax_row(logits + row * C, C, labels[row], 1.0f / (float)B, [&](int c, float g) {
      dz[row * C + c] = g;
      split::put_planes<kPlanes<QUANT>>(dz_pl, dz_plane, row * pitch_of(C) + c, g);
    });
    if (threadIdx.x % 32 == 0) row_loss[row] = loss;
  }
}

// ---------------------------------------------------------------------------------- host side
// (P: the learners that take their steps together)
struct SimtBuffers {
  __nv_bfloat16* xg[2];                    // planes [P, B, pitch]: the minibatch, alternate steps
  int32_t* labels[2];                      // [P, B]
  float* row_loss;                         // [P, B]
  float* logits;                           // [P, B, C], where the last layer is a product of its own
  __nv_bfloat16* a[MAVG_MAX_LAYERS + 1];   // planes: A_l, l < L
  __nv_bfloat16* dz[MAVG_MAX_LAYERS + 1];  // planes: dZ_l
  float* dz_f[MAVG_MAX_LAYERS + 1];        // [P, B, d_l]: dZ_l unrounded, for the bias gradients
  __nv_bfloat16* w[MAVG_MAX_LAYERS + 1];   // planes [P + 1, d_l, pitch]: W_l of the learners and of w~, where they are read
};

// Last layer in one launch (k_simt_tail) where its weights fit in an SM's shared memory.
constexpr size_t kTailSmem = 200 * 1024;
size_t tail_smem(int in, int C, bool quant) {
  if (quant)
    return ((size_t)((C + 15) / 16 * 16 + 16) * bf_pitch(in) + (size_t)16 * bf_pitch(C)) * 2 +
           (size_t)kTailRows * C * sizeof(float);
  return ((size_t)kTailRows * in + 2 * (size_t)kTailRows * C + (size_t)in * C) * sizeof(float);
}
bool use_tail(int in, int C) { return tail_smem(in, C, false) <= kTailSmem; }
// Layers whose weights are an operand of products.
int product_layers(const mavg_config* cfg) {
  const int L = cfg->n_layers;
  return use_tail(cfg->dims[L - 1], cfg->dims[L]) ? L - 1 : L;
}

// Layers whose weights are kept as planes: those, and with bf16 operands the last one (mma_tail).
int plane_layers(const mavg_config* cfg) { return cfg->gemm_bf16 ? cfg->n_layers : product_layers(cfg); }

size_t carve(const mavg_config* cfg, int learners, char* base, SimtBuffers* sb) {
  const size_t rows = (size_t)learners * cfg->B;
  const int np = cfg->gemm_bf16 ? kPlanes<true> : kPlanes<false>;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base + off;
    off += (bytes + 255) / 256 * 256;
    return p;
  };
  auto planes = [&](int d) { return (__nv_bfloat16*)take(np * rows * pitch_of(d) * 2); };
  for (int i = 0; i < 2; ++i) {
    sb->xg[i] = planes(cfg->dims[0]);
    sb->labels[i] = (int32_t*)take(rows * 4);
  }
  sb->row_loss = (float*)take(rows * 4);
  sb->logits = (float*)take(rows * cfg->dims[cfg->n_layers] * 4);
  for (int l = 1; l <= cfg->n_layers; ++l) {
    if (l < cfg->n_layers) sb->a[l] = planes(cfg->dims[l]);
    sb->dz[l] = planes(cfg->dims[l]);
    sb->dz_f[l] = (float*)take(rows * cfg->dims[l] * 4);
  }
  for (int l = 1; l <= plane_layers(cfg); ++l)
    sb->w[l] = (__nv_bfloat16*)take((size_t)np * (learners + 1) * cfg->dims[l] * pitch_of(cfg->dims[l - 1]) * 2);
  return off;
}

// Maps of the planes: as the column operand of a product (boxes of 64 columns x a tile's batch rows), and for the
// weight gradients (boxes of 64 x 64).
struct SimtState {
  SimtBuffers buf;
  int group;                               // learners that take their steps together: all of them where the scratch has room
  int n_tiles, N;                          // batch tiles of a product
  int resident[9];                         // resident_clusters()
  CUtensorMap x[2], x_mn[2];
  CUtensorMap a[MAVG_MAX_LAYERS + 1], a_mn[MAVG_MAX_LAYERS + 1], dz[MAVG_MAX_LAYERS + 1], dz_mn[MAVG_MAX_LAYERS + 1];
  CUtensorMap w[MAVG_MAX_LAYERS + 1], w_mn[MAVG_MAX_LAYERS + 1];   // boxes of 64 x 128, 64 x 64
};

// Every launch of the chain may begin while its predecessor finishes; the kernels wait for it
// before they touch memory.
template <typename... Params, typename... Args>
cudaError_t launch(mavg_ctx* c, int cls, void (*kernel)(Params...), dim3 grid, int threads,
                   int cluster, size_t smem, const Args&... args) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = grid;
  lc.dynamicSmemBytes = smem;
  lc.blockDim = dim3((unsigned)threads);
  lc.stream = c->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = cluster > 1 ? 2 : 1;
  prof_begin(c, cls);
  cudaError_t e = cudaLaunchKernelEx(&lc, kernel, args...);
  prof_end(c);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Forward product or data gradient.
template <bool QUANT, bool DGRAD>
cudaError_t launch_product(mavg_ctx* c, int cls, int n, const CUtensorMap& w, bool shared_w, const CUtensorMap& x, split::ProductArgs g) {
  constexpr int NP = kPlanes<QUANT>;
  const SimtState* st = (const SimtState*)c->simt;
  const split::LaunchShape sh = split::product_shape(NP, st->N);
  g.P = st->group;
  g.B = c->cfg.B;
  g.N = st->N;
  g.n_tiles = st->n_tiles;
  g.m_tiles = (g.M + split::kTile - 1) / split::kTile;
  g.w_first = shared_w ? g.P : 0;
  g.w_step = shared_w ? 0 : 1;
  g.w_plane = g.P + 1;
  g.plane = (int64_t)g.P * g.B * g.pitch;
  g.stages = sh.stages;
  g.tmem_cols = sh.tmem_cols;
  g.status = (int*)ws_ptr(c, c->ws.status);
  // Blocks of a tile: as many as the GPU holds for all tiles at once (a cluster's blocks share a GPC: 15 clusters of
  // eight are resident, 22 of six, 33 of four).  us a round with at least two slabs to a block / with one: 2310-309-187-94,
  // P = 4, K = 2, B = 42 143 / 134, 322-266-305-5, P = 2, K = 3, B = 37 151 / 138; with at most four blocks to a tile
  // 3072-512-512-10, P = 4, K = 4, B = 100 403 for 381.
  const int slabs = (g.K + split::kSlab - 1) / split::kSlab;
  const int64_t tiles = (int64_t)g.m_tiles * g.n_tiles * c->cfg.P;   // (of all learners: the same sums in groups)
  g.splits = 1;
  for (int s = 2; s <= 8 && slabs >= s; ++s)
    if (tiles <= st->resident[s]) g.splits = s;
  g.per_split = (slabs + g.splits - 1) / g.splits;
  g.splits = (slabs + g.per_split - 1) / g.per_split;
  return launch(c, cls, split::k_split_product<NP, DGRAD>, dim3((unsigned)(g.splits * g.m_tiles * g.n_tiles), 1, (unsigned)n),
                split::kProductThreads, g.splits, sh.smem, w, x, g);
}

typedef void (*WgradKernel)(split::WgradArgs);
template <bool QUANT>
WgradKernel wgrad_kernel(int B, bool momentum) {
  constexpr int NP = kPlanes<QUANT>, kTwo = NP == 3 ? 2 : 1;   // (one plane: never two)
  const int chains = split::wgrad_chains(NP, B);
  auto pick = [&](auto one, auto two, auto many) { return chains == 1 ? one : chains == 2 ? two : many; };
  return momentum ? pick(split::k_split_wgrad<NP, true, 1>, split::k_split_wgrad<NP, true, kTwo>, split::k_split_wgrad<NP, true, split::kManyChains>)
                  : pick(split::k_split_wgrad<NP, false, 1>, split::k_split_wgrad<NP, false, kTwo>, split::k_split_wgrad<NP, false, split::kManyChains>);
}

// Every kernel of a step asks for the same split of the SM's memory: a launch that needs another
// split than the kernel before it has to wait until the SM is empty.  Only kernels that the handle's steps launch are asked
// for: the first call for one loads it (1000-333-100 with bf16 operands: a process's first handle takes 9.6 ms, 10.7 with all).
template <bool QUANT>
cudaError_t set_attributes(const mavg_ctx* c) {
  constexpr int NP = kPlanes<QUANT>;
  const mavg_config& cfg = c->cfg;
  const bool tail = product_layers(&cfg) < cfg.n_layers;
  const struct { const void* kernel; size_t smem; bool used; } kernels[] = {
      {(const void*)split::k_split_product<NP, false>, split::kSmem, true},
      {(const void*)split::k_split_product<NP, true>, split::kSmem, !tail || cfg.n_layers > 2},
      {(const void*)wgrad_kernel<QUANT>(cfg.B, false), split::kSmem, true},
      {(const void*)wgrad_kernel<QUANT>(cfg.B, true), split::kSmem, c->buf.learner_u != nullptr},
      {(const void*)k_simt_begin<QUANT>, 0, true}, {(const void*)k_simt_loss<QUANT>, 0, !tail}, {(const void*)k_simt_tail<QUANT>, kTailSmem, tail}};
  for (const auto& k : kernels) {
    if (!k.used) continue;
    cudaError_t e = cudaFuncSetAttribute(k.kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess && k.smem) e = cudaFuncSetAttribute(k.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Clusters of s product blocks that the GPU holds at once, at [s]; 0 where the query is refused: such a split is not taken.
// Asked once per device and shape of a product (one or three planes, batch tiles of 16 to 128 rows).
void resident_clusters(int device, int np, int N, int (&resident)[9]) {
  static std::mutex mu;
  static std::map<std::array<int, 3>, std::array<int, 9>> known;
  std::lock_guard<std::mutex> lock(mu);
  const std::array<int, 3> key{device, np, N};
  auto it = known.find(key);
  std::array<int, 9> got{};
  if (it != known.end()) {
    got = it->second;
  } else {
    bool all = true;
    for (int s = 2; s <= 8; ++s) {
      cudaLaunchAttribute at[1];
      cudaLaunchConfig_t lc{};
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = (unsigned)s;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      lc.gridDim = dim3((unsigned)s);
      lc.blockDim = dim3(split::kProductThreads);
      lc.dynamicSmemBytes = split::product_shape(np, N).smem;
      lc.attrs = at;
      lc.numAttrs = 1;
      const cudaError_t e = np == 1 ? cudaOccupancyMaxActiveClusters(&got[s], split::k_split_product<1, false>, &lc)
                                    : cudaOccupancyMaxActiveClusters(&got[s], split::k_split_product<3, false>, &lc);
      if (e == cudaSuccess) continue;
      cudaGetLastError();
      got[s] = 0;
      all = false;
    }
    if (all) known[key] = got;
  }
  for (int s = 0; s <= 8; ++s) resident[s] = got[s];
}

// A step of the learners p0 .. p0 + n - 1.
template <bool QUANT>
cudaError_t step_impl(mavg_ctx* c, int64_t round, int step, int p0, int n) {
  constexpr int NP = kPlanes<QUANT>;
  const mavg_config& cfg = c->cfg;
  const int B = cfg.B, L = cfg.n_layers;
  const SimtState* st = (const SimtState*)c->simt;
  const int G = st->group;
  const SimtBuffers& sb = st->buf;
  auto plane_of = [&](int d) { return (int64_t)G * B * pitch_of(d); };
  const int cur = step & 1;
  GatherArgs ga{};
  ga.x = cfg.x; ga.x_bf16 = cfg.x_dtype == MAVG_X_BF16;
  ga.y = cfg.y; ga.seed = cfg.seed; ga.round = round;
  ga.round_ptr = c->capturing ? (const int64_t*)(ws_ptr(c, c->ws.status) + 64) : nullptr;
  ga.step = step; ga.P = cfg.P; ga.p0 = p0; ga.n = n; ga.B = B; ga.d = cfg.dims[0]; ga.S = cfg.n_samples;
  ga.out = sb.xg[cur]; ga.plane = plane_of(cfg.dims[0]); ga.labels = sb.labels[cur];
  GatherArgs next = ga;
  next.step = step + 1; next.out = sb.xg[cur ^ 1]; next.labels = sb.labels[cur ^ 1];
  const int gather_rows = step < cfg.K ? n * B : 0;
  cudaError_t e;
  // the weights before this step
  const int64_t rs = c->buf.replica_stride;
  float* rep = c->buf.replicas + p0 * rs;
  const float* win = starts_from_global(c) ? c->buf.global_w : rep;
  const int64_t ws = starts_from_global(c) ? 0 : rs;
  const bool shared_w = starts_from_global(c);
  auto w_matrix = [&](int l) { return (int64_t)cfg.dims[l] * pitch_of(cfg.dims[l - 1]); };
  if (step == 1) {
    split::SplitWeights w{};
    w.L = plane_layers(&cfg);
    w.copies = shared_w ? 1 : n;
    w.src_batch = ws;
    for (int l = 1; l <= w.L; ++l) {
      w.src[l - 1] = win + c->layers[l - 1].w_off;
      w.dst[l - 1] = sb.w[l] + (shared_w ? G * w_matrix(l) : 0);
      w.dst_batch[l - 1] = w_matrix(l);
      w.dst_plane[l - 1] = (G + 1) * w_matrix(l);
      w.in[l - 1] = cfg.dims[l - 1];
      w.first[l] = w.first[l - 1] + cfg.dims[l];
    }
    const int64_t blocks = (int64_t)n * B + ((int64_t)w.copies * w.first[w.L] + 7) / 8;
    if ((e = launch(c, MAVG_K_BATCH, k_simt_begin<QUANT>, dim3((unsigned)blocks), 256, 1, 0, ga, w)) != cudaSuccess) return e;
  }
  MomArgs mom = mom_args(c, c->replicas_equal_global);
  if (mom.u) mom.u += p0 * mom.u_stride;
  auto a_in = [&](int l) { return l == 1 ? sb.xg[cur] : sb.a[l - 1]; };
  const MlpLayer& top = c->layers[L - 1];
  const bool tail = product_layers(&cfg) < L;
  for (int l = 1; l <= (tail ? L - 1 : L); ++l) {
    const MlpLayer& ly = c->layers[l - 1];
    split::ProductArgs g{};
    g.M = ly.out; g.K = ly.in;
    g.bias = win + ly.b_off; g.bias_batch = ws;
    g.pitch = pitch_of(ly.out);
    g.hidden = l < L;
    if (l < L) g.out = sb.a[l];
    else g.out_f = sb.logits;
    if ((e = launch_product<QUANT, false>(c, MAVG_K_FWD, n, st->w[l], shared_w, l == 1 ? st->x[cur] : st->a[l - 1], g)) != cudaSuccess) return e;
  }
  if (tail) {
    TailArgs t{};
    t.a = a_in(L); t.a_plane = plane_of(top.in);
    t.w = win + top.w_off; t.b = win + top.b_off; t.w_batch = ws;
    t.labels = sb.labels[cur];
    t.P = n; t.B = B; t.in = top.in; t.C = top.out; t.row_blocks = (B + kTailRows - 1) / kTailRows;
    t.row_loss = sb.row_loss; t.dz = sb.dz_f[L];
    t.dz_pl = sb.dz[L]; t.dz_plane = plane_of(top.out);
    if (L >= 2) {
      t.dzp = sb.dz_f[L - 1];
      t.dzp_pl = sb.dz[L - 1];
      t.dzp_plane = plane_of(top.in);
    }
    // few classes on very wide rows: their padding to 16 would not fit
    t.mma = QUANT && tail_smem(t.in, t.C, true) <= kTailSmem;
    t.w16 = sb.w[L] + (shared_w ? G * w_matrix(L) : 0);
    t.w16_batch = shared_w ? 0 : w_matrix(L);
    if ((e = launch(c, MAVG_K_LOSS, k_simt_tail<QUANT>, dim3((unsigned)(n * t.row_blocks + gather_rows)),
                    kTailThreads, 1, tail_smem(t.in, t.C, t.mma), t, next)) != cudaSuccess)
      return e;
  } else {
    if ((e = launch(c, MAVG_K_LOSS, k_simt_loss<QUANT>, dim3((unsigned)(n + gather_rows)), 1024, 1, 0,
                    (const float*)sb.logits, (const int32_t*)sb.labels[cur], n, B, top.out, sb.row_loss,
                    sb.dz_f[L], sb.dz[L], plane_of(top.out), next)) != cudaSuccess)
      return e;
  }
  for (int l = tail ? L - 1 : L; l >= 2; --l) {
    const MlpLayer& ly = c->layers[l - 1];
    split::ProductArgs g{};
    g.M = ly.in; g.K = ly.out;
    g.out = sb.dz[l - 1]; g.out_f = sb.dz_f[l - 1];
    g.act = sb.a[l - 1]; g.pitch = pitch_of(ly.in);
    if ((e = launch_product<QUANT, true>(c, MAVG_K_DGRAD, n, st->w_mn[l], shared_w, st->dz[l], g)) != cudaSuccess) return e;
  }
  split::WgradArgs w{};
  w.L = L; w.P = G; w.B = B;
  w.write_planes = step < cfg.K;
  // Tiles of 128 x 64 where wider ones would leave SMs without any (us a round, 128 / 64 wide: 322-266-305-5, P = 2,
  // K = 3, B = 37 160 / 151, 357-761-217-96, P = 1, K = 4, B = 149 261 / 250; beyond the line 437-425-42, P = 6, K = 4,
  // B = 36 103 / 110, 3072-512-512-10, P = 4, K = 4, B = 100 382 / 394: a narrow tile takes in half as much again).
  int64_t wide = 0;
  for (const MlpLayer& ly : c->layers) wide += (int64_t)((ly.in + 127) / 128) * ((ly.out + 127) / 128) * cfg.P;
  w.bn = wide <= c->sm_count ? 64 : 128;
  for (int l = 1; l <= L; ++l) {
    const MlpLayer& ly = c->layers[l - 1];
    split::WgradLayer& g = w.layer[l - 1];
    w.a[l - 1] = l == 1 ? st->x_mn[cur] : st->a_mn[l - 1];
    w.dz[l - 1] = st->dz_mn[l];
    g.in = ly.in; g.out = ly.out;
    g.i_tiles = (ly.in + split::kTile - 1) / split::kTile;
    g.o_tiles = (ly.out + w.bn - 1) / w.bn;
    g.first = w.tiles;
    g.w_off = ly.w_off; g.b_off = ly.b_off;
    g.pairs = ly.in % 2 == 0 && ly.w_off % 2 == 0;
    g.dz = sb.dz_f[l];
    if (l <= plane_layers(&cfg)) {
      g.w16 = sb.w[l];
      g.w16_batch = w_matrix(l);
      g.w16_plane = (G + 1) * w_matrix(l);
    }
    w.tiles += g.i_tiles * g.o_tiles * n;
  }
  w.w_in = win; w.w_in_batch = ws;
  w.rep = rep; w.rep_stride = rs;
  w.mom = mom;
  w.gamma = cfg.local_lr;
  w.row_loss = sb.row_loss;
  w.loss_out = (float*)ws_ptr(c, c->ws.losses) + (size_t)p0 * cfg.K + (step - 1);
  w.loss_stride = cfg.K;
  w.status = (int*)ws_ptr(c, c->ws.status);
  const split::LaunchShape shape = split::wgrad_shape(NP);
  w.stages = shape.stages;
  return launch(c, MAVG_K_WGRAD_SGD, wgrad_kernel<QUANT>(B, mom.u != nullptr), dim3((unsigned)std::min(w.tiles, c->sm_count)),
                split::wgrad_threads(split::wgrad_chains(NP, B)), 1, shape.smem, w);
}

}  // namespace

size_t simt_workspace_bytes(const mavg_config* cfg, size_t base, size_t* act_off, size_t* least) {
  *act_off = base;
  SimtBuffers sb;
  *least = base + carve(cfg, 1, nullptr, &sb);
  // (models whose steps are one launch use none of it unless that launch is refused)
  return small_always(cfg) ? *least : base + carve(cfg, cfg->P, nullptr, &sb);
}

mavg_status simt_setup(mavg_ctx* c) {
  const mavg_config& cfg = c->cfg;
  const int L = cfg.n_layers, B = cfg.B, np = cfg.gemm_bf16 ? kPlanes<true> : kPlanes<false>;
  const EncodeTiledFn encode = tensor_map_encoder(&c->err);
  if (!encode) return MAVG_ERR_UNSUPPORTED;
  SimtState* st = new SimtState();
  c->simt = st;
  // The planes of the learners' weights are 1.5 times the replica array with fp32 operands: where the scratch has room for
  // fewer learners' they take their steps in groups, one after the other.
  const size_t room = c->buf.workspace_bytes - c->ws.act;
  int P = cfg.P;
  if (carve(&cfg, P, nullptr, &st->buf) > room) {
    int fits = 1;
    while (P - fits > 1) {
      const int half = fits + (P - fits) / 2;
      (carve(&cfg, half, nullptr, &st->buf) > room ? P : fits) = half;
    }
    P = (cfg.P + (cfg.P + fits - 1) / fits - 1) / ((cfg.P + fits - 1) / fits);   // of as many groups, the most even
  }
  st->group = P;
  carve(&cfg, P, ws_ptr(c, c->ws.act), &st->buf);
  st->n_tiles = (B + split::kMaxN - 1) / split::kMaxN;
  st->N = ((B + st->n_tiles - 1) / st->n_tiles + 15) / 16 * 16;
  bool ok = true;
  auto map = [&](CUtensorMap* k, CUtensorMap* mn, __nv_bfloat16* p, int d, int rows, int matrices, int box_rows) {
    const int pitch = pitch_of(d);
    for (int i = 0; i < 2; ++i)
      ok = ok && encode_tiled(encode, i ? mn : k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p, d, rows, np * matrices, pitch,
                              (int64_t)rows * pitch, split::kSlab, i ? split::kSlab : box_rows, CU_TENSOR_MAP_SWIZZLE_128B, &c->err);
  };
  for (int i = 0; i < 2; ++i) map(&st->x[i], &st->x_mn[i], st->buf.xg[i], cfg.dims[0], B, P, st->N);
  for (int l = 1; l <= L; ++l) {
    if (l < L) map(&st->a[l], &st->a_mn[l], st->buf.a[l], cfg.dims[l], B, P, st->N);
    map(&st->dz[l], &st->dz_mn[l], st->buf.dz[l], cfg.dims[l], B, P, st->N);
    if (l <= product_layers(&cfg)) map(&st->w[l], &st->w_mn[l], st->buf.w[l], cfg.dims[l - 1], cfg.dims[l], P + 1, split::kTile);
  }
  if (!ok) return MAVG_ERR_UNSUPPORTED;
  cudaError_t e = cfg.gemm_bf16 ? set_attributes<true>(c) : set_attributes<false>(c);
  // columns beyond the rows of W_L's plane, which mma_tail reads and nobody writes
  if (e == cudaSuccess && cfg.gemm_bf16 && cfg.dims[L - 1] % 8)
    e = cudaMemsetAsync(st->buf.w[L], 0, (size_t)(P + 1) * cfg.dims[L] * pitch_of(cfg.dims[L - 1]) * 2, c->stream);
  if (e == cudaSuccess) resident_clusters(c->device, np, st->N, st->resident);
  if (e == cudaSuccess) return MAVG_OK;
  c->err = std::string("kernel attributes: ") + cudaGetErrorString(e);
  return MAVG_ERR_CUDA;
}

void simt_teardown(mavg_ctx* c) {
  delete (SimtState*)c->simt;
  c->simt = nullptr;
}

cudaError_t simt_local_steps(mavg_ctx* c, int64_t round) {
  const bool from_broadcast = c->replicas_equal_global;
  const int group = ((const SimtState*)c->simt)->group;
  cudaError_t e = cudaSuccess;
  for (int p0 = 0; p0 < c->cfg.P && e == cudaSuccess; p0 += group) {
    c->replicas_equal_global = from_broadcast;
    const int n = std::min(group, c->cfg.P - p0);
    for (int k = 1; k <= c->cfg.K && e == cudaSuccess; ++k) {
      e = c->cfg.gemm_bf16 ? step_impl<true>(c, round, k, p0, n) : step_impl<false>(c, round, k, p0, n);
      c->replicas_equal_global = false;
    }
  }
  return e;
}

}  // namespace mavg
