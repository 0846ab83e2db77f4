// Factored local steps: the K steps of a round without the learners' hidden weights (see factored.cuh).
// Kernels of this file, in the order of a call:
//   k_fac_gather    the minibatches of all steps (the index stream depends on no weights)
//   k_fac_product   X W~_1^T of all steps (fp32), then per step the forward and data-gradient products:
//                   128 features x the batches of a few learners per block; the contraction runs over
//                   w~ (weights read once for those learners) and then, learner by learner, over the
//                   rows of the earlier steps with the Gram rows as the other operand
//   k_fac_gram      -gamma A A(i)^T and -gamma dZ dZ(i)^T of a step against all earlier ones, as bf16
//   k_fac_apply     W_l = w~_l - gamma dZ_l^T A_{l-1} over all steps' rows, every learner and hidden layer
//   k_fac_last      the last layer (at most 32 classes), which keeps its own weights and steps
//
// and the rebuilt local steps of rebuild.cuh, which share the gather; their products are the plain form's launches.
//
// All are launched with programmatic stream serialisation.
#include <cuda.h>

#include <algorithm>

#include "gemm_unit.cuh"
#include "mlp.cuh"
#include "rebuild.cuh"
#include "tc_state.cuh"

namespace mavg {
namespace {

using namespace tc;
using namespace gemm;

constexpr int kFacThreads = 320;   // warp 0: TMA producer, warp 1: MMA issuer, warps 2-9: epilogue
enum { PROD_FWD = 0, PROD_DGRAD = 1, PROD_RAW = 2, PROD_DGRAD_STEP = 3, PROD_FWD_RUNS = 4 };
constexpr size_t kGramBarBytes = 2 * sizeof(uint64_t);   // static shared memory of a product that forms its Gram rows, beside GemmShared

// Place in a ring of stages and the phase of its barriers, without a division per slab: the one thread that
// issues the copies and the one that issues the MMAs are on every slab's way.
struct Ring {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int stages) {
    if (++s == stages) { s = 0; ph ^= 1; }
  }
};

// The MMAs of one slab of 64 contraction elements; the steps count 16-byte units per 16 elements.
__device__ __forceinline__ void slab_mma(uint32_t d, uint64_t adesc, uint32_t a_step, uint64_t bdesc, uint32_t b_step,
                                         uint32_t idesc, bool add) {
  umma_bf16(d, adesc, bdesc, idesc, (uint32_t)add);
#pragma unroll
  for (int k = 1; k < kBK / 16; ++k) umma_bf16(d, adesc + a_step * k, bdesc + b_step * k, idesc, 1u);
}
// A last slab with fewer than 64: nk groups of 16.
__device__ __forceinline__ void part_mma(uint32_t d, uint64_t adesc, uint32_t a_step, uint64_t bdesc, uint32_t b_step,
                                         uint32_t idesc, bool add, int nk) {
  for (int k = 0; k < nk; ++k) umma_bf16(d, adesc + a_step * k, bdesc + b_step * k, idesc, (uint32_t)(add || k > 0));
}
constexpr uint32_t kStepK = 2, kStepMn = (16 * 128) >> 4;

// ------------------------------------------------------------------------------------- gather

template <typename TIN>
__device__ __forceinline__ uint4 load8_bf16(const TIN* src);
template <>
__device__ __forceinline__ uint4 load8_bf16<__nv_bfloat16>(const __nv_bfloat16* src) {
  return *reinterpret_cast<const uint4*>(src);
}
template <>
__device__ __forceinline__ uint4 load8_bf16<float>(const float* src) {
  const float4 a = reinterpret_cast<const float4*>(src)[0], b = reinterpret_cast<const float4*>(src)[1];
  __nv_bfloat162 h[4] = {__floats2bfloat162_rn(a.x, a.y), __floats2bfloat162_rn(a.z, a.w),
                         __floats2bfloat162_rn(b.x, b.y), __floats2bfloat162_rn(b.z, b.w)};
  return *reinterpret_cast<uint4*>(h);
}

// What the bf16 copy of w~'s hidden layers leaves over, as bf16: the forward products and the last layer read
// both parts (16 bits of the weights).  A rounding of the weights is the same for every sample, step and learner
// here, where the plain form rounds each learner's own weights at every step, so it does not average out: with
// one bf16 part v or the mean loss can be further from 64 bits than the plain form's.  Root mean square of
// v's relative error and of the mean loss's error over 12 seeds (both forms' roundings restated in torch), plain / one
// part / both parts in every hidden layer:
//   1000-312-10, P = 40, K = 4, B = 80:            v 3.6e-3 / 3.9e-3 / 0.4e-3, loss 1.1e-4 / 0.7e-4 / 0.4e-4
//   the same, inputs in [0, 1]:                    v 1.8e-3 / 2.0e-3 / 0.6e-3, loss 2.9e-4 / 3.3e-4 / 0.1e-4
//   520-200-136-12, P = 20, K = 9, B = 48, [0, 1]: v 3.0e-3 / 3.2e-3 / 2.1e-3, loss 2.1e-4 / 2.4e-4 / 0.3e-4
//   3072-512-512-10, P = 8, K = 8, B = 128:        v 7.9e-3 / 7.7e-3 / 4.7e-3, loss 2.5e-4 / 0.7e-4 / 0.5e-4
//   2048-1024-1024-1024-10, P = 8, K = 8, B = 128, inputs >= 0: v 6.3e-3 / 6.2e-3 / 4.5e-3, loss 1.6e-4 / 1.4e-4 / 0.3e-4
// (the last with low parts in the first and last hidden layer only: loss 1.6e-4).  Low parts in the data gradients
// and Gram rows of two parts change none of these by more than a tenth.
struct LowArgs {
  const float* w[MAVG_MAX_LAYERS - 1];            // the hidden layers in w~
  __nv_bfloat16* dst[MAVG_MAX_LAYERS - 1];
  int64_t total[MAVG_MAX_LAYERS - 1];             // weights, a multiple of 8
  int layers, blocks;                             // blocks of the launch that do this
};
__device__ __forceinline__ uint32_t low_pair(float a, float b) {
  const __nv_bfloat162 hi = __floats2bfloat162_rn(a, b);
  const __nv_bfloat162 lo = __floats2bfloat162_rn(a - __low2float(hi), b - __high2float(hi));
  return *reinterpret_cast<const uint32_t*>(&lo);
}
__device__ __forceinline__ uint4 low8(const float* src) {
  const float4 a = reinterpret_cast<const float4*>(src)[0], b = reinterpret_cast<const float4*>(src)[1];
  return make_uint4(low_pair(a.x, a.y), low_pair(a.z, a.w), low_pair(b.x, b.y), low_pair(b.z, b.w));
}

// A sum and what the low parts add to it.  An infinite operand (a diverging model's weight or activation) has an
// infinite product with the high part and with the low one, of either sign: the former alone is the result, as in
// the plain form.  Added up they would be NaN, which ReLU makes 0.
__device__ __forceinline__ float with_low(float high, float low) { return fabsf(high) <= 3.402823466e38f ? high + low : high; }

// A warp per row (learner p, step k, slot s): its sample's index, its label and its d inputs as bf16, learner by learner
// or (step_major) step by step.  The first la.blocks blocks write the low parts of w~ instead.
template <typename TIN>
__global__ void __launch_bounds__(256)
k_fac_gather(const TIN* __restrict__ x, const int32_t* __restrict__ y, uint64_t seed, int64_t round,
             const int64_t* __restrict__ round_ptr, int P, int K, int B, int64_t kb, int64_t S, int d,
             int32_t* __restrict__ labels, __nv_bfloat16* __restrict__ out, int step_major, const __grid_constant__ LowArgs la) {
  if ((int)blockIdx.x < la.blocks) {
    for (int l = 0; l < la.layers; ++l)
      for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < la.total[l] >> 3; t += (int64_t)la.blocks * blockDim.x)
        reinterpret_cast<uint4*>(la.dst[l])[t] = low8(la.w[l] + 8 * t);
    return;
  }
  const int64_t row = (int64_t)(blockIdx.x - la.blocks) * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= (int64_t)P * K * B) return;
  if (round_ptr) round = *round_ptr;
  const int p = (int)(row / ((int64_t)K * B)), r = (int)(row - (int64_t)p * K * B), k = r / B, s = r - k * B;
  const int32_t i = sample_index(seed, round, p, k + 1, s, P, S);
  if (lane == 0) labels[((size_t)k * P + p) * B + s] = y[i];
  const TIN* src = x + (size_t)i * d;
  uint4* dst = reinterpret_cast<uint4*>(out + (step_major ? ((size_t)k * P + p) * B + s : (size_t)p * kb + r) * d);
  const int n8 = d >> 3;
  for (int c0 = lane; c0 < n8; c0 += 4 * 32) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 32 * u < n8) v[u] = load8_bf16<TIN>(src + (size_t)(c0 + 32 * u) * 8);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c0 + 32 * u < n8) dst[c0 + 32 * u] = v[u];
  }
}

// ------------------------------------------------------------------------------------ products

struct ProdArgs {
  int M;                    // features of the result
  int m_tiles;
  int P;
  int64_t kb;               // rows per learner of the row arrays
  int row0;                 // first row of the batch inside a learner's rows
  int nl;                   // learners per block
  int cols;                 // columns per learner and block (RAW: the rows of a tile); B unless nl is 1
  int c_tiles;              // column tiles: B / cols (RAW: tiles of a learner's rows)
  int row_end;              // RAW: rows per learner
  int nkb;                  // slabs of the product with w~ (0: left out)
  int w_batched;            // the weights are each learner's own (one learner per block)
  // PROD_FWD_RUNS: sums of `run` groups of 16 contraction elements each, `runs` of them, added in ascending order; the first
  // whole_rows pairs of learner and row tile take one sum
  int run, runs, whole_rows;
  int hist;                 // rows of the earlier steps (0: left out)
  int s_row0;               // row of the batch inside a learner's Gram rows
  int stages;
  uint32_t tmem_cols;
  uint32_t low_col;         // LOW: first column of the low parts' sums
  const float* zbase;       // added to the result: fp32 [kb, M] per learner (null: nothing)
  float* raw;               // RAW: the result, laid out like zbase
  int64_t z_stride;         // floats from learner to learner of either
  __nv_bfloat16* out;       // relu(Z + b) or dZ of the layer below: [P, kb, M]
  const __nv_bfloat16* act; // dgrad: activations [P, kb, M] whose sign gates dZ
  const float* bias_in;     // bias read at bias_in[p * bias_in_stride + bias_off + m]
  int64_t bias_in_stride;
  float* bias_rep;          // dgrad: stepped bias written at bias_rep[p * rep_stride + bias_off + m]
  int64_t rep_stride, bias_off;
  // GRAM: contraction slabs of the Gram product, its rows [cols of the batch, history] per learner
  int gram_nkb;
  __nv_bfloat16* gram_out;
  int64_t gram_stride, gram_ld;
  float gamma;
  MomArgs mom;              // of the stepped bias (PROD_DGRAD_STEP)
  int* status;
};

// One batch operand, or Gram rows for each of `grams` history tiles.
__host__ __device__ __forceinline__ int product_stage_bytes(int tiles, int grams, int nl, int cols) {
  return tiles * kATileBytes + (nl > grams ? nl : grams) * cols * kBK * 2;
}

__device__ __forceinline__ void load16(uint32_t taddr, bool any, float (&z)[16]) {
  if (any) {
    uint32_t r[16];
    tmem_ld_16cols(taddr, r);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 16; ++j) z[j] = __uint_as_float(r[j]);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) z[j] = 0.f;
  }
}

// Bound by the operands' way into the SM and the tensor pipe and, late in a round, by the history in HBM: P = 32,
// B = 64, layers of 2048: data gradient 24 us in the first step, 45 us in the sixteenth (another 126 MB of history
// and 4 MB of Gram rows); forward with both parts of w~ 30 us (1140 TFLOP/s) and 50.  Per-slab divisions in the two issuing threads cost 2 to 6 us of that.
// grid (column tiles x m_tiles, learner groups).  dgrad with several column tiles: these are a cluster,
// whose first block adds their bias gradients in rank order.
// TILES: 16 KB tiles of the MMA's row operand per stage.  LOW (two tiles): the product with w~ reads its low
// parts as well, into columns of their own.
// GRAM: the Gram rows are formed here too, instead of by a launch of k_fac_gram before.  The blocks of a
// learner are a cluster; those of a column tile share its Gram tiles out among themselves (128 history
// rows each, row tile m_tile, m_tile + m_tiles, ...), write them to global memory and tell each other, while
// the product with w~ runs; the tiles come back through the L2 as an operand.  A launch less on the chain of
// a step for models whose launches are short.
template <int EPI, int TILES, bool LOW, bool GRAM>
__global__ void __launch_bounds__(kFacThreads, 2)
k_fac_product(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_lo,
              const __grid_constant__ CUtensorMap tm_in, const __grid_constant__ CUtensorMap tm_gram,
              const __grid_constant__ CUtensorMap tm_hist, const __grid_constant__ CUtensorMap tm_s,
              const ProdArgs g) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) GemmShared sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = g.stages;
  const int N = g.nl * g.cols;
  // A stage: the w~ tile (LOW: and its low part), then the batch operand; or TILES history slabs in the
  // tiles' places, with their Gram rows where the batch operand is.
  static_assert(!LOW || TILES == 2, "");
  constexpr bool kStep = EPI == PROD_DGRAD_STEP, kMn = EPI == PROD_DGRAD || kStep;   // kMn: the weights are read MN-major
  constexpr bool kRuns = EPI == PROD_FWD_RUNS, kFwd = EPI == PROD_FWD || kRuns;
  constexpr int kBOff = TILES * kATileBytes;
  const int stage_bytes = product_stage_bytes(TILES, EPI == PROD_RAW ? 1 : TILES, g.nl, g.cols), s_bytes = g.cols * kBK * 2;
  __shared__ __align__(8) uint64_t gram_bar, rows_bar;     // GRAM: Gram sums complete; Gram rows in global memory

  if (threadIdx.x == 0) {
    if (LOW) tma_prefetch_desc(&tm_lo);
    if (GRAM) {
      tma_prefetch_desc(&tm_gram);
      mbar_init(&gram_bar, 1);
      mbar_init(&rows_bar, 8u * g.m_tiles);        // the epilogue warps of the column tile's blocks
    }
    tma_prefetch_desc(&tm_w);
    tma_prefetch_desc(&tm_in);
    tma_prefetch_desc(&tm_hist);
    tma_prefetch_desc(&tm_s);
    gemm_init_barriers(sh, stages);
    sh.abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_slot, g.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  if (GRAM) cluster_sync_all();                    // every block's barriers exist before anyone arrives on them
  const uint32_t tmem_base = sh.tmem_slot;
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();

  const int c_tile = (int)blockIdx.x % g.c_tiles, m_tile = (int)blockIdx.x / g.c_tiles;
  const int m0 = m_tile * kBM, p0 = (int)blockIdx.y * g.nl;
  const int nl = min(g.nl, g.P - p0);
  const int r0 = g.row0 + c_tile * g.cols;
  const int s_row = g.s_row0 + c_tile * g.cols;
  const int nslab = (g.hist + kBK - 1) / kBK;
  volatile int* abortp = &sh.abort_flag;
  const bool any = g.nkb > 0 || g.hist > 0;
  const int w_of = g.w_batched ? p0 : 0;
  const int runs = kRuns && p0 * g.m_tiles + m_tile >= g.whole_rows ? g.runs : 1;
  const int gram_step = kBM * g.m_tiles;           // from one of this block's Gram tiles to the next, in rows

  if (warp == 0) {
    if (lane == 0) {
      Ring ring;
      int issued = 0;
      bool ok = true;
      if (GRAM)
        for (int s0 = m0; s0 < g.hist && ok; s0 += gram_step)
          for (int i = 0; i < g.gram_nkb; ++i, ++issued, ring.next(stages)) {
            uint64_t* full = &sh.full_bar[ring.s];
            if (!(ok = mbar_wait(&sh.empty_bar[ring.s], ring.ph ^ 1, abortp, g.status, ERR_PRODUCER))) break;
            uint8_t* sa = smem + (size_t)ring.s * stage_bytes;
            mbar_arrive_expect_tx(full, (uint32_t)(kATileBytes + s_bytes));
            tma_load_3d(sa, &tm_gram, full, i * kBK, s0, p0);
            tma_load_3d(sa + kBOff, &tm_in, full, i * kBK, r0, p0);
          }
      const uint32_t base_bytes = (uint32_t)((LOW ? 2 : 1) * kATileBytes + N * kBK * 2);
      for (int i = 0; i < g.nkb && ok; ++i, ++issued, ring.next(stages)) {
        uint64_t* full = &sh.full_bar[ring.s];
        if (!(ok = mbar_wait(&sh.empty_bar[ring.s], ring.ph ^ 1, abortp, g.status, ERR_PRODUCER))) break;
        uint8_t* sa = smem + (size_t)ring.s * stage_bytes;
        mbar_arrive_expect_tx(full, base_bytes);
        if (kMn) {
          tma_load_3d(sa, &tm_w, full, m0, i * kBK, w_of);
          tma_load_3d(sa + kATileBytes / 2, &tm_w, full, m0 + 64, i * kBK, w_of);
        } else {
          tma_load_3d(sa, &tm_w, full, i * kBK, m0, w_of);
        }
        if (LOW) tma_load_3d(sa + kATileBytes, &tm_lo, full, i * kBK, m0, 0);
        tma_load_3d(sa + kBOff, &tm_in, full, i * kBK, r0, p0);
      }
      if (GRAM && ok) {
        ok = mbar_wait_cluster(&rows_bar, 0, abortp, g.status, ERR_PRODUCER);
        fence_proxy_async_all();                   // the rows were written by ordinary stores
      }
      for (int q = 0; q < nl && ok; ++q)
        for (int i = 0; i < nslab; i += TILES, ++issued, ring.next(stages)) {
          uint64_t* full = &sh.full_bar[ring.s];
          if (!(ok = mbar_wait(&sh.empty_bar[ring.s], ring.ph ^ 1, abortp, g.status, ERR_PRODUCER))) break;
          uint8_t* sa = smem + (size_t)ring.s * stage_bytes;
          const int n = min(TILES, nslab - i);
          mbar_arrive_expect_tx(full, (uint32_t)(n * (kATileBytes + s_bytes)));
          for (int h = 0; h < n; ++h) {
            tma_load_3d(sa + h * kATileBytes, &tm_hist, full, m0, (i + h) * kBK, p0 + q);
            tma_load_3d(sa + h * kATileBytes + kATileBytes / 2, &tm_hist, full, m0 + 64, (i + h) * kBK, p0 + q);
            tma_load_3d(sa + kBOff + h * s_bytes, &tm_s, full, (i + h) * kBK, s_row, p0 + q);
          }
        }
      if (*abortp) drain_copies(sh.full_bar, issued, stages, g.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      Ring ring;
      bool ok = true;
      const uint32_t base = smem_u32(smem);
      const uint32_t idesc_base = idesc_bf16_f32(kBM, N, kMn ? 1 : 0);
      const uint64_t a_base = kMn ? smem_desc_mn_sw128(base) : smem_desc_k_sw128(base);
      const uint64_t b_base = smem_desc_k_sw128(base + kBOff);
      constexpr uint32_t kStepA = kMn ? kStepMn : kStepK;
      const uint32_t unit = (uint32_t)stage_bytes >> 4;
      if (GRAM) {
        const uint32_t idesc_gram = idesc_bf16_f32(kBM, g.cols);
        const uint64_t a_gram = smem_desc_k_sw128(base);
        uint32_t d = tmem_base + (uint32_t)N;
        for (int s0 = m0; s0 < g.hist && ok; s0 += gram_step, d += (uint32_t)g.cols)
          for (int i = 0; i < g.gram_nkb; ++i, ring.next(stages)) {
            if (!(ok = mbar_wait(&sh.full_bar[ring.s], ring.ph, abortp, g.status, ERR_MMA))) break;
            tc_fence_after_sync();
            const uint32_t off = (uint32_t)ring.s * unit;
            slab_mma(d, a_gram + off, kStepK, b_base + off, kStepK, idesc_gram, i > 0);
            umma_commit(&sh.empty_bar[ring.s]);
          }
        if (ok && m0 < g.hist) umma_commit(&gram_bar);
      }
      for (int i = 0; i < g.nkb && ok; ++i, ring.next(stages)) {
        if (!(ok = mbar_wait(&sh.full_bar[ring.s], ring.ph, abortp, g.status, ERR_MMA))) break;
        tc_fence_after_sync();
        const uint32_t off = (uint32_t)ring.s * unit;
        if (kRuns && runs > 1) {
          for (int k = 0; k < kBK / 16; ++k) {       // (what lies behind the last run's elements is zero)
            const int at = i * (kBK / 16) + k, r = min(at / g.run, runs - 1);
            umma_bf16(tmem_base + (uint32_t)(r * N), a_base + off + kStepA * k, b_base + off + kStepK * k, idesc_base, (uint32_t)(at > r * g.run));
          }
        } else {
          slab_mma(tmem_base, a_base + off, kStepA, b_base + off, kStepK, idesc_base, i > 0);
        }
        if (LOW) slab_mma(tmem_base + g.low_col, a_base + off + (kATileBytes >> 4), kStepA, b_base + off, kStepK, idesc_base, i > 0);
        umma_commit(&sh.empty_bar[ring.s]);
      }
      const uint32_t idesc_hist = idesc_bf16_f32(kBM, g.cols, 1);
      const uint64_t a_hist = smem_desc_mn_sw128(base);
      for (int q = 0; q < nl && ok; ++q)
        for (int i = 0; i < nslab; i += TILES, ring.next(stages)) {
          if (!(ok = mbar_wait(&sh.full_bar[ring.s], ring.ph, abortp, g.status, ERR_MMA))) break;
          tc_fence_after_sync();
          const uint32_t d = tmem_base + (uint32_t)(q * g.cols);
          for (int h = 0; h < min(TILES, nslab - i); ++h) {
            const uint32_t off = (uint32_t)ring.s * unit;
            const uint64_t ad = a_hist + off + (uint32_t)(h * (kATileBytes >> 4)), bd = b_base + off + (uint32_t)(h * (s_bytes >> 4));
            const bool add = g.nkb > 0 || i + h > 0;
            // the last slab ends with the history (a multiple of 16 rows): what lies behind it in either
            // operand is of this or a later step and must not enter, not even times zero
            const int rest = g.hist - (i + h) * kBK;
            if (rest >= kBK) slab_mma(d, ad, kStepMn, bd, kStepK, idesc_hist, add);
            else part_mma(d, ad, kStepMn, bd, kStepK, idesc_hist, add, rest / 16);
          }
          umma_commit(&sh.empty_bar[ring.s]);
        }
      if (ok && any) umma_commit(&sh.acc_bar);
    }
    __syncwarp();
  } else {
    // warp (q, half): TMEM lanes [32q, 32q + 32), one feature per lane, and every second group of 16 columns
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    const int row = q4 * 32 + lane, m = m0 + row;
    const bool m_ok = m < g.M;
    if (GRAM) {
      if (m0 < g.hist && mbar_wait_warp(&gram_bar, 0, abortp, g.status, ERR_EPILOGUE)) {
        tc_fence_after_sync();
        uint32_t d = tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)N;
        for (int s0 = m0; s0 < g.hist; s0 += gram_step, d += (uint32_t)g.cols) {
          const int s = s0 + row;
#pragma unroll 1
          for (int c0 = half * 16; c0 < g.cols; c0 += 32) {
            float z[16];
            load16(d + (uint32_t)c0, true, z);
            if (s >= g.hist) continue;
            __nv_bfloat16* dst = g.gram_out + (size_t)p0 * g.gram_stride + (size_t)(s_row + c0) * g.gram_ld + s;
#pragma unroll
            for (int j = 0; j < 16; ++j) dst[(size_t)j * g.gram_ld] = __float2bfloat16_rn(-g.gamma * z[j]);
          }
        }
      }
      __threadfence();
      fence_proxy_async_all();
      __syncwarp();
      if (lane < g.m_tiles) mbar_arrive_cluster(mapa_u32(smem_u32(&rows_bar), (uint32_t)(lane * g.c_tiles + c_tile)));
      __syncwarp();
    }
    float* colsum = reinterpret_cast<float*>(smem + (size_t)stages * stage_bytes);   // [2][nl][128]
    if (EPI == PROD_DGRAD)
      for (int q = 0; q < nl; ++q) colsum[(half * nl + q) * kBM + row] = 0.f;
    // What a group of columns needs besides the accumulator (the fp32 base of layer 1, the activations that
    // gate dZ) is in flight while the group before it, or the main loop, is still at work.
    const int end = EPI == PROD_RAW ? min(g.cols, g.row_end - r0) : nl * g.cols;
    const bool add_base = kFwd && g.zbase != nullptr;
    float zb[16], bias_next = 0.f;
    __nv_bfloat16 act[16];
    auto locate = [&](int c0, size_t& at, size_t& z_at, int& q) {
      q = EPI == PROD_RAW ? 0 : c0 / g.cols;
      const int r = r0 + c0 - q * g.cols;
      at = ((size_t)(p0 + q) * g.kb + r) * g.M + m;                    // element of column c0
      z_at = (size_t)(p0 + q) * g.z_stride + (size_t)r * g.M + m;
    };
    auto fetch = [&](int c0) {
      size_t at, z_at;
      int q;
      if (!m_ok || c0 >= end) return;
      locate(c0, at, z_at, q);
      if (kFwd) bias_next = g.bias_in[(size_t)(p0 + q) * g.bias_in_stride + g.bias_off + m];
      if (add_base) {
#pragma unroll
        for (int j = 0; j < 16; ++j) zb[j] = __ldg(g.zbase + z_at + (size_t)j * g.M);
      }
      if (EPI == PROD_DGRAD) {
#pragma unroll
        for (int j = 0; j < 16; ++j) act[j] = g.act[at + (size_t)j * g.M];
      }
    };
#pragma unroll
    for (int j = 0; j < 16; ++j) { zb[j] = 0.f; act[j] = __float2bfloat16_rn(0.f); }
    if (!kStep) fetch(half * 16);
    const bool ok = !any || mbar_wait_warp(&sh.acc_bar, 0, abortp, g.status, ERR_EPILOGUE);
    if (kStep && ok) {
      // The bias step's sums in the order of the plain form's tile: a sum over every second 32 columns of a learner, from
      // the first, and one over the others.  One learner: a sum to each half of the warps; several: a learner, both sums.
      tc_fence_after_sync();
      const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
      const int groups = g.cols / 16;
      int q = nl > 1 ? half : 0, which = nl > 1 ? 0 : half, gr = 2 * which;
      float s = 0.f;
      auto settle = [&] {                          // on to a group of 16 columns that exists, or behind the last learner
        while (q < nl && gr >= groups) {
          colsum[(which * nl + q) * kBM + row] = s;
          s = 0.f;
          if (nl > 1 && which == 0) {
            which = 1;
          } else {
            q += nl > 1 ? 2 : 1;
            which = nl > 1 ? 0 : half;
          }
          gr = 2 * which;
        }
      };
      auto place = [&] { return ((size_t)(p0 + q) * g.kb + r0 + 16 * gr) * g.M + m; };
      auto fetch_act = [&] {
        if (m_ok && q < nl) {
          const size_t at = place();
#pragma unroll
          for (int j = 0; j < 16; ++j) act[j] = g.act[at + (size_t)j * g.M];
        }
      };
      settle();
      fetch_act();
#pragma unroll 1
      while (q < nl) {
        const size_t at = place();
        float z[16];
        load16(lane_addr + (uint32_t)(q * g.cols + 16 * gr), true, z);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          z[j] = __bfloat162float(act[j]) > 0.f ? z[j] : 0.f;        // ReLU'(0) = 0
          s += z[j];
        }
        gr += gr & 1 ? 3 : 1;
        settle();
        fetch_act();
        if (m_ok) {
#pragma unroll
          for (int j = 0; j < 16; ++j) g.out[at + (size_t)j * g.M] = __float2bfloat16_rn(z[j]);
        }
      }
    }
    if (!kStep && ok) {
      tc_fence_after_sync();
      const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
#pragma unroll 1
      for (int c0 = half * 16; c0 < end; c0 += 32) {
        size_t at, z_at;
        int q;
        locate(c0, at, z_at, q);
        float z[16];
        load16(lane_addr + (uint32_t)c0, any, z);
        if (kRuns && runs > 1) {
#pragma unroll 1
          for (int r = 1; r < runs; ++r) {
            float t[16];
            load16(lane_addr + (uint32_t)(r * N + c0), true, t);
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] += t[j];
          }
        }
        if (LOW) {
          float low[16];
          load16(lane_addr + g.low_col + (uint32_t)c0, any, low);
#pragma unroll
          for (int j = 0; j < 16; ++j) z[j] = with_low(z[j], low[j]);
        }
        if (kFwd) {
#pragma unroll
          for (int j = 0; j < 16; ++j) z[j] = (add_base ? z[j] + zb[j] : z[j]) + bias_next;
          fetch(c0 + 32);
          if (m_ok) {
#pragma unroll
            for (int j = 0; j < 16; ++j) g.out[at + (size_t)j * g.M] = __float2bfloat16_rn(z[j] > 0.f ? z[j] : 0.f);
          }
        } else if (EPI == PROD_DGRAD) {
          float s = 0.f;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            z[j] = __bfloat162float(act[j]) > 0.f ? z[j] : 0.f;      // ReLU'(0) = 0
            s += z[j];
          }
          fetch(c0 + 32);
          if (m_ok) {
#pragma unroll
            for (int j = 0; j < 16; ++j) g.out[at + (size_t)j * g.M] = __float2bfloat16_rn(z[j]);
          }
          colsum[(half * nl + q) * kBM + row] += s;
        } else if (m_ok) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < end) g.raw[z_at + (size_t)j * g.M] = z[j];
        }
      }
    }
    if (kMn) {
      // bias step of the layer below, b[m] -= gamma * sum_b dZ[b, m]: the two warps that share a row add
      // their sums in a fixed order
      epilogue_barrier();
      if (g.c_tiles > 1) {
        if (half == 0) sh.colsum[0][row] = ok ? colsum[row] + colsum[kBM + row] : 0.f;
      } else if (ok && m_ok) {
        for (int q = half; q < nl; q += 2) {
          const float w_in = g.bias_in[(size_t)(p0 + q) * g.bias_in_stride + g.bias_off + m];
          float* u = kStep && g.mom.u ? g.mom.u + (size_t)(p0 + q) * g.mom.u_stride + g.bias_off + m : nullptr;
          local_update(g.bias_rep + (size_t)(p0 + q) * g.rep_stride + g.bias_off + m, w_in, u, g.mom.read_u,
                       colsum[q * kBM + row] + colsum[(nl + q) * kBM + row], g.gamma, g.mom.beta);
        }
      }
    }
  }
  if (EPI == PROD_DGRAD && g.c_tiles > 1) {
    __syncthreads();
    cluster_sync_all();
    const int row = (int)threadIdx.x, m = m0 + row, rank0 = GRAM ? m_tile * g.c_tiles : 0;
    if (c_tile == 0 && row < kBM && m < g.M) {
      float s = 0.f;
      for (int r = 0; r < g.c_tiles; ++r) s += ld_cluster_f32(mapa_u32(smem_u32(&sh.colsum[0][row]), (uint32_t)(rank0 + r)));
      const float w_in = g.bias_in[(size_t)p0 * g.bias_in_stride + g.bias_off + m];
      local_update(g.bias_rep + (size_t)p0 * g.rep_stride + g.bias_off + m, w_in, nullptr, 0, s, g.gamma, 0.f);
    }
    __syncwarp();
    cluster_sync_all();           // nobody leaves while its sums may still be read
  } else if (GRAM) {
    __syncwarp();
    cluster_sync_all();           // nobody leaves while a peer may still arrive on its barrier
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, g.tmem_cols);
}

// ---------------------------------------------------------------------------------------- Gram

struct GramArgs {
  int B, BN, m_tiles, n_tiles;
  int row0;                 // first batch row (inside a learner's rows) of column tile 0
  int row_end;              // rows from here on do not exist
  int s_row0;               // row of the result that batch row `row0` goes to
  int64_t s_stride, s_ld;   // elements from learner to learner and from row to row of the result
  int nkb, stages;
  uint32_t tmem_cols;
  __nv_bfloat16* out;
  float gamma;
  int* status;
};

// S[row, s] = -gamma <batch row, history row s> for the rows s of the steps before the batch row's own.
// grid (m_tiles x column tiles, P): 128 history rows x BN batch rows per block.
// The history is read once per batch column tile: 126 MB at P = 32, 960 rows of 2048, 26 us = 4.9 TB/s
// (35 us with one block per SM, whose 256 blocks took two waves).
__global__ void __launch_bounds__(kFacThreads, 2)
k_fac_gram(const __grid_constant__ CUtensorMap tm_hist, const __grid_constant__ CUtensorMap tm_b,
           const GramArgs g) {
  const int n_tile = (int)blockIdx.x % g.n_tiles, m_tile = (int)blockIdx.x / g.n_tiles;
  const int p = (int)blockIdx.y, s0 = m_tile * kBM, r0 = g.row0 + n_tile * g.BN;
  const int r1 = min(r0 + g.BN, g.row_end);
  const int limit = (r1 - 1) / g.B * g.B;          // rows of the steps before the tile's last row's own
  if (s0 >= limit) {                               // nothing here: let the next kernel begin
    grid_launch_dependents();
    return;
  }
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) GemmShared sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = g.stages;
  const int stage_bytes = kATileBytes + g.BN * kBK * 2;
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tm_hist);
    tma_prefetch_desc(&tm_b);
    gemm_init_barriers(sh, stages);
    sh.abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_slot, g.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = sh.tmem_slot;
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();
  volatile int* abortp = &sh.abort_flag;
  if (warp == 0) {
    if (lane == 0) {
      Ring ring;
      int issued = 0;
      for (int i = 0; i < g.nkb; ++i, ++issued, ring.next(stages)) {
        uint64_t* full = &sh.full_bar[ring.s];
        if (!mbar_wait(&sh.empty_bar[ring.s], ring.ph ^ 1, abortp, g.status, ERR_PRODUCER)) break;
        uint8_t* sa = smem + (size_t)ring.s * stage_bytes;
        mbar_arrive_expect_tx(full, (uint32_t)stage_bytes);
        tma_load_3d(sa, &tm_hist, full, i * kBK, s0, p);
        tma_load_3d(sa + kATileBytes, &tm_b, full, i * kBK, r0, p);
      }
      if (*abortp) drain_copies(sh.full_bar, issued, stages, g.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      Ring ring;
      const uint32_t idesc = idesc_bf16_f32(kBM, g.BN), unit = (uint32_t)stage_bytes >> 4;
      const uint64_t a0 = smem_desc_k_sw128(smem_u32(smem)), b0 = smem_desc_k_sw128(smem_u32(smem) + kATileBytes);
      bool ok = true;
      for (int i = 0; i < g.nkb; ++i, ring.next(stages)) {
        if (!(ok = mbar_wait(&sh.full_bar[ring.s], ring.ph, abortp, g.status, ERR_MMA))) break;
        tc_fence_after_sync();
        const uint32_t off = (uint32_t)ring.s * unit;
        slab_mma(tmem_base, a0 + off, kStepK, b0 + off, kStepK, idesc, i > 0);
        umma_commit(&sh.empty_bar[ring.s]);
      }
      if (ok) umma_commit(&sh.acc_bar);
    }
    __syncwarp();
  } else {
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    const int s = s0 + q4 * 32 + lane;
    if (mbar_wait_warp(&sh.acc_bar, 0, abortp, g.status, ERR_EPILOGUE)) {
      tc_fence_after_sync();
      const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
#pragma unroll 1
      for (int c0 = half * 16; c0 < r1 - r0; c0 += 32) {
        float z[16];
        load16(lane_addr + (uint32_t)c0, true, z);
        if (s >= limit) continue;
        __nv_bfloat16* dst = g.out + (size_t)p * g.s_stride + (size_t)(g.s_row0 + (r0 - g.row0) + c0) * g.s_ld + s;
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (r0 + c0 + j < r1) dst[(size_t)j * g.s_ld] = __float2bfloat16_rn(-g.gamma * z[j]);
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, g.tmem_cols);
}

// ---------------------------------------------------------------------------------- last layer
// Everything of the last layer in one launch: logits, loss, dZ_L, the data gradient with the ReLU mask,
// the weight gradient with the SGD step, and the bias steps of the last two layers.  A cluster per learner,
// each block a range of `cw` input columns: partial logits meet through distributed shared memory, added
// in rank order; the rest needs a block's own columns only.  At most 32 classes: the three products are
// warp-level MMAs on shared memory, a few hundred per block.  Latency throughout: 2048-10, B = 64, P = 32:
// 17 us, against 35 for the two tensor-core launches of the plain form and another 17 for its weight gradient.

constexpr int kLastThreads = 256;

struct LastArgs {
  const __nv_bfloat16* a;   // A_{L-1}: rows of `in` at a + (p * kb + row0 + b) * in
  __nv_bfloat16* dz;        // dZ_{L-1}, the same rows
  int64_t kb;
  int row0, B, in, C, cw;   // cw: a multiple of 16
  const float* w_in;        // W_L, b_L, b_{L-1} are read at w_in + p * w_in_stride (w~: stride 0) ...
  int64_t w_in_stride;
  float* rep;               // ... and written at rep + p * rep_stride
  int64_t rep_stride, w_off, b_off, bprev_off;
  const int32_t* labels;
  float* loss_out;
  int loss_stride;
  float gamma;
};

// Elements per row of a shared-memory array of `cols` columns (a multiple of 8): an odd number of 16-byte
// units, so that eight consecutive rows start in different banks.
__host__ __device__ constexpr int row_pitch(int cols) { return ((cols >> 3) | 1) << 3; }

// KC: 16-class blocks (1 or 2).  grid (blocks per learner, P), clusters of a learner's blocks.
template <int KC>
__global__ void __launch_bounds__(kLastThreads)
k_fac_last(const LastArgs g) {
  constexpr int CP = 16 * KC;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)blockIdx.x, ranks = (int)gridDim.x, p = (int)blockIdx.y;
  const int c0 = rank * g.cw, nc = min(g.cw, g.in - c0);       // nc: a multiple of 8, at least 8
  const int B = g.B, C = g.C;
  const int ap = row_pitch(g.cw), dp = row_pitch(CP);
  float* Wf = reinterpret_cast<float*>(smem_raw);                             // [C][cw] masters
  float* zp = Wf + (size_t)C * g.cw;                                          // [B][CP] partial logits
  float* sums = zp + (size_t)B * CP;                                          // [8][CP + 1] rank 0: bias gradients, loss
  float* wsum = sums + 8 * (CP + 1);                                          // [8][CP + 1] the same of a block's warps
  __nv_bfloat16* As = reinterpret_cast<__nv_bfloat16*>(wsum + 8 * (CP + 1));  // [B][ap]
  __nv_bfloat16* Ws = As + (size_t)B * ap;                                    // [CP][ap]
  __nv_bfloat16* Wl = Ws + (size_t)CP * ap;                                   // [CP][ap] what Ws leaves over
  __nv_bfloat16* Ds = Wl + (size_t)CP * ap;                                   // [B][dp] dZ_L, bf16
  static_assert((8 * (CP + 1) * 2) % 4 == 0, "As starts on 16 bytes");

  grid_launch_dependents();
  grid_dependency_wait();
  const float* w_in = g.w_in + (size_t)p * g.w_in_stride;
  float* rep = g.rep + (size_t)p * g.rep_stride;
  const size_t arow = (size_t)p * g.kb + g.row0;
  // this warp's rows of the softmax: a range of the batch per rank, its rows in turn
  const int rb = (B + ranks - 1) / ranks, b_first = rank * rb, b_end = min(B, b_first + rb);
  const float bias = lane < C ? w_in[g.b_off + lane] : 0.f;
  int label = b_first + warp < b_end ? g.labels[(size_t)p * B + b_first + warp] : 0;
  {
    const int u = g.cw >> 3;                                   // 16-byte units of a row
    const uint4 zero = make_uint4(0, 0, 0, 0);
    for (int i0 = tid; i0 < B * u; i0 += 8 * kLastThreads) {
      uint4 v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int i = i0 + j * kLastThreads, b = i / u, c = (i - b * u) * 8;
        v[j] = zero;
        if (i < B * u && c < nc) v[j] = *reinterpret_cast<const uint4*>(g.a + (arow + b) * g.in + c0 + c);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int i = i0 + j * kLastThreads, b = i / u, c = (i - b * u) * 8;
        if (i < B * u) *reinterpret_cast<uint4*>(As + (size_t)b * ap + c) = v[j];
      }
    }
    for (int i = tid; i < CP * u; i += kLastThreads) {
      const int c = i / u, k = (i - c * u) * 8;
      float4 v0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = v0;
      if (c < C && k < nc) {
        const float4* src = reinterpret_cast<const float4*>(w_in + g.w_off + (size_t)c * g.in + c0 + k);
        v0 = src[0];
        v1 = src[1];
      }
      if (c < C) {
        float4* dst = reinterpret_cast<float4*>(Wf + (size_t)c * g.cw + k);
        dst[0] = v0;
        dst[1] = v1;
      }
      __nv_bfloat162 h[4] = {__floats2bfloat162_rn(v0.x, v0.y), __floats2bfloat162_rn(v0.z, v0.w),
                             __floats2bfloat162_rn(v1.x, v1.y), __floats2bfloat162_rn(v1.z, v1.w)};
      *reinterpret_cast<uint4*>(Ws + (size_t)c * ap + k) = *reinterpret_cast<uint4*>(h);
      *reinterpret_cast<uint4*>(Wl + (size_t)c * ap + k) =
          make_uint4(low_pair(v0.x, v0.y), low_pair(v0.z, v0.w), low_pair(v1.x, v1.y), low_pair(v1.z, v1.w));
    }
  }
  __syncthreads();
  const int qr = lane >> 2, qc = 2 * (lane & 3);               // row and column of this lane in an MMA's result
  const int mi = lane >> 3, mr = lane & 7;                     // matrix and row this lane addresses for ldmatrix

  // partial logits: 16 rows x 8 classes per warp and turn
  for (int t = warp; t < (B >> 4) * (CP >> 3); t += kLastThreads / 32) {
    const int mt = t / (CP >> 3), nt = t - mt * (CP >> 3);
    float d[4] = {0.f, 0.f, 0.f, 0.f}, dl[4] = {0.f, 0.f, 0.f, 0.f};
    const __nv_bfloat16* arow_s = As + (size_t)(mt * 16 + (mi & 1) * 8 + mr) * ap + (mi >> 1) * 8;
    const __nv_bfloat16* wrow_s = Ws + (size_t)(nt * 8 + mr) * ap + (mi & 1) * 8;
    for (int k = 0; k < g.cw; k += 16) {
      uint32_t a[4], b[2], bl[2];
      ldsm_x4(a, arow_s + k);
      ldsm_x2(b, wrow_s + k);
      ldsm_x2(bl, wrow_s + k + (size_t)CP * ap);
      mma_bf16(d, a, b[0], b[1]);
      mma_bf16(dl, a, bl[0], bl[1]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = with_low(d[i], dl[i]);
    float* z = zp + (size_t)(mt * 16 + qr) * CP + nt * 8 + qc;
    *reinterpret_cast<float2*>(z) = make_float2(d[0], d[1]);
    *reinterpret_cast<float2*>(z + 8 * CP) = make_float2(d[2], d[3]);
  }
  __syncthreads();
  cluster_sync_all();
  // Softmax cross-entropy of this block's share of the rows: a warp per row, a lane per class; the row of
  // dZ_L goes to every block of the cluster.
  {
    float dsum = 0.f, lsum = 0.f;
    for (int b = b_first + warp; b < b_end; b += kLastThreads / 32) {
      const uint32_t at = smem_u32(zp + (size_t)b * CP + (lane < CP ? lane : 0));
      float v[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) v[r] = r < ranks ? ld_cluster_f32(mapa_u32(at, (uint32_t)r)) : 0.f;
      float z = v[0];
#pragma unroll
      for (int r = 1; r < 8; ++r)
        if (r < ranks) z += v[r];                              // ascending ranks
      z = lane < C ? z + bias : -INFINITY;
      float mx = z;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float se = lane < C ? __expf(z - mx) : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
      const float lse = mx + __logf(se);
      const float gr = lane < C ? (__expf(z - lse) - (lane == label ? 1.f : 0.f)) * (1.0f / (float)B) : 0.f;
      dsum += gr;
      lsum += lane == label ? lse - z : 0.f;
      if (b + kLastThreads / 32 < b_end) label = g.labels[(size_t)p * B + b + kLastThreads / 32];
      // two classes to a word, CP / 2 words to every rank: lane (word, first rank)
      const float other = __shfl_down_sync(0xffffffffu, gr, 1);
      __nv_bfloat162 h2 = __floats2bfloat162_rn(gr, other);
      const uint32_t word = *reinterpret_cast<uint32_t*>(&h2);
      const uint32_t mine = __shfl_sync(0xffffffffu, word, 2 * (lane % (CP / 2)));
      const uint32_t dst = smem_u32(Ds + (size_t)b * dp + 2 * (lane % (CP / 2)));
      for (int r = lane / (CP / 2); r < ranks; r += 64 / CP) st_cluster_u32(mapa_u32(dst, (uint32_t)r), mine);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane < C) wsum[warp * (CP + 1) + lane] = dsum;
    if (lane == 0) wsum[warp * (CP + 1) + CP] = lsum;
  }
  __syncthreads();
  if (tid <= CP && (tid < C || tid == CP)) {                   // to rank 0: this block's sums
    float s = 0.f;
    for (int w = 0; w < kLastThreads / 32; ++w) s += wsum[w * (CP + 1) + tid];
    st_cluster_u32(mapa_u32(smem_u32(sums + rank * (CP + 1) + tid), 0u), __float_as_uint(s));
  }
  __syncthreads();
  cluster_sync_all();             // dZ_L is whole everywhere; nobody reads another block's memory from here on
  if (rank == 0 && tid <= CP && (tid < C || tid == CP)) {
    float s = 0.f;
    for (int r = 0; r < ranks; ++r) s += sums[r * (CP + 1) + tid];
    if (tid < C) rep[g.b_off + tid] = fmaf(-g.gamma, s, w_in[g.b_off + tid]);
    else g.loss_out[(size_t)p * g.loss_stride] = s / (float)B;
  }
  // weight gradient and step: dW[classes, 8 columns] = dZ^T A per warp and turn
  for (int nt = warp; nt < nc >> 3; nt += kLastThreads / 32) {
    float d[KC][4];
#pragma unroll
    for (int m = 0; m < KC; ++m) d[m][0] = d[m][1] = d[m][2] = d[m][3] = 0.f;
    for (int b0 = 0; b0 < B; b0 += 16) {
      uint32_t b[2];
      ldsm_x2_t(b, As + (size_t)(b0 + (mi & 1) * 8 + mr) * ap + nt * 8);
#pragma unroll
      for (int m = 0; m < KC; ++m) {
        uint32_t a[4];
        ldsm_x4_t(a, Ds + (size_t)(b0 + (mi >> 1) * 8 + mr) * dp + m * 16 + (mi & 1) * 8);
        mma_bf16(d[m], a, b[0], b[1]);
      }
    }
#pragma unroll
    for (int m = 0; m < KC; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = m * 16 + h * 8 + qr;
        if (c < C) {
          const float2 w = *reinterpret_cast<const float2*>(Wf + (size_t)c * g.cw + nt * 8 + qc);
          *reinterpret_cast<float2*>(rep + g.w_off + (size_t)c * g.in + c0 + nt * 8 + qc) =
              make_float2(fmaf(-g.gamma, d[m][2 * h], w.x), fmaf(-g.gamma, d[m][2 * h + 1], w.y));
        }
      }
  }
  __syncthreads();                // A has been read as an operand; the masked dZ takes its place
  for (int nt = warp; nt < nc >> 3; nt += kLastThreads / 32) {
    uint32_t wb[KC][2];
#pragma unroll
    for (int k = 0; k < KC; ++k) ldsm_x2_t(wb[k], Ws + (size_t)(k * 16 + (mi & 1) * 8 + mr) * ap + nt * 8);
    float s0 = 0.f, s1 = 0.f;
    for (int b0 = 0; b0 < B; b0 += 16) {
      float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < KC; ++k) {
        uint32_t a[4];
        ldsm_x4(a, Ds + (size_t)(b0 + (mi & 1) * 8 + mr) * dp + k * 16 + (mi >> 1) * 8);
        mma_bf16(d, a, wb[k][0], wb[k][1]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        __nv_bfloat162* cell = reinterpret_cast<__nv_bfloat162*>(As + (size_t)(b0 + h * 8 + qr) * ap + nt * 8 + qc);
        const __nv_bfloat162 act = *cell;
        const float v0 = __low2float(act) > 0.f ? d[2 * h] : 0.f;                // ReLU'(0) = 0
        const float v1 = __high2float(act) > 0.f ? d[2 * h + 1] : 0.f;
        s0 += v0;
        s1 += v1;
        *cell = __floats2bfloat162_rn(v0, v1);
      }
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, o);
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
    }
    if (qr == 0) {
      const int64_t at = g.bprev_off + c0 + nt * 8 + qc;
      const float2 w = make_float2(w_in[at], w_in[at + 1]);
      rep[at] = fmaf(-g.gamma, s0, w.x);
      rep[at + 1] = fmaf(-g.gamma, s1, w.y);
    }
  }
  __syncthreads();
  {
    const int u = nc >> 3;
    for (int i = tid; i < B * u; i += kLastThreads) {
      const int b = i / u, c = (i - b * u) * 8;
      *reinterpret_cast<uint4*>(g.dz + (arow + b) * g.in + c0 + c) = *reinterpret_cast<const uint4*>(As + (size_t)b * ap + c);
    }
  }
}

// --------------------------------------------------------------------------------------- apply

constexpr int kApplyBN = 256;                       // input columns per tile
constexpr int kApplyChunk = 32;                     // columns of a master piece
constexpr int kPieceBytes = kBM * kApplyChunk * 4;  // 16 KB, rows of 128 bytes, 128-byte swizzle
constexpr int kApplyStageBytes = kATileBytes + kApplyBN * kBK * 2;
constexpr int kMaxHidden = MAVG_MAX_LAYERS - 1;
constexpr int kApplyStages = 3, kApplyPieces = 2;
constexpr size_t apply_smem(int stages, int pieces) {
  return (size_t)stages * kApplyStageBytes + (size_t)2 * pieces * kPieceBytes + 1024;
}

struct ApplyLayer { int m_tiles, n_tiles, in, first; };   // first: tiles of the layers before
struct ApplyArgs {
  CUtensorMap dz[kMaxHidden], a[kMaxHidden], w_in[kMaxHidden], w_out[kMaxHidden];
  ApplyLayer layer[kMaxHidden];
  int n_layers, per_learner, tiles;                 // tiles of one learner, of all
  int rows;                                         // contraction: K * B
  float gamma;
  int* status;
};
template <int STAGES, int PIECES>
struct alignas(16) ApplyShared {            // (whole 16 bytes, as static shared memory is counted)
  uint64_t full_bar[STAGES], empty_bar[STAGES];
  uint64_t acc_full[2], acc_empty[2];
  uint64_t piece_full[2][PIECES];
  uint32_t tmem_slot;
  int abort_flag;
};

// Persistent: 128 x 256 tiles of W_l, learner by learner (their factors then stay in the L2 while all
// tiles of the learner read them).  Two accumulators, so that a tile's contraction runs while the tile
// before it is subtracted from w~ and stored.
// Bound by what an SM takes in (48 KB of operands per 4.2 Mflop, w~ once more per learner): 1.01 ms at
// n = 14.7 M, P = 32, 1024 rows = 950 TFLOP/s; the weight-gradient launches it replaces took 12 ms there.
// n = 1.84 M, P = 48, 512 rows: 131 us.  Two stages and four pieces per group: 156 there; tiles of 256 x 256,
// which take in a third less but leave no room for a second accumulator or a third stage: 185 and 1.26 ms.
// STAGES operand slabs of 64 rows; PIECES buffers per epilogue group, of which a piece is worked on, one or
// two are being fetched and the rest is being stored.
template <int STAGES, int PIECES>
__global__ void __launch_bounds__(kFacThreads, 1)
k_fac_apply(const __grid_constant__ ApplyArgs g) {
  extern __shared__ uint8_t smem_raw[];
  static_assert(PIECES >= 2 && apply_smem(STAGES, PIECES) <= 225 * 1024, "");
  constexpr int kStores = PIECES > 2 ? 1 : 0;       // stores that may still be reading when a piece is begun
  constexpr int kAhead = PIECES - 1 - kStores;      // pieces fetched ahead
  __shared__ __align__(8) ApplyShared<STAGES, PIECES> sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  uint8_t* pieces = smem + STAGES * kApplyStageBytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&sh.full_bar[s], 1);
      mbar_init(&sh.empty_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sh.acc_full[b], 1);
      mbar_init(&sh.acc_empty[b], 8);
      for (int s = 0; s < PIECES; ++s) mbar_init(&sh.piece_full[b][s], 1);
    }
    sh.abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_slot, 2 * kApplyBN);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = sh.tmem_slot;
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();
  volatile int* abortp = &sh.abort_flag;
  const int nslab = (g.rows + kBK - 1) / kBK;
  auto decode = [&](int t, int& p, int& l, int& m0, int& n0) {
    p = t / g.per_learner;
    int r = t - p * g.per_learner;
    l = 0;
    while (l + 1 < g.n_layers && r >= g.layer[l + 1].first) ++l;
    r -= g.layer[l].first;
    m0 = (r % g.layer[l].m_tiles) * kBM;
    n0 = (r / g.layer[l].m_tiles) * kApplyBN;
  };

  if (warp == 0) {
    if (lane == 0) {
      Ring ring;
      int issued = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
        int p, l, m0, n0;
        decode(t, p, l, m0, n0);
        const CUtensorMap *tm_a = &g.dz[l], *tm_b = &g.a[l];
        for (int i = 0; i < nslab; ++i, ++issued, ring.next(STAGES)) {
          uint64_t* full = &sh.full_bar[ring.s];
          if (!(ok = mbar_wait(&sh.empty_bar[ring.s], ring.ph ^ 1, abortp, g.status, ERR_PRODUCER))) break;
          uint8_t* sa = smem + (size_t)ring.s * kApplyStageBytes;
          mbar_arrive_expect_tx(full, (uint32_t)kApplyStageBytes);
#pragma unroll
          for (int h = 0; h < kBM / 64; ++h) tma_load_3d(sa + h * 8192, tm_a, full, m0 + 64 * h, i * kBK, p);
#pragma unroll
          for (int h = 0; h < kApplyBN / 64; ++h)
            tma_load_3d(sa + kATileBytes + h * 8192, tm_b, full, n0 + 64 * h, i * kBK, p);
        }
      }
      if (*abortp) drain_copies(sh.full_bar, issued, STAGES, g.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      Ring ring;
      uint32_t n = 0;
      bool ok = true;
      const uint32_t idesc = idesc_bf16_f32(kBM, kApplyBN, 1, 1);
      const uint64_t a0 = smem_desc_mn_sw128(smem_u32(smem)), b0 = smem_desc_mn_sw128(smem_u32(smem) + kATileBytes);
      for (int t = blockIdx.x; t < g.tiles && ok; t += gridDim.x, ++n) {
        const uint32_t b = n & 1, d = tmem_base + b * kApplyBN;
        if (!mbar_wait(&sh.acc_empty[b], ((n >> 1) & 1) ^ 1, abortp, g.status, ERR_MMA)) break;
        tc_fence_after_sync();
        for (int i = 0; i < nslab; ++i, ring.next(STAGES)) {
          if (!(ok = mbar_wait(&sh.full_bar[ring.s], ring.ph, abortp, g.status, ERR_MMA))) break;
          tc_fence_after_sync();
          const uint32_t off = (uint32_t)ring.s * (kApplyStageBytes >> 4);
          if (g.rows - i * kBK >= kBK) slab_mma(d, a0 + off, kStepMn, b0 + off, kStepMn, idesc, i > 0);
          else part_mma(d, a0 + off, kStepMn, b0 + off, kStepMn, idesc, i > 0, (g.rows - i * kBK) / 16);
          umma_commit(&sh.empty_bar[ring.s]);
        }
        if (ok) umma_commit(&sh.acc_full[b]);
      }
    }
    __syncwarp();
  } else {
    // Two groups of four warps take a tile's pieces (128 rows x 32 columns) in turn.  A group's first
    // thread fetches the w~ pieces ahead of their use and stores the finished ones.
    const int grp = (warp - 2) >> 2, q4 = warp & 3, row = q4 * 32 + lane;
    const bool leader = ((warp - 2) & 3) == 0 && lane == 0;
    uint8_t* mine = pieces + (size_t)grp * PIECES * kPieceBytes;
    // the leader's place in the group's list of pieces: the next one to fetch
    int ft = blockIdx.x, fc = grp;
    uint32_t fn = 0;
    auto fetch = [&]() {
      while (ft < g.tiles) {
        int p, l, m0, n0;
        decode(ft, p, l, m0, n0);
        const int c = fc;
        if (c >= kApplyBN / kApplyChunk || n0 + c * kApplyChunk >= g.layer[l].in) {
          ft += gridDim.x;
          fc = grp;
          continue;
        }
        fc += 2;
        const uint32_t s = fn % PIECES;
        mbar_arrive_expect_tx(&sh.piece_full[grp][s], kPieceBytes);
        tma_load_3d(mine + (size_t)s * kPieceBytes, &g.w_in[l], &sh.piece_full[grp][s], n0 + c * kApplyChunk, m0, 0);
        ++fn;
        return;
      }
    };
    if (leader)
      for (int i = 0; i < kAhead; ++i) fetch();
    // A wait that was given up is carried to the group's next barrier, which all four warps leave
    // together: nobody is left behind at a counted barrier.
    uint32_t n = 0, pn = 0;
    bool failed = false, gone = false;
    for (int t = blockIdx.x; t < g.tiles && !gone; t += gridDim.x, ++n) {
      int p, l, m0, n0;
      decode(t, p, l, m0, n0);
      const uint32_t b = n & 1;
      if (!mbar_wait(&sh.acc_full[b], (n >> 1) & 1, abortp, g.status, ERR_EPILOGUE)) failed = true;
      tc_fence_after_sync();
      for (int c = grp; c < kApplyBN / kApplyChunk && n0 + c * kApplyChunk < g.layer[l].in; c += 2, ++pn) {
        const uint32_t s = pn % PIECES;
        if (leader) {
          // the store that last read the buffer of the next fetch is done with it
          tma_store_wait_read<kStores>();
          fetch();
        }
        uint32_t acc[32];
        tmem_ld_32x32(tmem_base + ((uint32_t)(q4 * 32) << 16) + b * kApplyBN + (uint32_t)(c * kApplyChunk), acc);
        if (!mbar_wait(&sh.piece_full[grp][s], (pn / PIECES) & 1, abortp, g.status, ERR_EPILOGUE)) failed = true;
        tmem_ld_wait();
        uint8_t* wrow = mine + (size_t)s * kPieceBytes + (size_t)row * 128;
#pragma unroll
        for (int v = 0; v < 8; ++v) {
          float4* cell = reinterpret_cast<float4*>(wrow + ((v ^ (row & 7)) << 4));
          float4 w = *cell;
          w.x = fmaf(-g.gamma, __uint_as_float(acc[4 * v]), w.x);
          w.y = fmaf(-g.gamma, __uint_as_float(acc[4 * v + 1]), w.y);
          w.z = fmaf(-g.gamma, __uint_as_float(acc[4 * v + 2]), w.z);
          w.w = fmaf(-g.gamma, __uint_as_float(acc[4 * v + 3]), w.w);
          *cell = w;
        }
        fence_proxy_async();
        if ((gone = barrier_any(failed, 2 + grp, 128))) break;
        if (leader) {
          tma_store_3d(&g.w_out[l], mine + (size_t)s * kPieceBytes, n0 + c * kApplyChunk, m0, p);
          tma_store_commit();
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.acc_empty[b]);
    }
    if (leader) {
      tma_store_wait_read<0>();
      if (*abortp) drain_copies(sh.piece_full[grp], (int)fn, PIECES, g.status);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, 2 * kApplyBN);
}

// ----------------------------------------------------------------------------------- host side
size_t up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Rows of X per tile where all steps' rows are one operand: at most 256, a multiple of 16, even tiles.
int row_tile_of(int64_t rows) {
  const int64_t tiles = (rows + 255) / 256;
  return (int)up((size_t)((rows + tiles - 1) / tiles), 16);
}

// How a product's columns are cut into blocks, given its row tiles: several learners to a block, up to 256
// columns (they share the w~ tile), while the blocks still take four fifths of the SMs; with fewer row
// tiles a learner's batch in pieces, of 32 columns at least.
FacCols cols_for(int P, int B, long row_tiles, int sm_count, int most_learners = 16, int most_tiles = 8) {
  FacCols c{std::min({std::max(1, 256 / B), P, most_learners}), B, 1};
  auto few = [&] { return row_tiles * ((P + c.nl - 1) / c.nl) * c.c_tiles * 5 < 4L * sm_count; };
  while (c.nl > 1 && few()) c.nl = (c.nl + 1) / 2;
  while (few() && c.cols % 32 == 0 && c.cols > 32 && 2 * c.c_tiles <= most_tiles) {
    c.cols /= 2;
    c.c_tiles *= 2;
  }
  return c;
}

// Cut of a product that forms its own Gram rows where it can: short launches (a learner per block at most, so
// that the blocks take the SMs) of at most four row tiles, which with the column tiles are one cluster.
// us a round with the Gram rows in launches of their own / in the product's: 3072-512-512-10, K = 8, P = 8,
// B = 128 475 / 469, P = 48, B = 64 876 / 861; 520-200-136-12, P = 20, K = 9, B = 48 372 / 339; six row tiles:
// 1504-672-672-11, P = 10, K = 8, B = 176 788 / 793; eight: 3072-1024-1024-1024-10, P = 16, K = 8, B = 64
// 977 / 1288 (clusters of eight blocks of one per SM).
FacCols product_cols(int P, int B, int rows, int sm_count) {
  const int m_tiles = (rows + kBM - 1) / kBM;
  FacCols c = cols_for(P, B, m_tiles, sm_count);
  if (c.nl > 1 || m_tiles > 4) return c;
  c = cols_for(P, B, m_tiles, sm_count, 1, 8 / m_tiles);
  c.own_gram = true;
  return c;
}
// Tensor memory of a block that does: its sums and its Gram tiles' (and as many columns again as its sums where
// the low parts' are apart).
int gram_columns(int cols, int m_tiles, int hist) {
  return cols * (1 + ((hist + kBM - 1) / kBM + m_tiles - 1) / m_tiles);
}

struct PdlLaunch {
  cudaLaunchConfig_t lc{};
  cudaLaunchAttribute at[2];
  PdlLaunch(dim3 grid, int threads, size_t smem, cudaStream_t stream, int cluster = 1) {
    lc.gridDim = grid;
    lc.blockDim = dim3((unsigned)threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = cluster > 1 ? 2 : 1;
  }
};

uint32_t tmem_columns(int n) {
  uint32_t c = 32;
  while ((int)c < n) c <<= 1;
  return c;
}

// Two blocks share an SM where there are more blocks than SMs and two stages leave room for them: not with
// two tiles to a stage and 128 columns or more (64 KB).
int stages_for(int slabs, int stage_bytes, long blocks, int sm_count) {
  const int budget = (blocks > sm_count && stage_bytes <= 48 * 1024 ? 96 : 196) * 1024;
  return std::max(2, std::min({kMaxStages, slabs, budget / stage_bytes}));
}

template <int EPI, int TILES, bool LOW = false, bool GRAM = false>
cudaError_t launch_product(mavg_ctx* c, int cls, const CUtensorMap& w, const CUtensorMap& lo, const CUtensorMap& in,
                           const CUtensorMap& hist, const CUtensorMap& s, ProdArgs g, const CUtensorMap* gram = nullptr) {
  g.m_tiles = (g.M + kBM - 1) / kBM;
  g.P = c->cfg.P;
  g.gamma = c->cfg.local_lr;
  g.rep_stride = c->buf.replica_stride;
  g.bias_rep = c->buf.replicas;
  g.status = (int*)ws_ptr(c, c->ws.status);
  const int stage_bytes = product_stage_bytes(TILES, EPI == PROD_RAW ? 1 : TILES, g.nl, g.cols);
  const dim3 grid((unsigned)(g.m_tiles * g.c_tiles), (unsigned)((g.P + g.nl - 1) / g.nl));
  const int hist_stages = ((g.hist + kBK - 1) / kBK + TILES - 1) / TILES;
  g.low_col = (uint32_t)(GRAM ? gram_columns(g.cols, g.m_tiles, g.hist) : g.nl * g.cols);
  g.tmem_cols = tmem_columns(EPI == PROD_FWD_RUNS ? g.runs * g.cols : (int)g.low_col + (LOW ? g.nl * g.cols : 0));
  g.stages = stages_for(std::max(1, g.gram_nkb + g.nkb + g.nl * hist_stages), stage_bytes,
                        EPI == PROD_FWD_RUNS && g.tmem_cols > 256 ? 1 : (long)grid.x * grid.y, c->sm_count);
  size_t smem = (size_t)g.stages * stage_bytes + 1024 +
                (EPI == PROD_DGRAD || EPI == PROD_DGRAD_STEP ? (size_t)2 * g.nl * kBM * sizeof(float) : 0);
  const int cluster = GRAM ? (int)grid.x : EPI == PROD_DGRAD ? g.c_tiles : 1;
  smem = std::max(smem, tmem_share_bytes(g.tmem_cols, sizeof(GemmShared) + (GRAM ? kGramBarBytes : 0)));
  PdlLaunch l(grid, kFacThreads, smem, c->stream, cluster);
  prof_begin(c, cls);
  cudaError_t e = cudaLaunchKernelEx(&l.lc, k_fac_product<EPI, TILES, LOW, GRAM>, w, lo, in, gram ? *gram : in, hist, s, g);
  prof_end(c);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_gram(mavg_ctx* c, int cls, const CUtensorMap& hist, const CUtensorMap& b, int dim, GramArgs g,
                        int hist_rows, bool pairs) {
  g.B = c->cfg.B;
  g.m_tiles = (hist_rows + kBM - 1) / kBM;
  g.nkb = (dim + kBK - 1) / kBK;
  const int stage_bytes = kATileBytes + g.BN * kBK * 2;
  const dim3 grid((unsigned)(g.m_tiles * g.n_tiles), (unsigned)c->cfg.P);
  g.stages = stages_for(g.nkb, stage_bytes, pairs ? (long)grid.x * grid.y : 1, c->sm_count);
  g.tmem_cols = tmem_columns(g.BN);
  g.gamma = c->cfg.local_lr;
  g.status = (int*)ws_ptr(c, c->ws.status);
  PdlLaunch l(grid, kFacThreads, std::max((size_t)g.stages * stage_bytes + 1024, tmem_share_bytes(g.tmem_cols, sizeof(GemmShared))),
              c->stream);
  prof_begin(c, cls);
  cudaError_t e = cudaLaunchKernelEx(&l.lc, k_fac_gram, hist, b, g);
  prof_end(c);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Last layer: blocks per learner and input columns per block.
constexpr size_t kLastSmem = 200 * 1024;
struct LastPlan { int ranks, cw; size_t smem; };
LastPlan last_plan(const mavg_config* cfg) {
  const int in = cfg->dims[cfg->n_layers - 1], B = cfg->B, cp = cfg->dims[cfg->n_layers] > 16 ? 32 : 16;
  LastPlan pl{};
  for (int r = 1; r <= 8; r *= 2) {
    pl.cw = (int)up((size_t)((in + r - 1) / r), 16);
    pl.ranks = (in + pl.cw - 1) / pl.cw;
    pl.smem = ((size_t)(B + 2 * cp) * row_pitch(pl.cw) + (size_t)B * row_pitch(cp)) * 2 +
              ((size_t)cfg->dims[cfg->n_layers] * pl.cw + (size_t)B * cp + 16 * (cp + 1)) * sizeof(float);
    // enough blocks for the SMs, of 64 columns or more; a learner's own products are short, and their
    // latency grows with the columns
    if (pl.smem <= kLastSmem && ((long)cfg->P * pl.ranks >= 148 || pl.cw <= 64)) break;
  }
  return pl;
}

// The minibatches of a call's steps and their labels; low: the low parts of w~ as well (factored steps), else ordered step
// by step (rebuilt ones).
cudaError_t gather_rows(mavg_ctx* c, const FacLayout& t, int rows, int64_t round, bool low) {
  const mavg_config& cfg = c->cfg;
  const int L = cfg.n_layers, P = cfg.P, B = cfg.B, K = cfg.K;
  int32_t* labels = (int32_t*)ws_ptr(c, t.labels);
  __nv_bfloat16* out = (__nv_bfloat16*)ws_ptr(c, t.h[0]);
  const int64_t* rp = c->capturing ? (const int64_t*)(ws_ptr(c, c->ws.status) + 64) : nullptr;
  LowArgs la{};
  int64_t all = 0;
  la.layers = low ? L - 1 : 0;
  for (int l = 1; l <= la.layers; ++l) {
    const MlpLayer& ly = c->layers[l - 1];
    la.w[l - 1] = c->buf.global_w + ly.w_off;
    la.dst[l - 1] = (__nv_bfloat16*)ws_ptr(c, t.w_lo[l]);
    all += la.total[l - 1] = (int64_t)ly.in * ly.out;
  }
  la.blocks = (int)std::min<int64_t>((all + 8191) / 8192, 2 * c->sm_count);
  const unsigned grid = (unsigned)(((int64_t)P * rows + 7) / 8 + la.blocks);
  prof_begin(c, MAVG_K_BATCH);
  if (cfg.x_dtype == MAVG_X_BF16)
    k_fac_gather<__nv_bfloat16><<<grid, 256, 0, c->stream>>>((const __nv_bfloat16*)cfg.x, cfg.y, cfg.seed, round, rp,
                                                            P, K, B, t.kb, cfg.n_samples, cfg.dims[0], labels, out, !low, la);
  else
    k_fac_gather<float><<<grid, 256, 0, c->stream>>>((const float*)cfg.x, cfg.y, cfg.seed, round, rp, P, K, B, t.kb,
                                                     cfg.n_samples, cfg.dims[0], labels, out, !low, la);
  prof_end(c);
  return cudaGetLastError();
}

bool enough_rows(const mavg_config* cfg, int K) { return K >= 2 && (int64_t)cfg->P * K * cfg->B >= 8192; }

}  // namespace

// Where the form is taken.
// Speed: what it saves goes with the weights (none is read or written per learner and step), what it adds
// with the square of a learner's rows K B: the Gram products and the products with them,
// K B (d_0 + d_1 + 2 sum_{l>=2} (d_{l-1} + d_l)) multiply-adds per row against one per hidden weight and
// product.  The lines are drawn through 860 measured models of 0.05 to 60 M hidden weights, P = 2 to 64, K = 2 to 24
// (plain / factored, us a round).  Never from a ratio of 5.5 on: 2024-424-408-88-32, P = 9, K = 9, B = 144 (6.2)
// 910 / 1142, 752-688-688-2, P = 34, K = 8, B = 176 (6.0) 1337 / 1482 (most large ones are faster still:
// 3048-1536-1536-10, P = 6, K = 19, B = 208 (6.0) 5757 / 3749).  Below it
//   - where the learners' weights are many for the launches of a step, P x weights / hidden layers = V:
//     ratio < 0.5 + 0.6 V / 10^6.  3072-2048-2048-2048-10, P = 32, K = 16, B = 64 (1.5, V = 154 M) 15380 / 6360,
//     3072-512-512-10, P = 48, K = 8, B = 64 (1.6, 44 M) 1845 / 862, P = 8, B = 128 (3.1, 7 M) 621 / 470; beyond
//     784-640-3, P = 8, K = 9, B = 176 (4.5, 4 M) 311 / 357, 1752-600-600-16, P = 8, K = 10, B = 144 (4.9, 6 M) 862 / 948,
//     2968-240-240-240-11, P = 16, K = 4, B = 128 (3.2, 4 M) 389 / 441;
//   - batches of up to 96 from V = 2 M on, 3 M with three hidden layers, and below a ratio of 5 with fewer from 1 M on (a
//     step's products then have few columns a learner): 1720-360-13, P = 10, K = 18, B = 80 (4.8, 6 M) 796 / 479,
//     520-200-136-12, P = 20, K = 9, B = 48 (4.6, 1.3 M) 342 / 338; not P = 16, K = 7, B = 80 of the latter (5.9, 1.0 M)
//     275 / 309 nor 336-296-296-296-27, P = 22, K = 5, B = 80 (4.4, 2.0 M) 346 / 364;
//   - one hidden layer, whose step is two launches, up to B = 128 and from V = 2 M on: 664-672-29, P = 7, K = 17, B = 96
//     (4.9, 3 M) 609 / 476; not 536-296-19, P = 10, K = 8, B = 128 (5.4, 1.6 M) 229 / 241.
// Within the lines 3 of 630 models are slower, by 2 to 4 %; 102 beyond them would be faster by a tenth or more.
// Models of fewer than 48 K hidden weights keep the plain form: a round is a chain of short launches either
// way (128-128-128-10, P = 148, B = 32: K = 2 124 / 103, K = 8 371 / 371; 256-128-10, P = 64, K = 4 119 / 110).
// Results: the plain form rounds W_l(k) to bf16 at every step, this one rounds w~ (to 16 bits in the forward
// products, see LowArgs) and the Gram rows; its error against 64 bits is the smaller one, at 2048 rows P K B as at
// 30000.  The two differ from each other by roundings and ReLU branches that vary from row to row: v by 4e-3 to
// 1e-2 from 8192 rows on (6e-3 to 1.6e-2 with three hidden layers and 16 steps), by 1.5e-2 to 3e-2 at 500 to
// 800.  Below 8192 rows the learners keep the rounding of their own weights: a cautious line, not one that the
// error draws.
int fac_steps(const mavg_config* cfg) {
  const int B = cfg->B, hidden = cfg->n_layers - 1;
  if (hidden < 1) return 0;
  int64_t span = cfg->dims[0] + cfg->dims[1], weights = (int64_t)cfg->dims[0] * cfg->dims[1];
  for (int l = 2; l <= hidden; ++l) {
    span += 2 * ((int64_t)cfg->dims[l - 1] + cfg->dims[l]);
    weights += (int64_t)cfg->dims[l - 1] * cfg->dims[l];
  }
  if (weights < 48 * 1024) return 0;
  const double v = 1e-6 * (double)cfg->P * (double)weights / hidden;
  double line = std::min(5.5, 0.5 + 0.6 * v);
  if (v >= (hidden < 3 ? 2.0 : 3.0) && (B <= 96 || (B <= 128 && hidden == 1))) line = 5.5;
  else if (v >= 1.0 && B <= 96 && hidden < 3) line = std::max(line, 5.0);
  const int most = (int)std::min<int64_t>({cfg->K, 4096 / B, ((int64_t)(line * (double)weights) - 1) / (span * B)});
  return enough_rows(cfg, most) && last_plan(cfg).smem <= kLastSmem ? most : 0;
}

bool fac_reserved(const mavg_config* cfg) { return cfg->learner_momentum == 0.f && fac_steps(cfg) == cfg->K; }

FacLayout fac_layout(const mavg_config* cfg, size_t base) {
  FacLayout t;
  const int L = cfg->n_layers, P = cfg->P, B = cfg->B;
  t.kb = (int64_t)fac_steps(cfg) * B;
  t.s_ld = (int64_t)up((size_t)t.kb, 64);
  const size_t rows = (size_t)P * t.kb;
  size_t off = up(base, 1024);
  auto take = [&](size_t bytes) { size_t r = off; off = up(off + bytes, 1024); return r; };
  for (int l = 0; l < L; ++l) {
    t.h[l] = take(rows * cfg->dims[l] * 2);
    if (l > 0) t.g[l] = take(rows * cfg->dims[l] * 2);
  }
  const size_t z_bytes = (size_t)t.kb * cfg->dims[1] * 4, s_bytes = (size_t)t.kb * t.s_ld * 2;
  t.in_rows = z_bytes + s_bytes <= (size_t)cfg->dims[0] * cfg->dims[1] * 4;
  t.zbase = t.in_rows ? 0 : take(P * z_bytes);
  t.s1 = t.in_rows ? z_bytes : take(P * s_bytes);
  for (size_t& s : t.s) s = take((size_t)P * B * t.s_ld * 2);
  t.labels = take(rows * sizeof(int32_t));
  for (int l = 1; l < L; ++l) t.w_lo[l] = take((size_t)cfg->dims[l - 1] * cfg->dims[l] * 2);
  t.end = off;
  return t;
}

void fac_setup(mavg_ctx* c, TcState* st) {
  std::string* why = nullptr;
  const mavg_config& cfg = c->cfg;
  const int L = cfg.n_layers, P = cfg.P, B = cfg.B;
  FacState* f = new FacState();
  f->lay = fac_layout(&cfg, st->lay.shared_end);
  f->K = fac_steps(&cfg);
  const FacLayout& t = f->lay;
  auto bf = [&](size_t off) { return (void*)ws_ptr(c, off); };
  const int kb = (int)t.kb;
  f->row_tile = row_tile_of(t.kb);
  bool ok = true;
  // columns of the Gram products: their row tiles are half the history's on average
  f->gram = cols_for(P, B, std::max<long>(1, (long)((t.kb / 2 + kBM - 1) / kBM)), c->sm_count, 1);
  for (int l = 0; l < L && ok; ++l) {
    const int d = cfg.dims[l];
    const int64_t per = t.kb * d;
    ok = ok && encode_map(st, &f->h_mn[l], bf(t.h[l]), d, kb, P, d, per, 64, why);
    ok = ok && encode_map(st, &f->h_k[l], bf(t.h[l]), d, kb, P, d, per, kBM, why);
    ok = ok && encode_map(st, &f->h_b[l], bf(t.h[l]), d, kb, P, d, per, l == 0 ? f->row_tile : f->gram.cols, why);
    if (l == 0) continue;
    ok = ok && encode_map(st, &f->g_mn[l], bf(t.g[l]), d, kb, P, d, per, 64, why);
    ok = ok && encode_map(st, &f->g_k[l], bf(t.g[l]), d, kb, P, d, per, kBM, why);
    ok = ok && encode_map(st, &f->g_b[l], bf(t.g[l]), d, kb, P, d, per, f->gram.cols, why);
  }
  f->s1_ptr = t.in_rows ? (char*)c->buf.replicas + t.s1 : (char*)bf(t.s1);
  f->z_ptr = t.in_rows ? (char*)c->buf.replicas + t.zbase : (char*)bf(t.zbase);
  f->s1_stride = t.in_rows ? 2 * c->buf.replica_stride : t.kb * t.s_ld;
  f->z_stride = t.in_rows ? c->buf.replica_stride : t.kb * cfg.dims[1];
  for (int l = 1; l < L && ok; ++l) {
    // forward product of layer l; data gradient through layer l
    f->fwd[l] = l == 1 ? cols_for(P, B, (cfg.dims[l] + kBM - 1) / kBM, c->sm_count)
                       : product_cols(P, B, cfg.dims[l], c->sm_count);
    ok = ok && encode_map(st, &f->w_lo[l], bf(t.w_lo[l]), cfg.dims[l - 1], cfg.dims[l], 1, cfg.dims[l - 1],
                          (int64_t)cfg.dims[l - 1] * cfg.dims[l], kBM, why);
    if (l == 1) {
      ok = ok && encode_map(st, &f->s_f[1], f->s1_ptr, (int)t.s_ld, kb, P, t.s_ld, f->s1_stride, f->fwd[1].cols, why);
      continue;
    }
    const int in = cfg.dims[l - 1], out = cfg.dims[l];
    f->dgrad[l] = product_cols(P, B, in, c->sm_count);
    ok = ok && encode_map(st, &f->in[l], bf(t.h[l - 1]), in, kb, P, in, t.kb * in, f->fwd[l].cols, why, f->fwd[l].nl);
    ok = ok && encode_map(st, &f->dz_in[l], bf(t.g[l]), out, kb, P, out, t.kb * out, f->dgrad[l].cols, why,
                          f->dgrad[l].nl);
    ok = ok && encode_map(st, &f->s_f[l], bf(t.s[0]), (int)t.s_ld, B, P, t.s_ld, B * t.s_ld, f->fwd[l].cols, why);
    ok = ok && encode_map(st, &f->s_d[l], bf(t.s[1]), (int)t.s_ld, B, P, t.s_ld, B * t.s_ld, f->dgrad[l].cols, why);
  }
  // what a block can have beside its static shared memory: all of it, for 512 columns of tensor memory
  constexpr size_t kFixed = sizeof(GemmShared), kGramFixed = kFixed + kGramBarBytes;
  const struct { const void* kernel; size_t fixed; } kernels[] = {
      {(const void*)k_fac_product<PROD_FWD, 2, false, false>, kFixed}, {(const void*)k_fac_product<PROD_FWD, 2, true, false>, kFixed},
      {(const void*)k_fac_product<PROD_RAW, 2, true, false>, kFixed}, {(const void*)k_fac_product<PROD_DGRAD, 1, false, false>, kFixed},
      {(const void*)k_fac_product<PROD_FWD, 2, true, true>, kGramFixed}, {(const void*)k_fac_product<PROD_DGRAD, 1, false, true>, kGramFixed},
      {(const void*)k_fac_gram, kFixed}, {(const void*)k_fac_last<1>, 0}, {(const void*)k_fac_last<2>, 0},
      {(const void*)k_fac_apply<kApplyStages, kApplyPieces>, sizeof(ApplyShared<kApplyStages, kApplyPieces>)}};
  for (const auto& k : kernels)
    ok = ok && cudaFuncSetAttribute(k.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(kSmSharedBytes - kBlockReservedBytes - k.fixed)) == cudaSuccess;
  if (ok) {
    st->fac = f;
  } else {
    cudaGetLastError();
    delete f;
  }
}

bool fac_usable(const mavg_ctx* c) {
  const TcState* st = (const TcState*)c->mlp;
  return st && st->fac && c->schedule == 0 && c->cfg.learner_momentum == 0.f &&
         c->cfg.K <= st->fac->K && enough_rows(&c->cfg, c->cfg.K);
}

#define FAC_TRY(call) do { if ((e = (call)) != cudaSuccess) return e; } while (0)

// The K steps of a round.  Chain of a step, layers L:
//   F_1 -> (S_2 -> F_2) -> ... -> last layer -> (T_{L-1} -> D_{L-1}) -> ... -> D_2
// S_l, T_l: the Gram products that the forward product F_l and the data gradient D_l through layer l
// need (none in the first step); a launch of their own or part of F_l and D_l.
cudaError_t fac_local_steps(mavg_ctx* c, int64_t round) {
  TcState* st = (TcState*)c->mlp;
  FacState* f = st->fac;
  const FacLayout& t = f->lay;
  const mavg_config& cfg = c->cfg;
  const int L = cfg.n_layers, P = cfg.P, B = cfg.B, K = cfg.K, rows = K * B;
  auto bfp = [&](size_t off) { return (__nv_bfloat16*)ws_ptr(c, off); };
  int32_t* labels = (int32_t*)ws_ptr(c, t.labels);
  cudaError_t e;

  FAC_TRY(gather_rows(c, t, rows, round, true));
  const int row_tiles = (rows + f->row_tile - 1) / f->row_tile;
  {
    ProdArgs g{};
    g.M = cfg.dims[1];
    g.kb = t.kb;
    g.nl = 1;
    g.cols = f->row_tile;
    g.c_tiles = row_tiles;
    g.row_end = rows;
    g.nkb = (cfg.dims[0] + kBK - 1) / kBK;
    g.raw = (float*)f->z_ptr;
    g.z_stride = f->z_stride;
    FAC_TRY((launch_product<PROD_RAW, 2, true>(c, MAVG_K_FWD, st->wg[1], f->w_lo[1], f->h_b[0], f->g_mn[1], f->s_f[1], g)));
  }
  {
    GramArgs g{};
    g.BN = f->row_tile;
    g.n_tiles = row_tiles;
    g.row_end = rows;
    g.out = (__nv_bfloat16*)f->s1_ptr;
    g.s_stride = f->s1_stride;
    g.s_ld = t.s_ld;
    FAC_TRY(launch_gram(c, MAVG_K_FWD, f->h_k[0], f->h_b[0], cfg.dims[0], g, rows - B, false));
  }
  // -gamma <batch rows, rows of the earlier steps> of one layer's rows
  auto gram = [&](int cls, const CUtensorMap& hist, const CUtensorMap& b, int dim, int i, int k) {
    GramArgs g{};
    g.BN = f->gram.cols;
    g.n_tiles = f->gram.c_tiles;
    g.row0 = (k - 1) * B;
    g.row_end = k * B;
    g.out = bfp(t.s[i]);
    g.s_stride = B * t.s_ld;
    g.s_ld = t.s_ld;
    return launch_gram(c, cls, hist, b, dim, g, (k - 1) * B, true);
  };
  const LastPlan lp = last_plan(&cfg);

  for (int k = 1; k <= K; ++k) {
    const int hist = (k - 1) * B;
    const float* w_in = k == 1 ? c->buf.global_w : c->buf.replicas;      // biases and last layer
    const int64_t w_in_stride = k == 1 ? 0 : c->buf.replica_stride;
    auto product = [&](int M, int bias_layer, const FacCols& cols) {
      ProdArgs g{};
      g.M = M;
      g.kb = t.kb;
      g.row0 = hist;
      g.hist = hist;
      g.nl = cols.nl;
      g.cols = cols.cols;
      g.c_tiles = cols.c_tiles;
      g.bias_off = c->layers[bias_layer - 1].b_off;
      g.bias_in = w_in;
      g.bias_in_stride = w_in_stride;
      return g;
    };
    // the product forms its Gram rows itself
    auto own_gram = [&](const FacCols& cols, int M, bool low) {
      return k > 1 && cols.own_gram && gram_columns(cols.cols, (M + kBM - 1) / kBM, hist) + (low ? cols.cols : 0) <= 256;
    };
    auto with_gram = [&](ProdArgs& g, int dim, int i) {
      g.gram_nkb = (dim + kBK - 1) / kBK;
      g.gram_out = bfp(t.s[i]);
      g.gram_stride = B * t.s_ld;
      g.gram_ld = t.s_ld;
    };
    for (int l = 1; l < L; ++l) {
      ProdArgs g = product(cfg.dims[l], l, f->fwd[l]);
      g.out = bfp(t.h[l]);
      if (l == 1) {
        g.s_row0 = hist;
        g.zbase = (const float*)f->z_ptr;
        g.z_stride = f->z_stride;
        FAC_TRY((launch_product<PROD_FWD, 2>(c, MAVG_K_FWD, st->wg[1], st->wg[1], f->h_b[0], f->g_mn[1], f->s_f[1], g)));
        continue;
      }
      const int in = cfg.dims[l - 1];
      const CUtensorMap &w = st->wg[l], &a = f->in[l], &d = f->g_mn[l], &s = f->s_f[l];
      g.nkb = (in + kBK - 1) / kBK;
      if (own_gram(f->fwd[l], cfg.dims[l], true)) {
        with_gram(g, in, 0);
        FAC_TRY((launch_product<PROD_FWD, 2, true, true>(c, MAVG_K_FWD, w, f->w_lo[l], a, d, s, g, &f->h_k[l - 1])));
        continue;
      }
      if (k > 1) FAC_TRY(gram(MAVG_K_FWD, f->h_k[l - 1], f->h_b[l - 1], in, 0, k));
      FAC_TRY((launch_product<PROD_FWD, 2, true>(c, MAVG_K_FWD, w, f->w_lo[l], a, d, s, g)));
    }
    {
      LastArgs g{};
      const MlpLayer& ly = c->layers[L - 1];
      g.a = bfp(t.h[L - 1]);
      g.dz = bfp(t.g[L - 1]);
      g.kb = t.kb;
      g.row0 = hist;
      g.B = B;
      g.in = ly.in;
      g.C = ly.out;
      g.cw = lp.cw;
      g.w_in = w_in;
      g.w_in_stride = w_in_stride;
      g.rep = c->buf.replicas;
      g.rep_stride = c->buf.replica_stride;
      g.w_off = ly.w_off;
      g.b_off = ly.b_off;
      g.bprev_off = c->layers[L - 2].b_off;
      g.labels = labels + (size_t)(k - 1) * P * B;
      g.loss_out = (float*)ws_ptr(c, c->ws.losses) + (k - 1);
      g.loss_stride = K;
      g.gamma = cfg.local_lr;
      PdlLaunch l(dim3((unsigned)lp.ranks, (unsigned)P), kLastThreads, lp.smem, c->stream, lp.ranks);
      prof_begin(c, MAVG_K_LOSS);
      e = g.C > 16 ? cudaLaunchKernelEx(&l.lc, k_fac_last<2>, g) : cudaLaunchKernelEx(&l.lc, k_fac_last<1>, g);
      prof_end(c);
      FAC_TRY(e);
      FAC_TRY(cudaGetLastError());
    }
    for (int l = L - 1; l > 1; --l) {
      ProdArgs g = product(cfg.dims[l - 1], l - 1, f->dgrad[l]);
      const CUtensorMap &w = st->wg_mn[l], &dz = f->dz_in[l], &a = f->h_mn[l - 1], &s = f->s_d[l];
      g.nkb = (cfg.dims[l] + kBK - 1) / kBK;
      g.out = bfp(t.g[l - 1]);
      g.act = bfp(t.h[l - 1]);
      if (own_gram(f->dgrad[l], cfg.dims[l - 1], false)) {
        with_gram(g, cfg.dims[l], 1);
        FAC_TRY((launch_product<PROD_DGRAD, 1, false, true>(c, MAVG_K_DGRAD, w, w, dz, a, s, g, &f->g_k[l])));
        continue;
      }
      if (k > 1) FAC_TRY(gram(MAVG_K_DGRAD, f->g_k[l], f->g_b[l], cfg.dims[l], 1, k));
      FAC_TRY((launch_product<PROD_DGRAD, 1>(c, MAVG_K_DGRAD, w, w, dz, a, s, g)));
    }
  }
  {
    ApplyArgs g{};
    g.n_layers = L - 1;
    g.rows = rows;
    g.gamma = cfg.local_lr;
    g.status = (int*)ws_ptr(c, c->ws.status);
    for (int l = 1; l < L; ++l) {
      ApplyLayer& a = g.layer[l - 1];
      a.m_tiles = (cfg.dims[l] + kBM - 1) / kBM;
      a.n_tiles = (cfg.dims[l - 1] + kApplyBN - 1) / kApplyBN;
      a.in = cfg.dims[l - 1];
      a.first = g.per_learner;
      g.per_learner += a.m_tiles * a.n_tiles;
      g.dz[l - 1] = f->g_mn[l];
      g.a[l - 1] = f->h_mn[l - 1];
      g.w_in[l - 1] = st->w32g[l];
      g.w_out[l - 1] = st->w32[l];
    }
    g.tiles = g.per_learner * P;
    PdlLaunch l(dim3((unsigned)std::min(g.tiles, c->sm_count)), kFacThreads,
                std::max(apply_smem(kApplyStages, kApplyPieces),
                         tmem_share_bytes(2 * kApplyBN, sizeof(ApplyShared<kApplyStages, kApplyPieces>))),
                c->stream);
    prof_begin(c, MAVG_K_WGRAD_SGD);
    e = cudaLaunchKernelEx(&l.lc, k_fac_apply<kApplyStages, kApplyPieces>, g);
    prof_end(c);
    FAC_TRY(e);
    FAC_TRY(cudaGetLastError());
  }
  return cudaSuccess;
}

// Where rounds are rebuilt instead of stepped in place: where they are not factored and what a step moves, 10 bytes per
// weight in place (18 with momentum), costs more than forming the weights anew from all rows so far, k B in step k.  V: P
// times the hidden layers' weights.  Time in place / rebuilt over 340 shapes (1 to 3 hidden layers of 128 to 2048, P = 2 ..
// 48, B = 16 .. 256, V = 12 .. 190 M):
//   with momentum (all steps' accumulators at once: K <= 4)   V >= 20 M: 1.003 .. 1.57; V = 12 .. 20 M: 0.92 .. 1.31
//   without, V >= 48 M        K <= 4: 1.07 .. 1.50; K = 5, 6: 1.05 .. 1.21 up to 384 rows a learner, 0.969 at 480
//            V = 20 .. 48 M   K <= 4: 0.949 .. 1.36; K = 5, 6: 0.866 .. 1.24
// Where the forward products ride on the weight gradients in place (280 shapes more): with momentum 1.07 .. 1.44; without
// K = 2, 3 1.04 .. 1.51, K = 4 1.09 .. 1.22 up to 64 batch rows and 0.897 .. 1.08 above, K = 5 0.965 and 0.981 (reb_riding).
int reb_steps(const mavg_config* cfg) {
  const int L = cfg->n_layers, B = cfg->B;
  const bool momentum = cfg->learner_momentum != 0.f;
  if (L < 2 || B > 256 || cfg->dims[L] > 32) return 0;
  int64_t weights = 0;
  for (int l = 1; l < L; ++l) weights += (int64_t)cfg->dims[l - 1] * cfg->dims[l];
  if (cfg->P * weights < (momentum ? 20 : 48) * 1000 * 1000) return 0;
  const int most = std::min({cfg->K, 512 / B, momentum || cfg->K * B > 384 ? 4 : 6});
  return most >= 2 ? most : 0;
}

bool reb_riding(const mavg_config* cfg) {
  return cfg->learner_momentum != 0.f || cfg->K <= 3 || (cfg->K == 4 && cfg->B <= 64);
}

bool reb_reserved(const mavg_config* cfg) { return reb_steps(cfg) == cfg->K && !fac_reserved(cfg); }

FacLayout reb_layout(const mavg_config* cfg, size_t base) {
  FacLayout t;
  const int L = cfg->n_layers, P = cfg->P;
  t.kb = (int64_t)reb_steps(cfg) * cfg->B;
  const size_t rows = (size_t)P * t.kb;
  size_t off = up(base, 1024);
  auto take = [&](size_t bytes) { size_t r = off; off = up(off + bytes, 1024); return r; };
  for (int l = 0; l < L; ++l) t.h[l] = take(rows * cfg->dims[l] * 2);
  for (int l = 1; l <= L; ++l) {
    t.g[l] = take(rows * up((size_t)cfg->dims[l], 8) * 2);
    t.w_own[l] = take((size_t)P * cfg->dims[l - 1] * cfg->dims[l] * 2);
    if (l < L) t.act_t[l] = take((size_t)P * cfg->B * cfg->dims[l] * 2);
  }
  t.dz_t = take((size_t)P * cfg->B * *std::max_element(cfg->dims + 1, cfg->dims + L) * 2);
  t.labels = take(rows * sizeof(int32_t));
  t.end = off;
  return t;
}

void reb_setup(mavg_ctx* c, TcState* st) {
  std::string* why = nullptr;
  const mavg_config& cfg = c->cfg;
  const int L = cfg.n_layers, P = cfg.P, B = cfg.B;
  FacState* f = new FacState();
  f->lay = reb_layout(&cfg, st->lay.shared_end);
  f->K = reb_steps(&cfg);
  const FacLayout& t = f->lay;
  auto bf = [&](size_t off) { return (__nv_bfloat16*)ws_ptr(c, off); };
  bool ok = true;
  // rows [n, B, d], a row `pitch` long
  auto rows = [&](CUtensorMap* m, __nv_bfloat16* at, int d, int n, int box_rows, int box_learners = 1) {
    const int pitch = (int)up((size_t)d, 8);
    ok = ok && encode_map(st, m, at, d, B, n, pitch, (int64_t)B * pitch, box_rows, why, box_learners);
  };
  // Products of k_fac_product where it sums in the plain form's order: over the whole contraction, or over the runs of a
  // product that rides on a weight gradient there, and for a bias step over the whole batch; the others are the plain form's launches, whose data gradients read A_{l-1} transposed.
  // (3072-2048-2048-2048-10, P = 8, B = 64: data gradients of a step 50 us, 57 as the plain form's launches; 1080-576-576-32,
  // P = 26, B = 176 27 and 32.)
  for (int l = 2; l <= L; ++l) {
    const int m_tiles = (cfg.dims[l - 1] + kBM - 1) / kBM;
    f->dgrad1[l] = cols_for(P, B, m_tiles, c->sm_count);
    f->dgrad[l] = cols_for(P, B, m_tiles, c->sm_count, 1);
    f->own_dgrad[l] = st->dgrad[l].splits == 1 && f->dgrad1[l].c_tiles == 1 && f->dgrad[l].c_tiles == 1;
  }
  for (int l = 1; l < L; ++l) {
    const int m_tiles = (cfg.dims[l] + kBM - 1) / kBM;
    f->fwd1[l] = cols_for(P, B, m_tiles, c->sm_count);
    f->fwd[l] = cols_for(P, B, m_tiles, c->sm_count, 1);
    for (int first = 0; first < 2; ++first) {
      const FwdForm form = fwd_form(st, l, first);
      // the plain form's product rides on a launch, with sums over whole rows or, added up, over runs of them
      const bool rides = !first && l <= st->fuse_upto;
      if (rides && partial_sums(P, st->wgrad_f[l])) f->runs[l] = st->wgrad_f[l].n_chunks;
      f->own_fwd[first][l] = (rides || form == FwdForm::DENSE || (form == FwdForm::TILES && st->fwd[l].splits == 1)) &&
                             ((l + 1 == L && st->tail_ok) || f->own_dgrad[l + 1]);
      ok = ok && (!rides || (f->own_fwd[first][l] && f->runs[l] * f->fwd[l].cols <= 512));
    }
  }
  f->step_in.resize((size_t)f->K * (MAVG_MAX_LAYERS + 1));
  f->step_dz.resize(f->step_in.size());
  for (int l = 1; l <= L && ok; ++l) {
    const int in = cfg.dims[l - 1], out = cfg.dims[l];
    const int64_t size = (int64_t)in * out;
    rows(&f->h_mn[l - 1], bf(t.h[l - 1]), in, f->K * P, 64);
    rows(&f->g_mn[l], bf(t.g[l]), out, f->K * P, 64);
    ok = ok && encode_map(st, &f->w_own[l], bf(t.w_own[l]), in, out, P, in, size, kBM, why);
    ok = ok && encode_map(st, &f->w_own_mn[l], bf(t.w_own[l]), in, out, P, in, size, 64, why);
    ok = ok && encode_any(st, &f->w_own_st[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, bf(t.w_own[l]), in, out, P, in, size,
                          kWgradTileCols, kWgradTileRows, CU_TENSOR_MAP_SWIZZLE_64B, why);
    for (int k = 1; k <= f->K && ok; ++k) {
      const size_t at = (size_t)(k - 1) * (MAVG_MAX_LAYERS + 1) + l;
      __nv_bfloat16* a = bf(t.h[l - 1]) + (size_t)(k - 1) * P * B * in;
      const FwdForm form = l < L ? fwd_form(st, l, k == 1) : FwdForm::TILES;
      const FacCols &fc = k == 1 ? f->fwd1[l] : f->fwd[l], &dc = k == 1 ? f->dgrad1[l] : f->dgrad[l];
      if (l < L && f->own_fwd[k == 1][l]) rows(&f->step_in[at], a, in, P, fc.cols, fc.nl);
      else if (form == FwdForm::DENSE) ok = encode_map(st, &f->step_in[at], a, in, P * B, 1, in, (int64_t)P * B * in, kDenseCols, why);
      else rows(&f->step_in[at], a, in, P, form == FwdForm::SPLIT ? B : st->fwd[l].BN);
      __nv_bfloat16* dz = bf(t.g[l]) + (size_t)(k - 1) * P * B * up((size_t)out, 8);
      if (l > 1 && f->own_dgrad[l]) rows(&f->step_dz[at], dz, out, P, dc.cols, dc.nl);
      else if (l > 1) rows(&f->step_dz[at], dz, out, P, st->dgrad[l].BN);
    }
  }
  for (const void* k : {(const void*)k_fac_product<PROD_FWD, 1, false, false>, (const void*)k_fac_product<PROD_FWD_RUNS, 1, false, false>,
                        (const void*)k_fac_product<PROD_DGRAD_STEP, 1, false, false>})
    ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(kSmSharedBytes - kBlockReservedBytes - sizeof(GemmShared))) == cudaSuccess;
  for (const void* k : {(const void*)rebuild::k_rebuild<false, false>, (const void*)rebuild::k_rebuild<false, true>,
                        (const void*)rebuild::k_rebuild<true, false>, (const void*)rebuild::k_rebuild<true, true>})
    ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)(kSmSharedBytes - kBlockReservedBytes - sizeof(rebuild::Shared))) == cudaSuccess;
  if (ok) {
    st->reb = f;
  } else {
    cudaGetLastError();
    delete f;
  }
}

bool reb_usable(const mavg_ctx* c) {
  const TcState* st = (const TcState*)c->mlp;
  // by the momentum and K of now, which may not be those the handle was made with
  return st && st->reb && c->schedule == 0 && c->cfg.K <= st->reb->K && reb_steps(&c->cfg) == c->cfg.K &&
         (!st->fuse_upto || reb_riding(&c->cfg));
}

// The K steps of a round: F_1 -> ... -> F_{L-1} -> last layer and loss -> D_L -> ... -> D_2 -> weights of the next step's
// products (of the call's end: the learners' own, and u).  Every sum is formed in the plain form's order, so that the two
// give the same bits: another order moves operands across a bf16 rounding boundary, and after a few steps v is 1e-3 to
// 1e-2 off and single rows of u more than their size.
cudaError_t reb_local_steps(mavg_ctx* c, int64_t round) {
  TcState* st = (TcState*)c->mlp;
  FacState* f = st->reb;
  const FacLayout& t = f->lay;
  const mavg_config& cfg = c->cfg;
  const int L = cfg.n_layers, P = cfg.P, B = cfg.B, K = cfg.K;
  const MomArgs first = mom_args(c, true);
  cudaError_t e;
  FAC_TRY(gather_rows(c, t, K * B, round, false));
  for (int k = 1; k <= K; ++k) {
    MomArgs mom = first;
    if (k > 1 && mom.u) mom.read_u = 1;
    auto slab = [&](size_t at, int d) { return (__nv_bfloat16*)ws_ptr(c, at) + (size_t)(k - 1) * P * B * up((size_t)d, 8); };
    StepOperands o{};
    o.step = k;
    o.shared_w = k == 1;
    o.mom = mom;
    const CUtensorMap* in = &f->step_in[(size_t)(k - 1) * (MAVG_MAX_LAYERS + 1)];
    const CUtensorMap* dz = &f->step_dz[(size_t)(k - 1) * (MAVG_MAX_LAYERS + 1)];
    auto operands = [&](int l, const CUtensorMap* w, const CUtensorMap* x, size_t out, int out_layer, size_t out_t) {
      o.l = l;
      o.w = w;
      o.in = x;
      o.out_bm = slab(out, cfg.dims[out_layer]);
      o.out_mb = (__nv_bfloat16*)ws_ptr(c, out_t);
    };
    auto own = [&](const FacCols& cols, int contraction, int bias_layer) {
      ProdArgs g{};
      g.M = cfg.dims[bias_layer];
      g.kb = B;
      g.nl = cols.nl;
      g.cols = cols.cols;
      g.c_tiles = cols.c_tiles;
      g.nkb = (contraction + kBK - 1) / kBK;
      g.w_batched = k > 1;
      g.bias_off = c->layers[bias_layer - 1].b_off;
      g.bias_in = k == 1 ? c->buf.global_w : c->buf.replicas;
      g.bias_in_stride = k == 1 ? 0 : c->buf.replica_stride;
      g.mom = mom;
      g.out = o.out_bm;
      return g;
    };
    for (int l = 1; l < L; ++l) {
      operands(l, k == 1 ? &st->wg[l] : &f->w_own[l], in + l, t.h[l], l, t.act_t[l]);
      if (!f->own_fwd[k == 1][l]) {
        FAC_TRY(st->run_forward(c, o));
        continue;
      }
      ProdArgs g = own(k == 1 ? f->fwd1[l] : f->fwd[l], cfg.dims[l - 1], l);
      if (k > 1 && f->runs[l] > 1) {
        g.run = 2 * st->wgrad_f[l].chunk;            // (tiles of 32 columns)
        g.runs = f->runs[l];
        g.whole_rows = st->wgrad_f[l].whole_rows;
        FAC_TRY((launch_product<PROD_FWD_RUNS, 1>(c, MAVG_K_FWD, *o.w, *o.w, *o.in, f->g_mn[l], *o.in, g)));
      } else {
        FAC_TRY((launch_product<PROD_FWD, 1>(c, MAVG_K_FWD, *o.w, *o.w, *o.in, f->g_mn[l], *o.in, g)));
      }
    }
    operands(L, k == 1 ? &st->wg[L] : &f->w_own[L], in + L, t.g[L - 1], L - 1, t.dz_t);
    o.labels = (const int32_t*)ws_ptr(c, t.labels) + (size_t)(k - 1) * P * B;
    o.dz_bm = slab(t.g[L], cfg.dims[L]);
    o.a_bm = slab(t.h[L - 1], cfg.dims[L - 1]);
    o.w16 = k == 1 ? (const __nv_bfloat16*)ws_ptr(c, st->lay.w16g) + st->lay.sh_off[L - 1] : (const __nv_bfloat16*)ws_ptr(c, t.w_own[L]);
    o.w16_stride = k == 1 ? 0 : (int64_t)cfg.dims[L - 1] * cfg.dims[L];
    FAC_TRY(st->run_last_layer(c, o));
    for (int l = st->tail_ok ? L - 1 : L; l > 1; --l) {
      operands(l, k == 1 ? &st->wg_mn[l] : &f->w_own_mn[l], dz + l, t.g[l - 1], l - 1, t.dz_t);
      o.mask_mb = (const __nv_bfloat16*)ws_ptr(c, t.act_t[l - 1]);
      if (f->own_dgrad[l]) {
        ProdArgs g = own(k == 1 ? f->dgrad1[l] : f->dgrad[l], cfg.dims[l], l - 1);
        g.act = slab(t.h[l - 1], cfg.dims[l - 1]);
        FAC_TRY((launch_product<PROD_DGRAD_STEP, 1>(c, MAVG_K_DGRAD, *o.w, *o.w, *o.in, f->h_mn[l - 1], *o.in, g)));
      } else {
        FAC_TRY(st->run_dgrad(c, o));
      }
    }
    rebuild::Args g{};
    g.n_layers = L;
    g.P = P;
    g.group = std::min(P, 4);
    g.B = B;
    g.steps = k;
    g.load_u = first.u && first.read_u;
    g.gamma = cfg.local_lr;
    g.beta = first.beta;
    g.status = (int*)ws_ptr(c, c->ws.status);
    for (int l = 1; l <= L; ++l) {
      rebuild::Layer& a = g.layer[l - 1];
      a.m_tiles = (cfg.dims[l] + kBM - 1) / kBM;
      a.n_tiles = (cfg.dims[l - 1] + rebuild::kBN - 1) / rebuild::kBN;
      a.in = cfg.dims[l - 1];
      a.first = g.tiles;
      g.tiles += a.m_tiles * a.n_tiles;
      g.dz[l - 1] = f->g_mn[l];
      g.a[l - 1] = f->h_mn[l - 1];
      g.w_in[l - 1] = st->w32g[l];
      g.u[l - 1] = first.u ? st->u32[l] : st->w32g[l];
      g.out[l - 1] = k == K ? st->w32[l] : f->w_own_st[l];
    }
    const int units = (P + g.group - 1) / g.group * g.tiles;
    PdlLaunch l(dim3((unsigned)std::min(units, c->sm_count)), rebuild::kThreads, rebuild::launch_bytes(k == K), c->stream);
    auto kernel = k == K ? (first.u ? rebuild::k_rebuild<true, true> : rebuild::k_rebuild<false, true>)
                         : (first.u ? rebuild::k_rebuild<true, false> : rebuild::k_rebuild<false, false>);
    prof_begin(c, MAVG_K_WGRAD_SGD);
    e = cudaLaunchKernelEx(&l.lc, kernel, g);
    prof_end(c);
    FAC_TRY(e);
    FAC_TRY(cudaGetLastError());
  }
  return cudaSuccess;
}
#undef FAC_TRY

}  // namespace mavg
