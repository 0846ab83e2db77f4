// Matrix products of models whose widths, batch or arithmetic the bf16 path does not take (mlp_simt.cu), on
// tcgen05.  An fp32 operand is the sum of three bf16 numbers, x = x0 + x1 + x2 (NP = 3 planes), exactly from 2^-110
// up; of the nine products of two such sums the six largest are formed, x0 y0 in one accumulator and the other five in
// another, and what is left out, x1 y2 + x2 y1 + x2 y2, is at most about 2^-24 of |x| |y|.  With bf16 operands (NP = 1) there is one plane and one accumulator.
// The tensor cores cut a sum off where they add to it, always towards zero, so an accumulator takes one slab of 64
// contraction elements (of a weight gradient two or four); the epilogue warps then add it to fp32 registers, rounded to
// nearest, while the next goes into the other accumulator.  Against 64 bits: see mlp_simt.cu.
//
// Operands are kept as planes [NP][matrices, rows, pitch] (pitch: the width to a multiple of 8), which TMA reads in
// either orientation: minibatches, activations and dZ [NP][P], weights [NP][P + 1] with those of w~ as the last.
#pragma once
#include <cuda.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace mavg {
namespace split {

using namespace tc;

constexpr int kTile = 128;                        // MMA M
constexpr int kSlab = 64;                         // contraction elements of a stage: 128 bytes of bf16
constexpr int kTileBytes = kTile * kSlab * 2;
constexpr int kMaxN = 128;                        // columns: four accumulators fill the tensor memory
constexpr int kMaxStages = 6;
// Warp 0: TMA producer, 1: MMA issuer, then the epilogue; of a weight gradient two more for the biases and the loss.
constexpr int kProductEpi = 8, kProductThreads = (2 + kProductEpi) * 32;
// Slabs of a weight gradient in one accumulator, and how many accumulators a sum takes: one, two that the epilogue adds where
// it uses them, or kManyChains, added one after the other to registers.  fp32 with four slabs to an accumulator: a sum of
// 160 like terms was 1.32 times as far from 64 bits as a chain of FMAs (192: 1.35; two slabs: 1.02 and 0.96), gradients of
// 301-131-66-5 with inputs in [0, 1] at B = 256 up to 1.21 times (0.75).  3072-512-512-10, P = 4, K = 4 takes 408 us a round
// at B = 160 (four slabs 377; two with sums in registers 436), 475 at 256 (438, 489).  bf16 operands are what limits one
// plane: four slabs, whose sums the accumulator cuts off less often than the former warp-level MMAs theirs.
constexpr int chain_slabs(int np) { return np == 3 ? 2 : 4; }
constexpr int kManyChains = 0;
constexpr int wgrad_chains(int np, int B) {
  const int chain = chain_slabs(np) * kSlab;
  return B <= chain ? 1 : np == 3 && B <= 2 * chain ? 2 : kManyChains;
}
constexpr int wgrad_epi(int chains) { return chains == kManyChains ? 8 : 16; }
constexpr int wgrad_threads(int chains) { return (4 + wgrad_epi(chains)) * 32; }
enum { ERR_SPLIT_PRODUCER = 41, ERR_SPLIT_MMA = 42, ERR_SPLIT_EPILOGUE = 43 };

__host__ __device__ constexpr int pitch_of(int d) { return (d + 7) / 8 * 8; }

// Two neighbours as NP bf16 planes.  Round to nearest leaves at most half a unit to the next plane.  The first of three is
// the largest finite bf16 number where a finite value rounds beyond it (from 3.39e38 on), which leaves 16 bits to the other
// two; that of an infinite value is infinite and stands alone: what it leaves over would be NaN.
template <int NP>
__device__ __forceinline__ void split2(float a, float b, uint32_t (&pl)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    if (NP > 1 && i == 0) {
      asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(pl[i]) : "f"(b), "f"(a));
    } else {
      const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
      pl[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    if (i + 1 < NP) {
      a -= __uint_as_float(pl[i] << 16);
      b -= __uint_as_float(pl[i] & 0xffff0000u);
      if (i == 0) {                                // the next number up is the infinite one
        const bool ia = fabsf(a) == INFINITY, ib = fabsf(b) == INFINITY;
        if (ia) pl[i] += 1u;
        if (ib) pl[i] += 0x10000u;
        a = ia ? 0.f : a;
        b = ib ? 0.f : b;
      }
    }
  }
}
template <int NP>
__device__ __forceinline__ void split8(const float (&x)[8], uint4 (&pl)[NP]) {
  uint32_t w[4][NP];
#pragma unroll
  for (int i = 0; i < 4; ++i) split2<NP>(x[2 * i], x[2 * i + 1], w[i]);
#pragma unroll
  for (int i = 0; i < NP; ++i) pl[i] = make_uint4(w[0][i], w[1][i], w[2][i], w[3][i]);
}
__device__ __forceinline__ void put16(__nv_bfloat16* p, uint32_t bits) { *reinterpret_cast<unsigned short*>(p) = (unsigned short)bits; }
// One value to element `at` of each plane.
template <int NP>
__device__ __forceinline__ void put_planes(__nv_bfloat16* p, int64_t plane, size_t at, float v) {
  uint32_t pl[NP];
  split2<NP>(v, 0.f, pl);
#pragma unroll
  for (int i = 0; i < NP; ++i) put16(p + i * plane + at, pl[i]);
}

// The MMAs of nk groups of 16 contraction elements: the leading planes' product into d, the others into lo, from zero
// where `first`, `first_low`.
template <int NP>
__device__ __forceinline__ void slab_mmas(uint32_t d, uint32_t lo, uint64_t a, uint32_t a_plane, uint32_t a_step, uint64_t b,
                                          uint32_t b_plane, uint32_t b_step, uint32_t idesc, bool first, bool first_low, int nk) {
#pragma unroll 1
  for (int k = 0; k < nk; ++k, a += a_step, b += b_step) {
    umma_bf16(d, a, b, idesc, !first || k > 0);
    if (NP == 3) {
      umma_bf16(lo, a + 2 * a_plane, b, idesc, !first_low || k > 0);
      umma_bf16(lo, a, b + 2 * b_plane, idesc, 1u);
      umma_bf16(lo, a + a_plane, b + b_plane, idesc, 1u);
      umma_bf16(lo, a + a_plane, b, idesc, 1u);
      umma_bf16(lo, a, b + b_plane, idesc, 1u);
    }
  }
}

struct alignas(16) Barriers {                    // (whole 16 bytes, as static shared memory is counted)
  uint64_t full[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2];
  uint32_t tmem_slot;
  int abort_flag;
};
__device__ __forceinline__ void init_barriers(Barriers& sh, int stages, int epilogue_warps) {
  for (int s = 0; s < stages; ++s) {
    mbar_init(&sh.full[s], 1);
    mbar_init(&sh.empty[s], 1);
  }
  for (int b = 0; b < 2; ++b) {
    mbar_init(&sh.acc_full[b], 1);
    mbar_init(&sh.acc_empty[b], epilogue_warps);
  }
  sh.abort_flag = 0;
  fence_barrier_init();
  fence_proxy_async();
}
// This thread's sums: tensor-memory lane 32 (warp % 4) + lane, 16 of every STEP columns.
template <int STEP>
struct Sums {
  float v[kMaxN / STEP * 16];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < kMaxN / STEP * 16; ++i) v[i] = 0.f;
  }
  // Adds an accumulator, of which this thread has columns c, c + STEP, ...  LAST: that of the smaller products, after
  // which the sums are whole; an infinite leading sum stands alone (the others may be infinite the other way).
  template <bool LAST>
  __device__ __forceinline__ void drain(uint32_t lane_addr, int c, int N) {
#pragma unroll
    for (int g = 0; g < kMaxN / STEP; ++g) {
      if (c + STEP * g < N) {
        uint32_t z[16];
        tmem_ld_16cols(lane_addr + (uint32_t)(c + STEP * g), z);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float& x = v[16 * g + j];
          x = LAST && !(fabsf(x) <= 3.402823466e38f) ? x : x + __uint_as_float(z[j]);
        }
      }
    }
  }
};

// ------------------------------------------------------------- forward products and data gradients
struct ProductArgs {
  int M, K, B, P, N;                              // N: batch rows of a tile
  int w_first, w_step, w_plane;                   // matrix of learner p, plane q: w_first + w_step p + w_plane q
  int m_tiles, n_tiles, splits, per_split;        // per_split: slabs of a block
  int stages; uint32_t tmem_cols;
  __nv_bfloat16* out; int64_t plane;              // planes [P, B, pitch], or null
  float* out_f; int pitch;                        // fp32 [P, B, M], or null
  const float* bias; int64_t bias_batch;          // forward
  const __nv_bfloat16* act;                       // data gradient: leading plane of the activations that gate it
  int hidden;                                     // forward: ReLU (and the operand rounding of the next products)
  int* status;
};
__host__ __device__ constexpr int product_stage_bytes(int np, int N) { return np * (kTileBytes + N * kSlab * 2); }

// One tile of 128 features x N batch rows.  A cluster of `splits` blocks shares the tile, each a range of the
// contraction; every block sends its sums to the blocks that finish them, each a share of the columns, and those add
// them in rank order.  DGRAD: W is read MN-major.
// Bound by what an SM takes in (90 KB a slab at 112 batch rows and three planes, about 50 GB/s an SM) and, while slabs are
// few, by latency: 3072-512, P = 4, B = 100 22 us of 8 slabs a block, 512-512 12.  The sums are sent in whole groups of 16
// columns and finished four features to a thread: element by element the epilogue's instructions took longer than the
// products (30 and 22 us).  Weights split by the blocks that read them, eight warps of loads and conversions in place of
// copies of the planes: 40 and 16.
template <int NP, bool DGRAD>
__global__ void __launch_bounds__(kProductThreads, 1)
k_split_product(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ ProductArgs g) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(16) Barriers sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N = g.N, stages = g.stages, stage_bytes = product_stage_bytes(NP, N);
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tm_w);
    tma_prefetch_desc(&tm_x);
    init_barriers(sh, stages, kProductEpi);
  }
  uint32_t* tmem_slot = &sh.tmem_slot;
  if (warp == 1) {
    tmem_alloc(tmem_slot, g.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = sh.tmem_slot;
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();
  const int rank = (int)blockIdx.x % g.splits, tile = (int)blockIdx.x / g.splits;
  const int m0 = tile % g.m_tiles * kTile, n0 = tile / g.m_tiles * N, p = (int)blockIdx.z;
  const int slab0 = rank * g.per_split, slabs = (g.K + kSlab - 1) / kSlab, ns = min(g.per_split, slabs - slab0);
  const int cols = min(N, g.B - n0), share = (N / 16 + g.splits - 1) / g.splits;   // groups of 16 columns a block finishes
  volatile int* abortp = &sh.abort_flag;
  float* recv = reinterpret_cast<float*>(smem);   // [splits][16 share][128] sums, once the operands have been read
  Sums<32> sums;
  bool ok = true;

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      for (int i = 0; i < ns; ++i, ++issued) {
        const int s = i % stages, k0 = (slab0 + i) * kSlab;
        if (!mbar_wait(&sh.empty[s], ((i / stages) & 1) ^ 1, abortp, g.status, ERR_SPLIT_PRODUCER)) break;
        uint8_t* sa = smem + (size_t)s * stage_bytes;
        mbar_arrive_expect_tx(&sh.full[s], (uint32_t)stage_bytes);
        for (int q = 0; q < NP; ++q) {
          const int w = g.w_first + g.w_step * p + g.w_plane * q;
          if (DGRAD) {
            tma_load_3d(sa + q * kTileBytes, &tm_w, &sh.full[s], m0, k0, w);
            tma_load_3d(sa + q * kTileBytes + kTileBytes / 2, &tm_w, &sh.full[s], m0 + 64, k0, w);
          } else {
            tma_load_3d(sa + q * kTileBytes, &tm_w, &sh.full[s], k0, m0, w);
          }
          tma_load_3d(sa + NP * kTileBytes + (size_t)q * N * kSlab * 2, &tm_x, &sh.full[s], k0, n0, q * g.P + p);
        }
      }
      if (*abortp) drain_copies(sh.full, issued, stages, g.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_f32(kTile, N, DGRAD ? 1 : 0), base = smem_u32(smem);
      const uint64_t a0 = DGRAD ? smem_desc_mn_sw128(base) : smem_desc_k_sw128(base);
      const uint64_t b0 = smem_desc_k_sw128(base + NP * kTileBytes);
      for (int i = 0; i < ns; ++i) {
        const int s = i % stages, b = i & 1;
        if (!mbar_wait(&sh.acc_empty[b], ((i >> 1) & 1) ^ 1, abortp, g.status, ERR_SPLIT_MMA)) break;
        if (!mbar_wait(&sh.full[s], (i / stages) & 1, abortp, g.status, ERR_SPLIT_MMA)) break;
        tc_fence_after_sync();
        const uint32_t off = (uint32_t)(s * stage_bytes) >> 4;
        const int nk = min(kSlab, g.K - (slab0 + i) * kSlab + 15) / 16;
        slab_mmas<NP>(tmem_base + (uint32_t)(b * N), tmem_base + (uint32_t)(2 * N), a0 + off, kTileBytes >> 4,
                      DGRAD ? (16 * 128) >> 4 : 2, b0 + off, (uint32_t)(N * kSlab * 2) >> 4, 2, idesc, true, i == 0, nk);
        umma_commit(&sh.empty[s]);
        umma_commit(&sh.acc_full[b]);
      }
    }
    __syncwarp();
  } else {
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    sums.clear();
    for (int i = 0; i < ns; ++i) {
      const int b = i & 1;
      if (!(ok = mbar_wait_warp(&sh.acc_full[b], (i >> 1) & 1, abortp, g.status, ERR_SPLIT_EPILOGUE))) break;
      tc_fence_after_sync();
      const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
      sums.drain<false>(lane_addr + (uint32_t)(b * N), 16 * half, N);
      if (NP == 3 && i + 1 == ns) sums.drain<true>(lane_addr + (uint32_t)(2 * N), 16 * half, N);
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.acc_empty[b]);
    }
  }
  // features 4 lane .. of this thread when the tile is finished
  const int m = m0 + 4 * lane;
  float bias[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) bias[j] = !DGRAD && m + j < g.M ? g.bias[(size_t)p * g.bias_batch + m + j] : 0.f;
  // the sums go where the operands were, in every block: none may still be multiplying
  __syncthreads();
  if (g.splits > 1) cluster_sync_all();
  if (warp >= 2 && ok) {
    const int row = (warp & 3) * 32 + lane, half = (warp - 2) >> 2;
    const uint32_t at = smem_u32(recv + rank * share * 16 * kTile + row);
#pragma unroll
    for (int gr = 0; gr < kMaxN / 32; ++gr) {
      const int c = 2 * gr + half;               // group of 16 columns
      if (16 * c < cols) {
        const int to = c / share;
        uint32_t dst = at + (uint32_t)((c - to * share) * 16 * kTile * 4);
        if (g.splits > 1) dst = mapa_u32(dst, (uint32_t)to);
#pragma unroll
        for (int j = 0; j < 16; ++j) st_cluster_u32(dst + (uint32_t)(j * kTile * 4), __float_as_uint(sums.v[16 * gr + j]));
      }
    }
  }
  __syncthreads();
  if (g.splits > 1) cluster_sync_all();

  // finish this block's share of the columns, a warp per column
  const int first = rank * share * 16, mine = min(cols - first, share * 16);
  if (m < g.pitch)
#pragma unroll 1
    for (int c = warp; c < mine; c += kProductThreads / 32) {
      float4 z = *reinterpret_cast<const float4*>(recv + c * kTile + 4 * lane);
      for (int r = 1; r < g.splits; ++r) {
        const float4 y = *reinterpret_cast<const float4*>(recv + (r * share * 16 + c) * kTile + 4 * lane);
        z.x += y.x; z.y += y.y; z.z += y.z; z.w += y.w;
      }
      const size_t row = (size_t)p * g.B + n0 + first + c;
      if (DGRAD) {
        const uint2 a = *reinterpret_cast<const uint2*>(g.act + row * g.pitch + m);      // positive: neither sign nor zero
        z.x = (a.x & 0xffff) - 1 < 0x7fff ? z.x : 0.f;
        z.y = (a.x >> 16) - 1 < 0x7fff ? z.y : 0.f;
        z.z = (a.y & 0xffff) - 1 < 0x7fff ? z.z : 0.f;
        z.w = (a.y >> 16) - 1 < 0x7fff ? z.w : 0.f;
      } else {
        z.x += bias[0]; z.y += bias[1]; z.z += bias[2]; z.w += bias[3];
        if (g.hidden) z = make_float4(z.x > 0.f ? z.x : 0.f, z.y > 0.f ? z.y : 0.f, z.z > 0.f ? z.z : 0.f, z.w > 0.f ? z.w : 0.f);
      }
      if (g.out) {
        uint32_t lo[NP], hi[NP];
        split2<NP>(z.x, z.y, lo);
        split2<NP>(z.z, z.w, hi);
#pragma unroll
        for (int q = 0; q < NP; ++q) *reinterpret_cast<uint2*>(g.out + q * g.plane + row * g.pitch + m) = make_uint2(lo[q], hi[q]);
      }
      if (g.out_f) {
        float* f = g.out_f + row * g.M + m;
        if (m < g.M) f[0] = z.x;
        if (m + 1 < g.M) f[1] = z.y;
        if (m + 2 < g.M) f[2] = z.z;
        if (m + 3 < g.M) f[3] = z.w;
      }
    }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, g.tmem_cols);
}

// ------------------------------------------------------------------- weight gradients and SGD steps
struct WgradLayer {
  int in, out, i_tiles, o_tiles, first;           // first: tiles of the layers before, over all learners
  int pairs;                                      // rows of W have even length and start on 8 bytes
  int64_t w_off, b_off;
  const float* dz;                                // fp32 [P, B, out]
  __nv_bfloat16* w16; int64_t w16_batch, w16_plane;   // planes of the weights after the step, rows of pitch_of(in); null: no product reads them
};
struct WgradArgs {
  CUtensorMap a[MAVG_MAX_LAYERS], dz[MAVG_MAX_LAYERS];   // planes, read MN-major: boxes of 64 columns x 64 samples
  WgradLayer layer[MAVG_MAX_LAYERS];
  int L, tiles, P, B, stages;
  int bn;                                         // outputs of a tile: 128 or 64
  int write_planes;                               // not in a call's last step
  const float* w_in; int64_t w_in_batch;          // the models before the step
  float* rep; int64_t rep_stride;
  MomArgs mom;
  float gamma;
  const float* row_loss;                          // [P, B]
  float* loss_out; int loss_stride;
  int* status;
};
__host__ __device__ constexpr int wgrad_stage_bytes(int np) { return np * 2 * kTileBytes; }

// 16 columns of a thread's part of a tile, in pairs.  PAIRS (rows of even length that start on 8 bytes): two neighbours
// of a row, for which the lanes 2 k and 2 k + 1 exchange half of their sums; else two rows' elements of the thread's own
// input.
struct Place { int i, c, in, outs; };             // input, first column, row length, columns that exist
struct Weights {
  float2 v[8];
  template <bool PAIRS>
  __device__ __forceinline__ static int64_t offset(const Place& at) {   // of the first pair; the others two rows apart
    const int odd = at.i & 1;
    return (int64_t)(at.c + (PAIRS ? odd : 0)) * at.in + (PAIRS ? at.i - odd : at.i);
  }
  // whether the pair's elements exist
  template <bool PAIRS>
  __device__ __forceinline__ static int count(const Place& at, int j) {
    const int c = at.c + 2 * j + (PAIRS ? at.i & 1 : 0);
    if (at.i >= at.in) return 0;
    return PAIRS ? (c < at.outs ? 2 : 0) : min(2, max(0, at.outs - c));
  }
  template <bool PAIRS>
  __device__ __forceinline__ static float2 load(const float* p, int n, int in) {
    float2 r = make_float2(0.f, 0.f);
    if (PAIRS) {
      if (n) r = *reinterpret_cast<const float2*>(p);
    } else {
      if (n > 0) r.x = p[0];
      if (n > 1) r.y = p[in];
    }
    return r;
  }
  template <bool PAIRS>
  __device__ __forceinline__ static void store(float* p, int n, int in, float2 x) {
    if (PAIRS) {
      if (n) *reinterpret_cast<float2*>(p) = x;
    } else {
      if (n > 0) p[0] = x.x;
      if (n > 1) p[in] = x.y;
    }
  }
  template <bool PAIRS>
  __device__ __forceinline__ void fetch(const float* src, const Place& at) {
    src += offset<PAIRS>(at);
#pragma unroll
    for (int j = 0; j < 8; ++j, src += 2 * at.in) v[j] = load<PAIRS>(src, count<PAIRS>(at, j), at.in);
  }
  template <int NP, bool MOM, bool PAIRS>
  __device__ __forceinline__ void step(const float (&z)[16], const Place& at, float gamma, const MomArgs& mom, float* dst,
                                       float* u, __nv_bfloat16* w16, int64_t plane, int pitch) {
    const int64_t first = offset<PAIRS>(at);
    dst += first;
    if (MOM) u += first;
    if (w16) w16 += offset<PAIRS>(Place{at.i, at.c, pitch, at.outs});
#pragma unroll
    for (int j = 0; j < 8; ++j, dst += 2 * at.in) {
      float2 d = make_float2(z[2 * j], z[2 * j + 1]), x = v[j];
      if (PAIRS) {
        const bool odd = at.i & 1;
        const float got = __shfl_xor_sync(0xffffffffu, odd ? d.x : d.y, 1);
        d = odd ? make_float2(got, d.y) : make_float2(d.x, got);
      }
      const int n = count<PAIRS>(at, j);
      if (MOM) {
        float2 m = mom.read_u ? load<PAIRS>(u, n, at.in) : make_float2(0.f, 0.f);
        msgd(x.x, m.x, d.x, gamma, mom.beta);
        msgd(x.y, m.y, d.y, gamma, mom.beta);
        store<PAIRS>(u, n, at.in, m);
        u += 2 * at.in;
      } else {
        x = make_float2(fmaf(-gamma, d.x, x.x), fmaf(-gamma, d.y, x.y));
      }
      store<PAIRS>(dst, n, at.in, x);
      if (w16) {
        uint32_t pl[NP];
        split2<NP>(x.x, x.y, pl);
        __nv_bfloat16* q = w16;
        w16 += 2 * pitch;
#pragma unroll
        for (int r = 0; r < NP; ++r, q += plane) {
          if (PAIRS) {
            if (n) *reinterpret_cast<uint32_t*>(q) = pl[r];
          } else {
            if (n > 0) put16(q, pl[r]);
            if (n > 1) put16(q + pitch, pl[r] >> 16);
          }
        }
      }
    }
  }
};

// Weight gradients, SGD steps, bias steps of all layers and the losses: persistent over tiles of 128 inputs x 128
// outputs, dW^T = A^T dZ, so that the lanes of a warp finish neighbours of a row of W.  A tile's weights are fetched
// while the tile before it is finished.  CHAINS: see wgrad_chains; without sums in registers there is room for twice the warps.
// Bound by what an SM takes in (three planes: 154 KB a tile at B = 100) and by the epilogue's stores: 3072-512-512-10,
// P = 4, B = 100 32 us, 24 in a call's last step, which writes no planes.  On the way: eight warps with sums in registers 46,
// biases summed by the epilogue 40, weights fetched at the tile's own beginning 44, a word at a time 46.
template <int NP, bool MOM, int CHAINS>
__global__ void __launch_bounds__(wgrad_threads(CHAINS), 1)
k_split_wgrad(const __grid_constant__ WgradArgs g) {
  constexpr bool MANY = CHAINS == kManyChains;
  constexpr int kChainSlabs = chain_slabs(NP);
  constexpr int kEpi = wgrad_epi(CHAINS), kStep = MANY ? 32 : 64, kGroups = kMaxN / kStep;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(16) Barriers sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int stages = g.stages;
  constexpr int kStageBytes = wgrad_stage_bytes(NP);
  if (threadIdx.x == 0) init_barriers(sh, stages, kEpi);
  uint32_t* tmem_slot = &sh.tmem_slot;
  if (warp == 1) {
    tmem_alloc(tmem_slot, NP == 3 ? 512 : 256);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = sh.tmem_slot;
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();
  volatile int* abortp = &sh.abort_flag;
  const int slabs = (g.B + kSlab - 1) / kSlab;
  auto decode = [&](int t, int& l, int& p, int& i0, int& o0) {
    l = 0;
    while (l + 1 < g.L && t >= g.layer[l + 1].first) ++l;
    const WgradLayer& ly = g.layer[l];
    t -= ly.first;
    const int per = ly.i_tiles * ly.o_tiles;
    p = t / per;
    t -= p * per;
    i0 = t / ly.o_tiles * kTile;
    o0 = t % ly.o_tiles * g.bn;
  };
  auto columns = [&](int l, int o0) { return g.bn > 64 && g.layer[l].out - o0 > 64 ? 128 : 64; };   // whole groups of 64, see smem_desc_mn_sw128
  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
        int l, p, i0, o0;
        decode(t, l, p, i0, o0);
        const int boxes = 2 + columns(l, o0) / 64;
        for (int i = 0; i < slabs; ++i, ++issued) {
          const int s = issued % stages;
          if (!(ok = mbar_wait(&sh.empty[s], ((issued / stages) & 1) ^ 1, abortp, g.status, ERR_SPLIT_PRODUCER))) break;
          uint8_t* sa = smem + (size_t)s * kStageBytes;
          mbar_arrive_expect_tx(&sh.full[s], (uint32_t)(NP * boxes * 8192));
          for (int q = 0; q < NP; ++q) {
            for (int h = 0; h < 2; ++h)
              tma_load_3d(sa + q * kTileBytes + h * 8192, &g.a[l], &sh.full[s], i0 + 64 * h, i * kSlab, q * g.P + p);
            for (int h = 0; h < boxes - 2; ++h)
              tma_load_3d(sa + (NP + q) * kTileBytes + h * 8192, &g.dz[l], &sh.full[s], o0 + 64 * h, i * kSlab, q * g.P + p);
          }
        }
      }
      if (*abortp) drain_copies(sh.full, issued, stages, g.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t base = smem_u32(smem);
      const uint64_t a0 = smem_desc_mn_sw128(base), b0 = smem_desc_mn_sw128(base + NP * kTileBytes);
      int it = 0, chain = 0, tile = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < g.tiles && ok; t += gridDim.x, ++tile) {
        int l, p, i0, o0;
        decode(t, l, p, i0, o0);
        const int N = columns(l, o0);
        const uint32_t idesc = idesc_bf16_f32(kTile, N, 1, 1);
        for (int i = 0; i < slabs; ++i, ++it) {
          const int s = it % stages, b = chain & 1;
          if (i % kChainSlabs == 0 && !(ok = mbar_wait(&sh.acc_empty[b], ((chain >> 1) & 1) ^ 1, abortp, g.status, ERR_SPLIT_MMA))) break;
          if (!(ok = mbar_wait(&sh.full[s], (it / stages) & 1, abortp, g.status, ERR_SPLIT_MMA))) break;
          tc_fence_after_sync();
          const uint32_t off = (uint32_t)(s * kStageBytes) >> 4;
          slab_mmas<NP>(tmem_base + (uint32_t)(b * kMaxN), tmem_base + (uint32_t)((2 + (tile & 1)) * kMaxN), a0 + off, kTileBytes >> 4,
                        (16 * 128) >> 4, b0 + off, kTileBytes >> 4, (16 * 128) >> 4, idesc, i % kChainSlabs == 0, i == 0,
                        min(kSlab, g.B - i * kSlab + 15) / 16);
          umma_commit(&sh.empty[s]);
          if (i % kChainSlabs == kChainSlabs - 1 || i + 1 == slabs) {
            umma_commit(&sh.acc_full[b]);
            ++chain;
          }
        }
      }
    }
    __syncwarp();
  } else if (warp >= 2 + kEpi) {
    // The bias steps of the first column of tiles (unrounded dZ), half of a tile's outputs each, and
    // the losses: beside the epilogue, whose tiles would wait for them.
    const int half = warp - 2 - kEpi;
    for (int t = blockIdx.x; t < g.tiles; t += gridDim.x) {
      int l, p, i0, o0;
      decode(t, l, p, i0, o0);
      if (i0 > 0) continue;
      const WgradLayer& ly = g.layer[l];
      const int n = min(g.bn, ly.out - o0) - 64 * half;
      const float* d = ly.dz + (size_t)p * g.B * ly.out + o0 + 64 * half + lane;
      float s[2][4] = {};                           // every fourth sample's, added in pairs
      for (int b0 = 0; b0 < g.B; b0 += 16) {
        float v[2][16];
#pragma unroll
        for (int b = 0; b < 16; ++b, d += ly.out) {
          v[0][b] = b0 + b < g.B && lane < n ? d[0] : 0.f;
          v[1][b] = b0 + b < g.B && lane + 32 < n ? d[32] : 0.f;
        }
#pragma unroll
        for (int b = 0; b < 16; ++b) {
          s[0][b & 3] += v[0][b];
          s[1][b & 3] += v[1][b];
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (lane + 32 * k < n) {
          const size_t at = (size_t)ly.b_off + o0 + 64 * half + lane + 32 * k;
          local_update(g.rep + (size_t)p * g.rep_stride + at, g.w_in[(size_t)p * g.w_in_batch + at],
                       MOM ? g.mom.u + (size_t)p * g.mom.u_stride + at : nullptr, g.mom.read_u, (s[k][0] + s[k][1]) + (s[k][2] + s[k][3]), g.gamma, g.mom.beta);
        }
      if (l == 0 && o0 == 0 && half == 1) {
        float sum = 0.f;
        for (int b = lane; b < g.B; b += 32) sum += g.row_loss[(size_t)p * g.B + b];
        for (int q = 16; q > 0; q >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, q);
        if (lane == 0) g.loss_out[(size_t)p * g.loss_stride] = sum / (float)g.B;
      }
      __syncwarp();
    }
  } else {
    const int q4 = warp & 3;
    const uint32_t lane_addr = tmem_base + ((uint32_t)(q4 * 32) << 16);
    struct Tile { int l, p, i0, o0; };
    auto tile_at = [&](int t) {
      Tile x{0, 0, 0, 0};
      if (t < g.tiles) decode(t, x.l, x.p, x.i0, x.o0);
      return x;
    };
    auto place = [&](const Tile& x, int gr) {
      return Place{x.i0 + q4 * 32 + lane, kStep * gr + 16 * ((warp - 2) >> 2), g.layer[x.l].in, min(g.bn, g.layer[x.l].out - x.o0)};
    };
    auto w_place = [&](const Tile& x) { return (size_t)g.layer[x.l].w_off + (size_t)x.o0 * g.layer[x.l].in; };
    Weights w[2];
    auto fetch = [&](const Tile& x, int gr) {
      const float* src = g.w_in + (size_t)x.p * g.w_in_batch + w_place(x);
      if (g.layer[x.l].pairs) w[gr & 1].fetch<true>(src, place(x, gr));
      else w[gr & 1].fetch<false>(src, place(x, gr));
    };
    int chain = 0, tile = 0;
    bool ok = true;
    Tile next = tile_at(blockIdx.x);
    fetch(next, 0);
    fetch(next, 1);
#pragma unroll 1
    for (int t = blockIdx.x; t < g.tiles; t += gridDim.x, ++tile) {
      const Tile x = next;
      next = tile_at(t + gridDim.x);
      const int l = x.l, p = x.p, o0 = x.o0;
      const WgradLayer& ly = g.layer[l];
      const int N = columns(l, o0);
      const size_t w_at = w_place(x);
      const uint32_t low = lane_addr + (uint32_t)((2 + (tile & 1)) * kMaxN);
      const int c = 16 * ((warp - 2) >> 2);
      Sums<kStep> sums;                            // (not MANY: unused)
      int b = CHAINS == 2 ? 0 : chain & 1;
      if (MANY) {
        sums.clear();
        for (int s = 0; s < slabs; s += kChainSlabs, ++chain) {
          b = chain & 1;
          if (!(ok = mbar_wait_warp(&sh.acc_full[b], (chain >> 1) & 1, abortp, g.status, ERR_SPLIT_EPILOGUE))) break;
          tc_fence_after_sync();
          sums.template drain<false>(lane_addr + (uint32_t)(b * kMaxN), c, N);
          if (NP == 3 && s + kChainSlabs >= slabs) sums.template drain<true>(low, c, N);
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.acc_empty[b]);
        }
      } else {
        ok = mbar_wait_warp(&sh.acc_full[b], (chain >> 1) & 1, abortp, g.status, ERR_SPLIT_EPILOGUE);
        if (CHAINS == 2 && ok) ok = mbar_wait_warp(&sh.acc_full[1], (chain >> 1) & 1, abortp, g.status, ERR_SPLIT_EPILOGUE);
        tc_fence_after_sync();
        chain += CHAINS;
      }
      if (barrier_any(!ok, 1, kEpi * 32)) break;   // a wait that was given up: all leave together
      const int pitch = pitch_of(ly.in);
      float* dst = g.rep + (size_t)p * g.rep_stride + w_at;
      float* u = MOM ? g.mom.u + (size_t)p * g.mom.u_stride + w_at : nullptr;
      __nv_bfloat16* w16 = g.write_planes && ly.w16 ? ly.w16 + (size_t)p * ly.w16_batch + (size_t)o0 * pitch : nullptr;
#pragma unroll
      for (int gr = 0; gr < kGroups; ++gr) {
        if (c + kStep * gr < N) {
          float z[16];
          if (MANY) {
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = sums.v[16 * gr + j];
          } else {
            uint32_t r[16], rl[16];
            tmem_ld_16cols(lane_addr + (uint32_t)(b * kMaxN + c + kStep * gr), r);
            if (CHAINS == 2) {                     // (both accumulators are this tile's)
              tmem_ld_16cols(lane_addr + (uint32_t)(kMaxN + c + kStep * gr), rl);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(rl[j]));
            }
            if (NP == 3) tmem_ld_16cols(low + (uint32_t)(c + kStep * gr), rl);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const float h = __uint_as_float(r[j]);
              z[j] = NP == 3 && fabsf(h) <= 3.402823466e38f ? h + __uint_as_float(rl[j]) : h;
            }
          }
          if (ly.pairs) w[gr & 1].step<NP, MOM, true>(z, place(x, gr), g.gamma, g.mom, dst, u, w16, ly.w16_plane, pitch);
          else w[gr & 1].step<NP, MOM, false>(z, place(x, gr), g.gamma, g.mom, dst, u, w16, ly.w16_plane, pitch);
        }
        if (gr + 2 < kGroups) fetch(x, gr + 2);
        else fetch(next, gr + 2 - kGroups);
      }
      if (!MANY) {
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.acc_empty[b]);
        if (CHAINS == 2 && lane == 0) mbar_arrive(&sh.acc_empty[1]);
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, NP == 3 ? 512 : 256);
}

// What a launch asks of an SM.
constexpr size_t kSmem = kSmSharedBytes - kBlockReservedBytes - sizeof(Barriers);
struct LaunchShape { int stages; uint32_t tmem_cols; size_t smem; };
inline LaunchShape launch_shape(int stage_bytes, uint32_t tmem_cols, size_t least) {
  LaunchShape s{std::min(kMaxStages, (int)((kSmem - 1024) / stage_bytes)), tmem_cols, 0};
  s.smem = std::max({(size_t)s.stages * stage_bytes + 1024, least, tmem_share_bytes(tmem_cols, sizeof(Barriers))});
  return s;
}
inline LaunchShape product_shape(int np, int N) {
  uint32_t cols = 32;
  while ((int)cols < (np == 3 ? 3 : 2) * N) cols <<= 1;
  return launch_shape(product_stage_bytes(np, N), cols, (size_t)(N / 16 + 7) * 16 * kTile * 4 + 1024);   // the sums a block receives
}
inline LaunchShape wgrad_shape(int np) { return launch_shape(wgrad_stage_bytes(np), np == 3 ? 512 : 256, 0); }

// The weights that a call's first step finds, as planes: a warp per row of a matrix.
struct SplitWeights {
  const float* src[MAVG_MAX_LAYERS];
  __nv_bfloat16* dst[MAVG_MAX_LAYERS];
  int64_t dst_batch[MAVG_MAX_LAYERS], dst_plane[MAVG_MAX_LAYERS];
  int in[MAVG_MAX_LAYERS], first[MAVG_MAX_LAYERS + 1];   // first: rows of the layers before
  int L, copies;                                  // learners (1: w~)
  int64_t src_batch;
};
template <int NP>
__device__ __forceinline__ void split_weight_row(const SplitWeights& g, int row) {
  const int lane = threadIdx.x & 31, p = row / g.first[g.L];
  int r = row - p * g.first[g.L], l = 0;
  while (l + 1 < g.L && r >= g.first[l + 1]) ++l;
  r -= g.first[l];
  const int in = g.in[l], pitch = pitch_of(in);
  const float* src = g.src[l] + (size_t)p * g.src_batch + (size_t)r * in;
  __nv_bfloat16* dst = g.dst[l] + (size_t)p * g.dst_batch[l] + (size_t)r * pitch;
  for (int c0 = 2 * lane; c0 < in; c0 += 8 * 64) {
    float x[8][2];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int k = 0; k < 2; ++k) x[u][k] = c0 + 64 * u + k < in ? src[c0 + 64 * u + k] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (c0 + 64 * u >= in) break;
      uint32_t pl[NP];
      split2<NP>(x[u][0], x[u][1], pl);
#pragma unroll
      for (int q = 0; q < NP; ++q) *reinterpret_cast<uint32_t*>(dst + q * g.dst_plane[l] + c0 + 64 * u) = pl[q];
    }
  }
}

}  // namespace split
}  // namespace mavg
