// Tensor-core MLP learner step: the three matrix products of every layer run on tcgen05 with
// TMA-fed shared-memory operands and the accumulator in tensor memory.  This file holds the
// forward and dgrad kernel and the schedule of a step; the weight-gradient kernel, which carries
// the SGD step, is in wgrad_tc.cu.
//
// Every product is arranged so that the 128-row MMA dimension is a feature dimension and the
// batch (16..256 rows) is the MMA's N or K:
//   forward   Z^T[out, B]  = W[out, in]    . A[B, in]^T        contraction over in
//   dgrad     dA^T[in, B]  = W^T[in, out]  . dZ[B, out]^T      contraction over out (W^T = W read MN-major)
//   wgrad     dW[out, in]  = dZ^T[out, B]  . A^T[in, B]^T      contraction over the batch
// Activations and dZ are kept in both orientations ([B, f] and [f, B]; the producing epilogues
// write both) so that they are K-major wherever they are an operand.  The weights have one bf16
// copy, [out, in]: forward reads it K-major, dgrad reads the same tiles MN-major.  fp32 master
// weights take the SGD step of Algorithm 1 in the wgrad kernel, which also refreshes the bf16
// copy.
// When a layer has too few output tiles to fill the GPU, forward and dgrad split the contraction
// over several blocks; each writes an fp32 partial tile and the block that finishes last adds
// the partials in ascending split order (so the result does not depend on which block that is).
// That block -- or the only block, when there is no split -- applies the layer's tail in the
// same kernel: bias + ReLU, or the ReLU mask with the bias step of the layer below, or for the
// last layer the softmax cross-entropy loss, dZ_L and the last bias step.
#include <cuda.h>

#include <algorithm>

#include "factored.cuh"
#include "gemm_unit.cuh"
#include "mlp.cuh"
#include "tc_ptx.cuh"
#include "tc_state.cuh"
#include "wgrad_tc.cuh"

namespace mavg {
namespace {

using namespace tc;

constexpr int kThreads = 320;   // warp 0: TMA producer, warp 1: MMA issuer, warps 2-9: epilogue
using namespace gemm;

// MINB = 2 caps the registers so that two blocks fit an SM (used when a launch has more blocks
// than SMs; costs a few spills in the tail), MINB = 1 leaves the compiler free.
template <int EPI, int MINB>
__global__ void __launch_bounds__(kThreads, MINB)
k_tc_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
          const TcArgs g) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) GemmShared sh;

  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    gemm_init_barriers(sh, g.stages);
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
  // Everything above touched only this block's own shared and tensor memory.  When the launch
  // allowed it, that much ran while the previous kernel of the stream was still finishing; from
  // here on its results are read, so wait for it to complete (returns at once otherwise).
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();
  // the split path is compiled out of the register-capped build, which is never used with a split
  gemm_tile<EPI, MINB == 1>(tmA, tmB, g, (int)blockIdx.x, (int)blockIdx.y, smem, sh, tmem_base);
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, g.tmem_cols);
}

// Hidden-layer forward tile with its contraction split over the blocks of a cluster (see
// gemm_tile, CLUSTER): grid.x = row tiles x splits, cluster = the `splits` blocks of a row tile.
__global__ void __launch_bounds__(kThreads, 1)
k_tc_gemm_ks(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
             const TcArgs g) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) GemmShared sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
    gemm_init_barriers(sh, g.stages);
    // every lane of the four sending warps of each other block arrives once
    mbar_init(&sh.recv_bar, (uint32_t)(g.splits - 1) * 128u);
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
  cluster_sync_all();           // every block's barriers exist before anyone arrives on them
  const uint32_t tmem_base = sh.tmem_slot;
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();
  gemm_tile<EPI_FWD_HIDDEN, false, true>(tmA, tmB, g, (int)blockIdx.x, (int)blockIdx.y, smem, sh,
                                         tmem_base);
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync_all();           // nobody leaves while a peer may still write into its shared memory
  if (warp == 1) tmem_dealloc(tmem_base, g.tmem_cols);
}

// bf16 copy of the global model w~ (shared by all learners at the first step of a round, when
// every replica equals w~).  One launch for all layers: block row y takes layer y, grid-stride
// over that layer's weights.
struct ShadowArgs {
  int64_t w_off[MAVG_MAX_LAYERS], total[MAVG_MAX_LAYERS], sh_off[MAVG_MAX_LAYERS];
};
__global__ void __launch_bounds__(256)
k_shadow_from_global(const float* __restrict__ w, __nv_bfloat16* __restrict__ w16,
                     const ShadowArgs a) {
  const int l = blockIdx.y;
  const float* src = w + a.w_off[l];
  __nv_bfloat16* dst = w16 + a.sh_off[l];
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < a.total[l];
       t += (int64_t)gridDim.x * blockDim.x)
    dst[t] = __float2bfloat16_rn(src[t]);
}

// The learners' own bf16 copies from their masters: grid (x, layers, P).
__global__ void __launch_bounds__(256)
k_copies_from_replicas(const float* __restrict__ rep, int64_t rep_stride, __nv_bfloat16* __restrict__ w16,
                       int64_t n16, const ShadowArgs a) {
  const int l = blockIdx.y;
  const float* src = rep + (size_t)blockIdx.z * rep_stride + a.w_off[l];
  __nv_bfloat16* dst = w16 + (size_t)blockIdx.z * n16 + a.sh_off[l];
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < a.total[l];
       t += (int64_t)gridDim.x * blockDim.x)
    dst[t] = __float2bfloat16_rn(src[t]);
}

// ---------------------------------------------------------------------------------- host side
size_t up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Forward / dgrad plan.  To fill the GPU the batch may be cut into column tiles (`tile_n`: only
// the hidden-layer forward can, its tail needs no sum over the batch) and, if blocks are still
// few and the contraction long, the contraction is split; a block never gets fewer than 8 slabs
// (512 elements), below which the split's fix-up costs more than it saves.
GemmPlan plan_partial(int M, int N, int K, int P, int sm_count, bool tile_n) {
  GemmPlan g{};
  g.BN = (N + 15) / 16 * 16;
  g.m_tiles = (M + kBM - 1) / kBM;
  g.n_tiles = 1;
  g.nkb = (K + kBK - 1) / kBK;
  const int enough = sm_count - sm_count / 5;   // ~80 % of the SMs busy counts as full
  if (tile_n)
    while (g.m_tiles * g.n_tiles * P < enough && g.BN % 64 == 0) {
      g.BN /= 2;
      g.n_tiles *= 2;
    }
  int tiles = g.m_tiles * g.n_tiles * P;
  int want = tiles >= enough ? 1 : (sm_count + tiles - 1) / tiles;
  if (want > g.nkb / 8) want = g.nkb / 8;
  if (want < 1) want = 1;
  g.kb_per_split = (g.nkb + want - 1) / want;
  g.splits = (g.nkb + g.kb_per_split - 1) / g.kb_per_split;
  int stage_bytes = kATileBytes + g.BN * kBK * 2;
  // more blocks than SMs: two blocks share an SM, so that one block's set-up and tail overlap
  // the other's main loop; otherwise one block takes the whole shared memory
  g.two_per_sm = (g.splits == 1 && g.m_tiles * g.n_tiles * P > sm_count) ? 1 : 0;
  const int budget = g.two_per_sm ? 104 * 1024 : 200 * 1024;
  g.stages = budget / stage_bytes;
  if (g.stages > kMaxStages) g.stages = kMaxStages;
  if (g.stages > g.kb_per_split) g.stages = g.kb_per_split < 2 ? 2 : g.kb_per_split;
  g.tmem_cols = 32;
  while ((int)g.tmem_cols < g.BN) g.tmem_cols <<= 1;
  return g;
}

// Whether the weight gradients are large enough to be launches of their own (more than 64 tiles per SM
// in layer 1) and can take the next step's forward products along.
bool rides(const mavg_config* cfg, int sm_count) {
  const long m_tiles = (cfg->dims[1] + kWgradTileRows - 1) / kWgradTileRows;
  const long n_tiles = (cfg->dims[0] + kWgradTileCols - 1) / kWgradTileCols;
  return cfg->n_layers >= 2 && cfg->B <= 128 && cfg->P * m_tiles * n_tiles > 64L * sm_count;
}

TcLayout make_layout(const mavg_config* cfg, size_t base, int sm_count) {
  TcLayout t{};
  const int L = cfg->n_layers, P = cfg->P, B = cfg->B;
  const size_t rows = (size_t)P * B;
  t.L = L;
  t.cpad = (cfg->dims[L] + 7) / 8 * 8;
  int64_t o16 = 0;
  for (int l = 0; l < L; ++l) {
    t.sh_off[l] = o16;
    o16 += (int64_t)up((size_t)cfg->dims[l] * cfg->dims[l + 1], 64);
  }
  t.n16 = o16;
  size_t off = up(base, 1024);
  auto take = [&](size_t bytes) { size_t r = off; off = up(off + bytes, 1024); return r; };
  int max_m_tiles = 1;
  for (int l = 1; l <= L; ++l)
    max_m_tiles = std::max(max_m_tiles, 8 * ((cfg->dims[l] + kBM - 1) / kBM));   // up to 8 column tiles
  size_t pb = 1024;
  for (int l = 1; l <= L; ++l) {
    GemmPlan f = plan_partial(cfg->dims[l], B, cfg->dims[l - 1], P, sm_count, l < L);
    if (f.splits > 1) pb = std::max(pb, (size_t)f.splits * rows * cfg->dims[l] * 4);
    if (l > 1) {
      GemmPlan d = plan_partial(cfg->dims[l - 1], B, cfg->dims[l], P, sm_count, false);
      if (d.splits > 1) pb = std::max(pb, (size_t)d.splits * rows * cfg->dims[l - 1] * 4);
    }
  }
  t.part_bytes = pb;
  t.part = take(pb);
  t.counters_bytes = (size_t)P * max_m_tiles * sizeof(int);
  t.counters = take(t.counters_bytes);
  t.w16g = take((size_t)t.n16 * 2);
  t.tail_part = take(tail_fused_supported(cfg) ? tail_fused_part_bytes(cfg) : 16);
  t.dz[L] = take(rows * t.cpad * 2);
  t.dz_t[L] = take(rows * cfg->dims[L] * 2);
  t.zpart_bytes = 16;
  t.zcount_bytes = 16;
  if (B <= 128)
    for (int l = 1; l < L; ++l) {
      const WgradPlan w = plan_wgrad_stream(cfg->dims[l], cfg->dims[l - 1], B, P, sm_count, false, true, true);
      t.zpart_bytes = std::max(t.zpart_bytes, (size_t)P * w.m_tiles * w.n_chunks * B * kBM * sizeof(float));
      t.zcount_bytes = std::max(t.zcount_bytes, (size_t)P * w.m_tiles * sizeof(int));
    }
  t.zcount = take(t.zcount_bytes);
  t.shared_end = off;
  for (int i = 0; i < 2; ++i) {
    t.xg[i] = take(rows * cfg->dims[0] * 2);
    t.xt[i] = take(rows * cfg->dims[0] * 2);
  }
  for (int l = 1; l < L; ++l) {
    const int d = cfg->dims[l];
    t.act[l] = take(rows * d * 2);
    t.act_t[l] = take(rows * d * 2);
    t.act_b[l] = take(rows * d * 2);
    t.act_t_b[l] = take(rows * d * 2);
    t.dz[l] = take(rows * d * 2);
    t.dz_t[l] = take(rows * d * 2);
  }
  t.w16 = take((size_t)P * t.n16 * 2);
  // partial sums of a forward product that rides along with a weight-gradient launch: one 128 x B fp32
  // tile per (learner, row tile, run of column tiles) of that launch's plan; the layers use the space
  // one after the other
  t.zpart = take(t.zpart_bytes);
  t.w16b_stride = L >= 3 ? (int64_t)up((size_t)cfg->dims[L - 2] * cfg->dims[L - 1], 64) : 0;
  t.w16b = take(L >= 3 ? (size_t)P * t.w16b_stride * 2 : 16);
  // Split masters take no room of their own (an array of low halves would be another 2 bytes per hidden
  // weight and learner, 537 MB on the large MLP).  Where forward products ride, the second copy of layer
  // L-1 is not used at all -- it belongs to the merged weight-gradient launch -- and layer 1's bf16 copy
  // is not from the first step's forward product to the last step's weight gradient.  The halves lie
  // there, lower layers in the former first; layers that find no room keep fp32 masters.
  if (rides(cfg, sm_count)) {
    const int64_t room_b = t.w16b_stride, room_1 = (int64_t)up((size_t)cfg->dims[0] * cfg->dims[1], 64);
    int64_t at_b = 0, at_1 = 0;
    for (int l = 2; l < L; ++l) {
      const int64_t size = (int64_t)up((size_t)cfg->dims[l] * cfg->dims[l - 1], 64);
      if (at_b + size <= room_b) {
        t.lo16[l] = t.w16b + (size_t)at_b * 2;
        t.lo_stride[l] = t.w16b_stride;
        at_b += size;
      } else if (at_1 + size <= room_1) {
        t.lo16[l] = t.w16 + (size_t)(t.sh_off[0] + at_1) * 2;
        t.lo_stride[l] = t.n16;
        at_1 += size;
        if (!t.lo_on_w1) t.lo_on_w1 = l;
      }
    }
  }
  t.end = off;
  return t;
}

// SM count the plans (and with them the size of the partial buffer) are made for, so that the
// workspace size does not depend on the device that later runs the problem.
constexpr int kPlanSmCount = 148;

template <int EPI>
cudaError_t launch_gemm(mavg_ctx* c, int cls, const CUtensorMap& a, const CUtensorMap& b,
                        const GemmPlan& pl, TcArgs g) {
  g.BN = pl.BN;
  g.m_tiles = pl.m_tiles;
  g.n_tiles = pl.n_tiles;
  g.splits = pl.splits;
  g.kb_per_split = pl.kb_per_split;
  g.nkb = pl.nkb;
  g.stages = pl.stages;
  g.tmem_cols = pl.tmem_cols;
  g.P = c->cfg.P;
  g.rep_stride = c->buf.replica_stride;
  g.gamma = c->cfg.local_lr;
  g.status = (int*)ws_ptr(c, c->ws.status);
  size_t pipe = (size_t)pl.stages * (kATileBytes + pl.BN * kBK * 2);
  size_t smem = pipe + 1024;
  if (EPI == EPI_FWD_LAST)   // the loss tail reuses the pipeline buffers: logits, dZ, row losses
    smem = std::max(pipe, ((size_t)2 * g.N * g.M + g.N) * sizeof(float)) + 1024;
  smem = std::max(smem, tmem_share_bytes(pl.tmem_cols, sizeof(GemmShared)));
  dim3 grid((unsigned)(pl.m_tiles * pl.n_tiles * pl.splits), (unsigned)c->cfg.P);
  cudaLaunchConfig_t lc{};
  lc.gridDim = grid;
  lc.blockDim = dim3(kThreads);
  lc.dynamicSmemBytes = smem;
  lc.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  prof_begin(c, cls);
  cudaError_t e = pl.two_per_sm ? cudaLaunchKernelEx(&lc, k_tc_gemm<EPI, 2>, a, b, g)
                                : cudaLaunchKernelEx(&lc, k_tc_gemm<EPI, 1>, a, b, g);
  prof_end(c);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Plan of the cluster-split forward product of a hidden layer, or splits = 1 if it does not apply:
// the default plan would cut the batch into B / 32 column tiles (so every block would stream the
// whole weight tile for a quarter or half of the batch), and the contraction is long enough.
GemmPlan plan_cluster_split(const GemmPlan& f, int M, int B, int K) {
  GemmPlan ks{};
  ks.splits = 1;
  const int S = B / 32;
  if ((B != 64 && B != 128) || f.splits != 1 || f.n_tiles != S || f.BN != 32) return ks;
  const int nkb = (K + kBK - 1) / kBK;
  const int per = (nkb + S - 1) / S;
  if (nkb < 4 * S || per * (S - 1) >= nkb) return ks;
  ks.BN = B;
  ks.m_tiles = (M + kBM - 1) / kBM;
  ks.n_tiles = 1;
  ks.nkb = nkb;
  ks.splits = S;
  ks.kb_per_split = per;
  const int stage_bytes = kATileBytes + B * kBK * 2;
  ks.stages = (216 * 1024 - S * kBM * 32 * 4) / stage_bytes;
  if (ks.stages > kMaxStages) ks.stages = kMaxStages;
  if (ks.stages > per) ks.stages = per;
  if (ks.stages < 2) { ks.splits = 1; return ks; }
  ks.tmem_cols = 32;
  while ((int)ks.tmem_cols < B) ks.tmem_cols <<= 1;
  return ks;
}

cudaError_t launch_gemm_ks(mavg_ctx* c, const CUtensorMap& a, const CUtensorMap& b,
                           const GemmPlan& pl, TcArgs g) {
  g.BN = pl.BN;
  g.m_tiles = pl.m_tiles;
  g.n_tiles = 1;
  g.splits = pl.splits;
  g.kb_per_split = pl.kb_per_split;
  g.nkb = pl.nkb;
  g.stages = pl.stages;
  g.tmem_cols = pl.tmem_cols;
  g.P = c->cfg.P;
  g.rep_stride = c->buf.replica_stride;
  g.gamma = c->cfg.local_lr;
  g.status = (int*)ws_ptr(c, c->ws.status);
  const size_t smem = std::max((size_t)pl.stages * (kATileBytes + pl.BN * kBK * 2) + (size_t)pl.splits * kBM * 32 * 4 + 1024,
                               tmem_share_bytes(pl.tmem_cols, sizeof(GemmShared)));
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)(pl.m_tiles * pl.splits), (unsigned)c->cfg.P);
  lc.blockDim = dim3(kThreads);
  lc.dynamicSmemBytes = smem;
  lc.stream = c->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)pl.splits;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  prof_begin(c, MAVG_K_FWD);
  cudaError_t e = cudaLaunchKernelEx(&lc, k_tc_gemm_ks, a, b, g);
  prof_end(c);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

bool tc_shapes_ok(const mavg_config* cfg, std::string* why) {
  if (cfg->B % 16 != 0 || cfg->B > 256) {
    if (why) *why = "the tensor-core path needs B to be a multiple of 16 and at most 256";
    return false;
  }
  for (int l = 0; l < cfg->n_layers; ++l)
    if (cfg->dims[l] % 8 != 0) {
      if (why) *why = "the tensor-core path needs every layer's input width to be a multiple of 8";
      return false;
    }
  if (cfg->dims[cfg->n_layers] > 32) {
    if (why) *why = "the tensor-core path needs at most 32 classes";
    return false;
  }
  return true;
}

namespace {

// Small problems (a few dozen weight tiles per SM in the largest layer): one persistent launch
// takes the weight gradients of all layers, instead of one launch per layer on a side stream.
bool wgrad_merges(const mavg_config* cfg, int sm_count, const WgradPlan* w) {
  if (cfg->n_layers < 2 || (long)cfg->P * w[1].m_tiles * w[1].n_tiles > 64L * sm_count) return false;
  for (int l = 2; l <= cfg->n_layers; ++l)
    if (w[l].slots != w[1].slots || w[l].a_bufs != w[1].a_bufs) return false;
  return true;
}

// Plans of the weight-gradient launches that can take the next step's forward product along, of layers 1..n: n.
int riding_plans(const mavg_config* cfg, const TcLayout& t, int sm_count, bool momentum, bool streaming, WgradPlan* f) {
  if (cfg->B > 128) return 0;
  for (int l = 1; l < cfg->n_layers; ++l) {
    f[l] = plan_wgrad_stream(cfg->dims[l], cfg->dims[l - 1], cfg->B, cfg->P, sm_count, momentum, streaming, true, t.lo_stride[l] > 0);
    const size_t need = (size_t)cfg->P * f[l].m_tiles * f[l].n_chunks * cfg->B * kBM * sizeof(float);
    if (f[l].slots < 2 || need > t.zpart_bytes || (size_t)cfg->P * f[l].m_tiles * sizeof(int) > t.zcount_bytes) return l - 1;
  }
  return cfg->n_layers - 1;
}

// Whether rebuilt steps can form those products' sums in their order: partial sums have columns of tensor memory.
bool sums_fit(const mavg_config* cfg, int riding, const WgradPlan* f) {
  for (int l = 1; l <= riding; ++l)
    if (partial_sums(cfg->P, f[l]) && f[l].n_chunks * cfg->B > 512) return false;
  return true;
}

// Whether a handle's rounds may be rebuilt, from the configuration alone (their masters are beyond the L2).
bool may_rebuild(const mavg_config* cfg, const TcLayout& t) {
  WgradPlan w[MAVG_MAX_LAYERS + 1], f[MAVG_MAX_LAYERS + 1];
  const bool momentum = cfg->learner_momentum != 0.f;
  for (int l = 1; l <= cfg->n_layers; ++l)
    w[l] = plan_wgrad_stream(cfg->dims[l], cfg->dims[l - 1], cfg->B, cfg->P, kPlanSmCount, momentum, true);
  if (wgrad_merges(cfg, kPlanSmCount, w)) return true;
  const int riding = riding_plans(cfg, t, kPlanSmCount, momentum, true, f);
  return sums_fit(cfg, riding, f) && (!riding || reb_riding(cfg));
}

}  // namespace

size_t tc_workspace_bytes(const mavg_config* cfg, size_t base, size_t* act_off, size_t* least) {
  *act_off = base;
  const TcLayout t = make_layout(cfg, base, kPlanSmCount);
  *least = t.end;
  if (fac_reserved(cfg)) return std::max(t.end, fac_layout(cfg, t.shared_end).end);
  return reb_reserved(cfg) && may_rebuild(cfg, t) ? std::max(t.end, reb_layout(cfg, t.shared_end).end) : t.end;
}

namespace {

TcArgs product_args(mavg_ctx* c, const StepOperands& o, int features, int bias_layer) {
  const TcLayout& t = ((const TcState*)c->mlp)->lay;
  TcArgs g{};
  g.M = features; g.N = c->cfg.B;
  g.a_batched = o.shared_w ? 0 : 1; g.b_batched = 1;
  g.part = (float*)ws_ptr(c, t.part); g.counters = (int*)ws_ptr(c, t.counters);
  g.bias_rep = c->buf.replicas; g.bias_off = c->layers[bias_layer - 1].b_off;
  g.bias_in = o.shared_w ? c->buf.global_w : c->buf.replicas;
  g.bias_in_stride = o.shared_w ? 0 : c->buf.replica_stride;
  g.out_bm = o.out_bm; g.out_mb = o.out_mb;
  g.mom = o.mom;
  return g;
}

cudaError_t forward(mavg_ctx* c, const StepOperands& o) {
  const TcState* st = (const TcState*)c->mlp;
  const MlpLayer& ly = c->layers[o.l - 1];
  const FwdForm form = c->schedule == 0 ? fwd_form(st, o.l, o.shared_w) : FwdForm::TILES;
  if (form == FwdForm::DENSE)
    return launch_fwd_dense(c, st->dense[o.l], *o.w, *o.in, ly.out, c->buf.global_w + ly.b_off, o.out_bm, o.out_mb);
  const TcArgs g = product_args(c, o, ly.out, o.l);
  return form == FwdForm::SPLIT ? launch_gemm_ks(c, *o.w, *o.in, st->fwd_ks[o.l], g)
                                : launch_gemm<EPI_FWD_HIDDEN>(c, MAVG_K_FWD, *o.w, *o.in, st->fwd[o.l], g);
}

TailLaunch tail_launch(mavg_ctx* c, const StepOperands& o) {
  const TcLayout& t = ((const TcState*)c->mlp)->lay;
  TailLaunch tl{};
  tl.a_bm = o.a_bm;
  tl.w16 = o.w16; tl.w16_stride = o.w16_stride;
  tl.shared_w = o.shared_w;
  tl.labels = o.labels;
  tl.loss_out = (float*)ws_ptr(c, c->ws.losses) + (o.step - 1); tl.loss_stride = c->cfg.K;
  tl.dz_t = (__nv_bfloat16*)ws_ptr(c, t.dz_t[o.l]);
  tl.dz_bm = o.dz_bm; tl.cpad = t.cpad;
  tl.dzp_bm = o.out_bm; tl.dzp_mb = o.out_mb;
  tl.part = (float*)ws_ptr(c, t.tail_part);
  tl.mom = o.mom;
  return tl;
}

cudaError_t last_layer(mavg_ctx* c, const StepOperands& o) {
  const TcState* st = (const TcState*)c->mlp;
  const TcLayout& t = st->lay;
  if (st->tail_ok && c->schedule == 0) {
    const TailLaunch tl = tail_launch(c, o);
    const cudaError_t e = launch_tail_fused(c, tl);
    return e != cudaSuccess ? e : launch_tail_finish(c, tl);
  }
  TcArgs g = product_args(c, o, c->cfg.dims[o.l], o.l);
  g.labels = o.labels; g.loss_out = (float*)ws_ptr(c, c->ws.losses) + (o.step - 1); g.loss_stride = c->cfg.K;
  g.dz_bm = o.dz_bm; g.cpad = t.cpad; g.dz_mb = (__nv_bfloat16*)ws_ptr(c, t.dz_t[o.l]);
  return launch_gemm<EPI_FWD_LAST>(c, MAVG_K_FWD, *o.w, *o.in, st->fwd[o.l], g);
}

cudaError_t dgrad(mavg_ctx* c, const StepOperands& o) {
  TcArgs g = product_args(c, o, c->cfg.dims[o.l - 1], o.l - 1);
  g.mask_mb = o.mask_mb;
  g.a_mn = 1;
  return launch_gemm<EPI_DGRAD>(c, MAVG_K_DGRAD, *o.w, *o.in, ((const TcState*)c->mlp)->dgrad[o.l], g);
}

}  // namespace

mavg_status tc_setup(mavg_ctx* c) {
  const mavg_config& cfg = c->cfg;
  TcState* st = new TcState();
  c->mlp = st;
  st->lay = make_layout(&cfg, c->ws.act, kPlanSmCount);
  st->encode = tensor_map_encoder(&c->err);
  if (!st->encode) return MAVG_ERR_UNSUPPORTED;
  const TcLayout& t = st->lay;
  const int L = cfg.n_layers, P = cfg.P, B = cfg.B;
  char* ws = (char*)c->buf.workspace;
  auto bf = [&](size_t off) { return (void*)(ws + off); };
  std::string why;
  bool ok = true;
  for (int l = 1; l <= L && ok; ++l) {
    const int in = cfg.dims[l - 1], out = cfg.dims[l];
    const int dz_ld = l < L ? out : t.cpad;
    st->fwd[l] = plan_partial(out, B, in, P, kPlanSmCount, l < L);
    st->fwd_ks[l] = GemmPlan{};
    st->fwd_ks[l].splits = 1;
    if (l < L) st->fwd_ks[l] = plan_cluster_split(st->fwd[l], out, B, in);
    st->wgrad_mom = c->buf.learner_u != nullptr;
    st->wgrad[l] = plan_wgrad_stream(out, in, B, P, c->sm_count, st->wgrad_mom, !masters_fit_l2(c));
    if (st->wgrad_mom)
      ok = ok && encode_any(st, &st->u32[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4,
                            c->buf.learner_u + c->layers[l - 1].w_off, in, out, P, in,
                            c->buf.replica_stride, kWgradTileCols, kWgradTileRows,
                            CU_TENSOR_MAP_SWIZZLE_128B, &why);
    __nv_bfloat16* w16 = (__nv_bfloat16*)bf(t.w16) + t.sh_off[l - 1];
    __nv_bfloat16* w16g = (__nv_bfloat16*)bf(t.w16g) + t.sh_off[l - 1];
    ok = ok && encode_map(st, &st->w[l], w16, in, out, P, in, t.n16, kBM, &why);
    ok = ok && encode_map(st, &st->wg[l], w16g, in, out, 1, in, t.n16, kBM, &why);
    ok = ok && encode_map(st, &st->w_mn[l], w16, in, out, P, in, t.n16, 64, &why);
    if (L >= 3 && l == L - 1) {      // second copy of this layer's bf16 weights
      st->dbl_layer = l;
      __nv_bfloat16* wb = (__nv_bfloat16*)bf(t.w16b);
      ok = ok && encode_map(st, &st->w_b, wb, in, out, P, in, t.w16b_stride, kBM, &why);
      ok = ok && encode_map(st, &st->w_mn_b, wb, in, out, P, in, t.w16b_stride, 64, &why);
      ok = ok && encode_any(st, &st->w16_st_b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, wb, in, out, P,
                            in, t.w16b_stride, kWgradTileCols, kWgradTileRows,
                            CU_TENSOR_MAP_SWIZZLE_64B, &why);
    }
    ok = ok && encode_map(st, &st->wg_mn[l], w16g, in, out, 1, in, t.n16, 64, &why);
    if (l == 1) {
      for (int i = 0; i < 2 && ok; ++i) {
        ok = ok && encode_map(st, &st->x_in[i], bf(t.xg[i]), in, B, P, in, (int64_t)B * in,
                              st->fwd[l].BN, &why);
        ok = ok && encode_map(st, &st->x_in_t[i], bf(t.xt[i]), B, in, P, B, (int64_t)B * in,
                              kWgradTileCols, &why);
        if (st->fwd_ks[l].splits > 1)
          ok = ok && encode_map(st, &st->x_in_ks[i], bf(t.xg[i]), in, B, P, in, (int64_t)B * in,
                                B, &why);
      }
    } else {
      ok = ok && encode_map(st, &st->act_in[l], bf(t.act[l - 1]), in, B, P, in, (int64_t)B * in,
                            st->fwd[l].BN, &why);
      ok = ok && encode_map(st, &st->act_in_t[l], bf(t.act_t[l - 1]), B, in, P, B,
                            (int64_t)B * in, kWgradTileCols, &why);
      if (st->fwd_ks[l].splits > 1)
        ok = ok && encode_map(st, &st->act_in_ks[l], bf(t.act[l - 1]), in, B, P, in,
                              (int64_t)B * in, B, &why);
      // the same three views of the second set of activation buffers
      ok = ok && encode_map(st, &st->act_in_b[l], bf(t.act_b[l - 1]), in, B, P, in, (int64_t)B * in,
                            st->fwd[l].BN, &why);
      ok = ok && encode_map(st, &st->act_in_t_b[l], bf(t.act_t_b[l - 1]), B, in, P, B,
                            (int64_t)B * in, kWgradTileCols, &why);
      if (st->fwd_ks[l].splits > 1)
        ok = ok && encode_map(st, &st->act_in_ks_b[l], bf(t.act_b[l - 1]), in, B, P, in,
                              (int64_t)B * in, B, &why);
    }
    ok = ok && encode_map(st, &st->dz_t[l], bf(t.dz_t[l]), B, out, P, B, (int64_t)B * out, kBM,
                          &why);
    ok = ok && encode_any(st, &st->w32[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4,
                          c->buf.replicas + c->layers[l - 1].w_off, in, out, P, in,
                          c->buf.replica_stride, kWgradTileCols, kWgradTileRows,
                          CU_TENSOR_MAP_SWIZZLE_128B, &why);
    ok = ok && encode_any(st, &st->w32g[l], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4,
                          c->buf.global_w + c->layers[l - 1].w_off, in, out, 1, in,
                          c->buf.replica_stride, kWgradTileCols, kWgradTileRows,
                          CU_TENSOR_MAP_SWIZZLE_128B, &why);
    ok = ok && encode_any(st, &st->w16_st[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, w16, in, out, P,
                          in, t.n16, kWgradTileCols, kWgradTileRows, CU_TENSOR_MAP_SWIZZLE_64B,
                          &why);
    if (l > 1) {
      st->dgrad[l] = plan_partial(in, B, out, P, kPlanSmCount, false);
      ok = ok && encode_map(st, &st->dz[l], bf(t.dz[l]), out, B, P, dz_ld, (int64_t)B * dz_ld,
                            st->dgrad[l].BN, &why);
    }
  }
  if (!ok) {
    c->err = why;
    return MAVG_ERR_CUDA;
  }
  // 227 KB per block in all, of which a few hundred bytes are the kernel's static variables
  constexpr int kMaxDynSmem = 225 * 1024;
  cudaError_t e = cudaSuccess;
  const void* kernels[] = {(const void*)k_tc_gemm<EPI_FWD_HIDDEN, 1>, (const void*)k_tc_gemm<EPI_FWD_HIDDEN, 2>,
                           (const void*)k_tc_gemm<EPI_FWD_LAST, 1>,   (const void*)k_tc_gemm<EPI_FWD_LAST, 2>,
                           (const void*)k_tc_gemm<EPI_DGRAD, 1>,      (const void*)k_tc_gemm<EPI_DGRAD, 2>,
                           (const void*)k_tc_gemm_ks};
  for (const void* k : kernels)
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
  if (e == cudaSuccess) e = wgrad_stream_prepare();
  st->wgrad_merged = wgrad_merges(&cfg, c->sm_count, st->wgrad);
  // Where the weight gradients are launches of their own, the launch of layer l can take the
  // next step's forward product of layer l along (layers 1..fuse_upto, a prefix of the hidden
  // layers): its plan gets room for the next step's input tile and long runs, and the input
  // buffers get a view with 32-column boxes.
  st->fuse_upto = 0;
  const int riding = st->wgrad_merged ? 0 : riding_plans(&cfg, t, c->sm_count, st->wgrad_mom, !masters_fit_l2(c), st->wgrad_f);
  for (int l = 1; l <= riding && ok; ++l) {
    const int in = cfg.dims[l - 1], out = cfg.dims[l];
    bool enc = true;
    for (int i = 0; i < 2 && enc; ++i) {
      const size_t src = l == 1 ? t.xg[i] : (i == 0 ? t.act[l - 1] : t.act_b[l - 1]);
      enc = encode_any(st, &st->a_next[l][i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, bf(src), in, B,
                       P, in, (int64_t)B * in, kWgradTileCols, B, CU_TENSOR_MAP_SWIZZLE_64B, &why);
    }
    if (enc && t.lo_stride[l] > 0)
      enc = encode_any(st, &st->lo16[l], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, bf(t.lo16[l]), in, out, P,
                       in, t.lo_stride[l], kWgradTileCols, kWgradTileRows, CU_TENSOR_MAP_SWIZZLE_64B,
                       &why);
    if (!enc) break;
    st->fuse_upto = l;
  }
  // First step of a round: the hidden layers' forward products as one dense product each, where
  // that gives enough tiles (the input buffers seen as one [P*B, in] array).
  for (int l = 1; l <= L; ++l) st->dense[l] = DensePlan{};
  for (int l = 1; l < L && ok; ++l) {
    const int in = cfg.dims[l - 1];
    DensePlan pl = plan_fwd_dense(cfg.dims[l], in, B, P, c->sm_count);
    if (!pl.ok) continue;
    bool enc = true;
    for (int i = 0; i < 2 && enc; ++i) {
      const size_t src = l == 1 ? t.xg[i] : (i == 0 ? t.act[l - 1] : t.act_b[l - 1]);
      enc = encode_map(st, &st->in2d[l][i], bf(src), in, P * B, 1, in, (int64_t)P * B * in,
                       kDenseCols, &why);
    }
    if (enc) st->dense[l] = pl;
  }
  if (e == cudaSuccess) e = fwd_dense_prepare();
  // the meta-update writes the bf16 copy of w~ itself where its vector kernel takes the whole model
  c->shadow.dst = (__nv_bfloat16*)(ws + t.w16g);
  c->shadow.L = L;
  for (int l = 1; l <= L; ++l) {
    c->shadow.w_off[l - 1] = c->layers[l - 1].w_off;
    c->shadow.total[l - 1] = (int64_t)c->layers[l - 1].in * c->layers[l - 1].out;
    c->shadow.sh_off[l - 1] = t.sh_off[l - 1];
  }
  // The fused CUDA-core last layer pays where the tensor-core products of that layer would leave most of
  // the GPU idle (at most half a wave of its data gradient's tiles), and again where these take more but
  // its forward product, one tile per learner, is less than a wave with little to do: from three quarters
  // of a wave of data-gradient tiles on for layers of at most 16 K weights, at any number for at most
  // 4 K.  Its own work grows with the batch rows times the weights: up to 32 M of them, 48 M where the
  // layer below is four row tiles wide or wider (that much less is left of the tensor form's advantage),
  // and at most 32 K rows.  Measured, us a round of 4 steps, fused / tensor tiles:
  //   128-24, B = 64: P = 148 262 / 291, P = 160 286 / 282, P = 300 532 / 506; 64-10, B = 128: P = 148
  //   282 / 319, P = 200 357 / 335 (more than a wave of learners); 600-800-800-16, B = 32: P = 16 363 / 399;
  //   200-16, B = 64: P = 148 (29 M) 357 / 367; 128-24, B = 128: P = 100 (38 M) 269 / 274, P = 148 (56 M)
  //   376 / 365; four row tiles and more: 504-32, B = 128: P = 24 (47 M) 382 / 404, P = 28 (55 M) 447 / 443;
  //   512-10, B = 64: P = 48 923 / 978, P = 100 (31 M) 1748 / 1761;
  //   64-64-4, B = 256: P = 100 (26 K rows) 405 / 427, P = 148 (38 K) 562 / 549.
  {
    const int row_tiles = (cfg.dims[L - 1] + kBM - 1) / kBM;
    const long tiles = (long)P * row_tiles;
    const long weights = (long)cfg.dims[L - 1] * cfg.dims[L];
    const int64_t work = (int64_t)P * B * weights;
    const bool few = 2 * tiles <= c->sm_count;
    st->tail_ok = tail_fused_supported(&cfg) &&
                  (few || (P <= c->sm_count && (int64_t)P * B <= 32 * 1024 &&
                           (weights <= 4096 || (4 * tiles >= 3 * c->sm_count && weights <= 16 * 1024)) &&
                           work <= (row_tiles >= 4 ? 48 : 32) * 1024 * 1024));
    // Beside the fused last layer the last two layers' weight gradients may run beside the data gradients
    // that are left, on the SMs these do not take.  With more tiles than half a wave too few SMs are left:
    // 600-800-800-16, B = 64, P = 16 (36 SMs) 615 us a round against 433 in one launch at the end of the
    // step; 512-256-256-8, P = 56 (36 SMs) 363 against 295, P = 40 (68 SMs) 269 against 245.
    st->wgrad_beside = few;
  }
  if (e == cudaSuccess && st->tail_ok) e = tail_fused_prepare();
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&st->s_wgrad, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&st->s_gather, cudaStreamNonBlocking);
  cudaEvent_t* evs[] = {&st->ev_fork, &st->ev_wgrad_done, &st->ev_gather_done, &st->ev_tail_done,
                        &st->ev_x_free[0], &st->ev_x_free[1]};
  for (cudaEvent_t* ev : evs)
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming);
  // (also for calls of fewer steps or another momentum than the handle was made for, where the room is there)
  if (e == cudaSuccess && fac_steps(&cfg) &&
      c->buf.workspace_bytes >= std::max(t.end, fac_layout(&cfg, t.shared_end).end))
    fac_setup(c, st);
  st->run_forward = forward;
  st->run_last_layer = last_layer;
  st->run_dgrad = dgrad;
  if (e == cudaSuccess && reb_steps(&cfg) && sums_fit(&cfg, st->fuse_upto, st->wgrad_f) && c->buf.workspace_bytes >= std::max(t.end, reb_layout(&cfg, t.shared_end).end))
    reb_setup(c, st);
  if (e == cudaSuccess)
    e = cudaMemsetAsync(ws + t.counters, 0, t.counters_bytes, c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(ws + t.zcount, 0, t.zcount_bytes, c->stream);

  if (e != cudaSuccess) {
    c->err = std::string("tensor-core path set-up: ") + cudaGetErrorString(e);
    cudaGetLastError();   // reported here; do not leave it pending for a later call
    return MAVG_ERR_CUDA;
  }
  return MAVG_OK;
}

void tc_teardown(mavg_ctx* c) {
  TcState* st = (TcState*)c->mlp;
  if (st) {
    if (st->s_wgrad) cudaStreamDestroy(st->s_wgrad);
    if (st->s_gather) cudaStreamDestroy(st->s_gather);
    cudaEvent_t evs[] = {st->ev_fork, st->ev_wgrad_done, st->ev_gather_done, st->ev_tail_done,
                         st->ev_x_free[0], st->ev_x_free[1]};
    for (cudaEvent_t ev : evs)
      if (ev) cudaEventDestroy(ev);
    delete st->fac;
    delete st->reb;
  }
  delete st;
  c->mlp = nullptr;
}

int tc_get_w16_cur(mavg_ctx* c) { return c->mlp ? ((TcState*)c->mlp)->w16_cur : 0; }
void tc_set_w16_cur(mavg_ctx* c, int cur) {
  if (c->mlp) ((TcState*)c->mlp)->w16_cur = cur;
}

// After an abandoned wait the arrival counters of split tiles and of riding forward products may
// have been left mid-count: zero them (stream-ordered), so that the handle's next launches count
// from a clean state.
void tc_reset_counters(mavg_ctx* c) {
  const TcState* st = (const TcState*)c->mlp;
  if (!st) return;
  char* ws = (char*)c->buf.workspace;
  cudaMemsetAsync(ws + st->lay.counters, 0, st->lay.counters_bytes, c->stream);
  cudaMemsetAsync(ws + st->lay.zcount, 0, st->lay.zcount_bytes, c->stream);
}

bool tc_factored(const mavg_ctx* c) { return fac_usable(c); }
bool tc_rebuilt(const mavg_ctx* c) { return reb_usable(c) && !fac_usable(c); }

void tc_step_plan(mavg_ctx* c, int32_t* out) {
  const TcState* st = (const TcState*)c->mlp;
  if (!st) return;
  out[MAVG_PLAN_TENSOR_PATH] = 1;
  out[MAVG_PLAN_WGRAD_MERGED] = st->wgrad_merged ? 1 : 0;
  out[MAVG_PLAN_FWD_WITH_WGRAD] = st->fuse_upto;
  for (int l = 1; l <= st->fuse_upto; ++l) {
    out[MAVG_PLAN_FWD_RUN_TILES + l - 1] = st->wgrad_f[l].chunk;
    out[MAVG_PLAN_FWD_WHOLE_ROWS + l - 1] = st->wgrad_f[l].whole_rows;
  }
  for (int l = 1; l <= MAVG_MAX_LAYERS; ++l)
    if (st->dense[l].ok) out[MAVG_PLAN_DENSE_FIRST_STEP] |= 1 << (l - 1);
}

namespace {
ShadowArgs copy_args(const mavg_ctx* c, int64_t* most) {
  const TcLayout& t = ((const TcState*)c->mlp)->lay;
  ShadowArgs a{};
  *most = 0;
  for (int l = 1; l <= c->cfg.n_layers; ++l) {
    const MlpLayer& ly = c->layers[l - 1];
    a.w_off[l - 1] = ly.w_off;
    a.total[l - 1] = (int64_t)ly.in * ly.out;
    a.sh_off[l - 1] = t.sh_off[l - 1];
    *most = std::max(*most, a.total[l - 1]);
  }
  return a;
}

// The learners' bf16 copies (copy 0 of the doubled layer), which factored steps leave behind unwritten.
cudaError_t rebuild_copies(mavg_ctx* c) {
  const TcLayout& t = ((const TcState*)c->mlp)->lay;
  int64_t most = 0;
  const ShadowArgs a = copy_args(c, &most);
  const int gx = (int)std::min<int64_t>((most + 1023) / 1024, std::max(1, c->sm_count * 16 / c->cfg.P));
  prof_begin(c, MAVG_K_AUX);
  k_copies_from_replicas<<<dim3((unsigned)gx, (unsigned)c->cfg.n_layers, (unsigned)c->cfg.P), 256, 0, c->stream>>>(
      c->buf.replicas, c->buf.replica_stride, (__nv_bfloat16*)ws_ptr(c, t.w16), t.n16, a);
  prof_end(c);
  return cudaGetLastError();
}
}  // namespace

cudaError_t tc_refresh_shared_operands(mavg_ctx* c) {
  const TcLayout& t = ((const TcState*)c->mlp)->lay;
  int64_t most = 0;
  const ShadowArgs a = copy_args(c, &most);
  const int gx = (int)std::min<int64_t>((most + 255) / 256, (int64_t)c->sm_count * 4);
  prof_begin(c, MAVG_K_AUX);
  k_shadow_from_global<<<dim3((unsigned)gx, (unsigned)c->cfg.n_layers), 256, 0, c->stream>>>(
      c->buf.global_w, (__nv_bfloat16*)ws_ptr(c, t.w16g), a);
  prof_end(c);
  return cudaGetLastError();
}

cudaError_t tc_local_steps(mavg_ctx* c, int64_t round) {
  if (c->replicas_equal_global && (tc_factored(c) || tc_rebuilt(c))) {
    cudaError_t e = tc_factored(c) ? fac_local_steps(c, round) : reb_local_steps(c, round);
    if (e != cudaSuccess) return e;
    tc_set_w16_cur(c, kW16Stale);
    c->replicas_equal_global = false;
    return cudaSuccess;
  }
  for (int k = 1; k <= c->cfg.K; ++k) {
    cudaError_t e = tc_step(c, round, k);
    if (e != cudaSuccess) return e;
    c->replicas_equal_global = false;
  }
  return cudaSuccess;
}

// One local step of all learners.  Dependencies inside a step:
//   gather -> fwd_1 -> ... -> fwd_L (+loss) -> dgrad_L -> ... -> dgrad_2 -> wgrad_1
//   wgrad_l (l >= 2) needs dZ_l and must follow dgrad_l, which still reads W_l; it does not feed
//   anything else of this step, so it runs on a side stream beside the rest of the chain.
//   The gather of the next step touches no weights; it runs on a second side stream into the
//   other of two batch buffers as soon as that buffer's last reader (wgrad_1 of the step before
//   last) is done.
// With `overlap` false (profiled runs) everything is issued in order on the main stream.
cudaError_t tc_step(mavg_ctx* c, int64_t round, int step) {
  TcState* st = (TcState*)c->mlp;
  const TcLayout& t = st->lay;
  const mavg_config& cfg = c->cfg;
  const int L = cfg.n_layers, K = cfg.K;
  char* ws = (char*)c->buf.workspace;
  auto bfp = [&](size_t off) { return (__nv_bfloat16*)(ws + off); };
  int32_t* idx = (int32_t*)ws_ptr(c, c->ws.idx);
  int32_t* labels = (int32_t*)ws_ptr(c, c->ws.labels);
  const bool shared_w = c->replicas_equal_global;   // first step after a (re-)broadcast
  const MomArgs mom = mom_args(c, shared_w);
  const bool overlap = !c->profiling;
  const bool fused_tail = st->tail_ok && c->schedule == 0;
  bool tail_on_side = false;
  const bool merged = st->wgrad_merged && c->schedule == 0;
  // Forward products of the NEXT step ride along with this step's weight-gradient launches of
  // layers 1..ride (default schedule, those launches standing alone, a next step in this call);
  // the step after finds the activations of its first fwd_done layers in place.
  const int ride = (c->schedule == 0 && !merged && step < K) ? st->fuse_upto : 0;
  const int done = step == 1 ? 0 : st->fwd_done;
  st->fwd_done = 0;
  const int was_split = step == 1 ? 0 : st->split_done;
  st->split_done = 0;
  auto split_of = [&](int l, bool out) {
    WgradSplit sp;
    sp.in = l <= was_split && t.lo_stride[l] > 0;
    sp.out = out && t.lo_stride[l] > 0;
    if (sp.in || sp.out) {
      sp.lo = &st->lo16[l];
      sp.master = c->buf.replicas + c->layers[l - 1].w_off;
      sp.in_cols = c->layers[l - 1].in;
    }
    return sp;
  };
  // activation buffers of this step and of the next
  const int ab = st->fuse_upto >= 1 ? (step & 1) : 0;
  auto act_of = [&](int l, int set) { return bfp(set ? t.act_b[l] : t.act[l]); };
  auto act_t_of = [&](int l, int set) { return bfp(set ? t.act_t_b[l] : t.act_t[l]); };
  auto act_in = [&](int l) -> const CUtensorMap& { return ab ? st->act_in_b[l] : st->act_in[l]; };
  auto act_in_t = [&](int l) -> const CUtensorMap& { return ab ? st->act_in_t_b[l] : st->act_in_t[l]; };
  auto act_in_ks = [&](int l) -> const CUtensorMap& { return ab ? st->act_in_ks_b[l] : st->act_in_ks[l]; };
  // Weight gradients of the last two layers beside the remaining dgrad products (their dZ comes
  // out of the fused last-layer kernel): layer L-1 then writes the other of its two bf16 copies,
  // because dgrad through it still reads the current one.
  if (st->w16_cur == kW16Stale) {
    if (!shared_w) {
      cudaError_t er = rebuild_copies(c);
      if (er != cudaSuccess) return er;
    }
    st->w16_cur = 0;
  }
  const bool split_wg = merged && fused_tail && st->wgrad_beside && overlap && L >= 3 && st->dbl_layer == L - 1;
  const int rd = st->w16_cur;                                  // copy read in this step
  const int wr = split_wg ? (shared_w ? 0 : 1 - rd) : rd;      // copy written in this step
  auto w_k = [&](int l) -> const CUtensorMap& {
    return (l == st->dbl_layer && rd == 1) ? st->w_b : st->w[l]; };
  auto w_mn = [&](int l) -> const CUtensorMap& {
    return (l == st->dbl_layer && rd == 1) ? st->w_mn_b : st->w_mn[l]; };
  auto w_st = [&](int l) -> const CUtensorMap* {
    return (l == st->dbl_layer && wr == 1) ? &st->w16_st_b : &st->w16_st[l]; };
  const int xb = step & 1;                          // batch buffer of this step
  cudaStream_t main_s = c->stream;
  auto layer_ref = [&](int l) {
    WgradLayerRef r{};
    r.plan = &st->wgrad[l];
    r.dzt = &st->dz_t[l];
    r.at = l == 1 ? &st->x_in_t[xb] : &act_in_t(l);
    r.w32 = &st->w32[l];
    r.w16 = w_st(l);
    r.w32_shared = shared_w ? &st->w32g[l] : nullptr;
    r.u32 = st->wgrad_mom ? &st->u32[l] : nullptr;
    return r;
  };

  cudaError_t e;
#define TC_TRY(call) do { if ((e = (call)) != cudaSuccess) { c->stream = main_s; return e; } } while (0)

  // labels and indices are per step as well: they live beside the batch buffer they belong to
  int32_t* idx_b = idx;
  int32_t* labels_b = labels;
  if (step == 1) st->gathered_step = 0;
  if (st->gathered_step == step) {
    // the launch-by-launch form gathered this step's batch before the previous step's layer-1
    // weight gradient, which read it
  } else if (step == 1 || !overlap) {
    TC_TRY(launch_sample_gather(c, round, step, idx_b, labels_b, bfp(t.xg[xb]), bfp(t.xt[xb])));
  } else {
    // issued during the previous step on the gather stream
    TC_TRY(cudaStreamWaitEvent(main_s, st->ev_gather_done, 0));
  }

  for (int l = 1; l <= L; ++l) {
    StepOperands o{};
    o.l = l; o.step = step;
    o.shared_w = shared_w;
    o.w = shared_w ? &st->wg[l] : &w_k(l);
    o.in = l == 1 ? &st->x_in[xb] : &act_in(l);
    o.labels = labels_b;
    o.mom = mom;
    if (l <= done) {
      // A_l of this step came out of the previous step's weight-gradient launch of this layer
    } else if (l < L) {
      const FwdForm form = c->schedule == 0 ? fwd_form(st, l, shared_w) : FwdForm::TILES;
      if (form == FwdForm::DENSE) o.in = &st->in2d[l][l == 1 ? xb : ab];   // the batch rows of all learners
      else if (form == FwdForm::SPLIT) o.in = l == 1 ? &st->x_in_ks[xb] : &act_in_ks(l);
      o.out_bm = act_of(l, ab); o.out_mb = act_t_of(l, ab);
      TC_TRY(forward(c, o));
    } else if (fused_tail) {
      // last layer forward, loss, dZ_L and dgrad_L in one CUDA-core kernel
      o.a_bm = L >= 2 ? act_of(L - 1, ab) : bfp(t.xg[xb]);
      o.w16 = (shared_w ? bfp(t.w16g) : bfp(t.w16)) + t.sh_off[L - 1];
      o.w16_stride = shared_w ? 0 : t.n16;
      if (L >= 2) { o.out_bm = bfp(t.dz[L - 1]); o.out_mb = bfp(t.dz_t[L - 1]); }
      const TailLaunch tl = tail_launch(c, o);
      TC_TRY(launch_tail_fused(c, tl));
      // bias steps and loss: beside the backward pass, joined at the end of the step
      if (overlap) {
        TC_TRY(cudaEventRecord(st->ev_fork, main_s));
        TC_TRY(cudaStreamWaitEvent(st->s_wgrad, st->ev_fork, 0));
        c->stream = st->s_wgrad;
        if (split_wg) {
          // the last two layers' weight gradients first (they are on the way of the next
          // step), leaving the SMs of the dgrad tiles alone; then the bias steps and the loss
          WgradLayerRef refs[2] = {layer_ref(L), layer_ref(L - 1)};
          const int busy = cfg.P * st->dgrad[L - 1].m_tiles;
          const int cap = c->sm_count - busy >= 32 ? c->sm_count - busy : 0;
          TC_TRY(launch_wgrad_multi(c, 2, refs, mom, cap));
        }
        TC_TRY(launch_tail_finish(c, tl));
        c->stream = main_s;
        tail_on_side = true;
        TC_TRY(cudaEventRecord(st->ev_tail_done, st->s_wgrad));
      } else {
        TC_TRY(launch_tail_finish(c, tl));
      }
    } else {
      o.dz_bm = bfp(t.dz[L]);
      TC_TRY(last_layer(c, o));
    }
  }
  // the labels of this step have been consumed: the next step's gather may run now
  if (overlap && step < K) {
    const int nb = (step + 1) & 1;
    TC_TRY(cudaEventRecord(st->ev_fork, main_s));
    TC_TRY(cudaStreamWaitEvent(st->s_gather, st->ev_fork, 0));
    if (step >= 2) TC_TRY(cudaStreamWaitEvent(st->s_gather, st->ev_x_free[nb], 0));
    c->stream = st->s_gather;
    TC_TRY(launch_sample_gather(c, round, step + 1, idx_b, labels_b, bfp(t.xg[nb]), bfp(t.xt[nb])));
    c->stream = main_s;
    TC_TRY(cudaEventRecord(st->ev_gather_done, st->s_gather));
  }

  bool side_used = tail_on_side, lo_on_w1_read = false;
  for (int l = L; l >= 1; --l) {
    const MlpLayer& ly = c->layers[l - 1];
    if (l > 1 && !(fused_tail && l == L)) {
      StepOperands o{};
      o.l = l; o.step = step;
      o.shared_w = shared_w;
      o.w = shared_w ? &st->wg_mn[l] : &w_mn(l);
      o.in = &st->dz[l];
      o.out_bm = bfp(t.dz[l - 1]); o.out_mb = bfp(t.dz_t[l - 1]);
      o.mask_mb = act_t_of(l - 1, ab);
      o.mom = mom;
      TC_TRY(dgrad(c, o));
    }
    const CUtensorMap& bm = l == 1 ? st->x_in_t[xb] : act_in_t(l);
    if (merged) continue;        // all layers' weight gradients follow in one launch
    if (l <= ride) continue;     // after the dgrad chain, in ascending order (below)
    // layer 1's launch writes its bf16 copy again: the low halves that lie there have to be read first
    // (the side stream takes the layers in descending order)
    if (overlap && l == 1 && lo_on_w1_read) TC_TRY(cudaStreamWaitEvent(main_s, st->ev_wgrad_done, 0));
    if (overlap && l > 1) {
      // Behind the fused last layer the side stream already follows all that its launch for layer L
      // reads.  A second dependence on the same kernel would be one more edge of the graph, and these cost
      // at its instantiation: with P = 48 1.57 ms for 113 edges, 1.07 for 105, in a first round of 3.75.
      if (!(l == L && tail_on_side)) {
        TC_TRY(cudaEventRecord(st->ev_fork, main_s));
        TC_TRY(cudaStreamWaitEvent(st->s_wgrad, st->ev_fork, 0));
      }
      c->stream = st->s_wgrad;
      TC_TRY(launch_wgrad_stream(c, st->wgrad[l], st->dz_t[l], bm, st->w32[l], *w_st(l),
                                 shared_w ? &st->w32g[l] : nullptr, &st->u32[l], mom, nullptr,
                                 split_of(l, false)));
      if (l == t.lo_on_w1 && l <= was_split) {
        TC_TRY(cudaEventRecord(st->ev_wgrad_done, st->s_wgrad));
        lo_on_w1_read = true;
      }
      c->stream = main_s;
      side_used = true;
    } else {
      TC_TRY(launch_wgrad_stream(c, st->wgrad[l], st->dz_t[l], bm, st->w32[l], *w_st(l),
                                 shared_w ? &st->w32g[l] : nullptr, &st->u32[l], mom, nullptr,
                                 split_of(l, false)));
    }
  }
  // Layers whose launch takes the next step's forward product along: layer l's needs A_{l-1} of
  // the next step, so they run in ascending order, each leaving A_l of the next step behind (in
  // the other set of activation buffers: this step's A_l is still an operand of layer l+1's
  // launch).  Layer 1 reads the next step's gathered
  // batch; only layer 1's bf16 copy has no other reader and is left unwritten.
  for (int l = 1; l <= ride; ++l) {
    const MlpLayer& ly = c->layers[l - 1];
    const int nb = (step + 1) & 1;
    if (l == 1) {
      if (overlap) {
        TC_TRY(cudaStreamWaitEvent(main_s, st->ev_gather_done, 0));
      } else {
        TC_TRY(launch_sample_gather(c, round, step + 1, idx_b, labels_b, bfp(t.xg[nb]), bfp(t.xt[nb])));
        st->gathered_step = step + 1;
      }
    }
    // the riding product adds the bias that the fused last layer steps on the side stream
    if (l == L - 1 && tail_on_side) TC_TRY(cudaStreamWaitEvent(main_s, st->ev_tail_done, 0));
    const CUtensorMap& bm = l == 1 ? st->x_in_t[xb] : act_in_t(l);
    WgradFwdNext fn{};
    fn.xn = &st->a_next[l][nb];
    fn.zpart = (float*)(ws + t.zpart);
    fn.zcount = (int*)(ws + t.zcount);
    fn.bias_off = ly.b_off;
    fn.out_rows = ly.out;
    fn.out_bm = act_of(l, nb);
    fn.out_mb = act_t_of(l, nb);
    fn.store_w16 = l > 1;
    TC_TRY(launch_wgrad_stream(c, st->wgrad_f[l], st->dz_t[l], bm, st->w32[l], *w_st(l),
                               shared_w ? &st->w32g[l] : nullptr, &st->u32[l], mom, &fn,
                               split_of(l, true)));
    st->fwd_done = l;
    st->split_done = l;
  }
  if (merged) {
    // largest layer first, so that the small ones fill the ragged end of the launch
    WgradLayerRef refs[MAVG_MAX_LAYERS];
    const int top = split_wg ? L - 2 : L;      // the last two layers already run on the side
    for (int l = 1; l <= top; ++l) refs[l - 1] = layer_ref(l);
    TC_TRY(launch_wgrad_multi(c, top, refs, mom));
  }
  st->w16_cur = wr;
  if (overlap) {
    TC_TRY(cudaEventRecord(st->ev_x_free[xb], main_s));     // wgrad_1 was the buffer's last reader
    if (side_used) {
      TC_TRY(cudaEventRecord(st->ev_wgrad_done, st->s_wgrad));
      TC_TRY(cudaStreamWaitEvent(main_s, st->ev_wgrad_done, 0));
    }
  }
#undef TC_TRY
  return cudaSuccess;
}

}  // namespace mavg
