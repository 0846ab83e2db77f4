// Declarations shared by the files of the MLP learner level (batch.cu, mlp.cu, mlp_simt.cu,
// mlp_tc.cu).
#pragma once
#include "common.cuh"

namespace mavg {

// First sample of learner j's shard, floor(j S / P); j <= 2^31 and S < 2^31: 64 bits hold the product.
__device__ __forceinline__ int64_t shard_begin(int64_t j, int P, int64_t S) {
  return (int64_t)((uint64_t)j * (uint64_t)S / (uint32_t)P);
}
// idx = lo_j + floor(u * len_j / 2^32), u = top 32 bits of the stream value (see mavg.h).
__device__ __forceinline__ int32_t sample_index(uint64_t seed, int64_t round, int j, int step,
                                                int s, int P, int64_t S) {
  const int64_t lo = shard_begin(j, P, S), hi = shard_begin((int64_t)j + 1, P, S);
  uint64_t key = fold(learner_key(seed, kTagBatch, (uint64_t)round, (uint64_t)j), (uint64_t)step);
  uint64_t u = fold(key, (uint64_t)s) >> 32;
  return (int32_t)(lo + (int64_t)((u * (uint64_t)(hi - lo)) >> 32));
}

// Where the paths of gemm_bf16 0 and 2 find the learners' models at the start of a round: in w~ while a deferred
// re-broadcast has not been carried out, in the replica array otherwise (whose rows a program may have
// edited since they were written).
inline bool starts_from_global(const mavg_ctx* c) {
  return c->replicas_equal_global && !c->replicas_materialized;
}

// batch.cu
cudaError_t launch_batch_indices(mavg_ctx* c, int64_t round, int step, int j, int32_t* idx);
cudaError_t launch_sample_gather(mavg_ctx* c, int64_t round, int step, int32_t* idx,
                                 int32_t* labels, __nv_bfloat16* out_bf, __nv_bfloat16* out_bft);

// fp32 arithmetic, or bf16 operands of any shape (mlp_simt.cu).
size_t simt_workspace_bytes(const mavg_config* cfg, size_t base, size_t* act_off, size_t* least);
mavg_status simt_setup(mavg_ctx* c);      // once per handle
void simt_teardown(mavg_ctx* c);
cudaError_t simt_local_steps(mavg_ctx* c, int64_t round);    // all K of them

// Small models on the CUDA cores (mlp_small.cu): all local steps of a round in one launch.
bool small_always(const mavg_config* cfg);   // taken whenever the device grants the launch
void small_setup(mavg_ctx* c);            // once per handle: c->small_splits > 0 where it is used
cudaError_t small_local_steps(mavg_ctx* c, int64_t round);

// Tensor-core path (mlp_tc.cu): tcgen05 GEMMs fed by TMA.
bool tc_shapes_ok(const mavg_config* cfg, std::string* why);
// least: what the path cannot do without (a smaller figure where factored steps would need more).
size_t tc_workspace_bytes(const mavg_config* cfg, size_t base, size_t* act_off, size_t* least);
mavg_status tc_setup(mavg_ctx* c);
void tc_teardown(mavg_ctx* c);
cudaError_t tc_refresh_shared_operands(mavg_ctx* c);
cudaError_t tc_step(mavg_ctx* c, int64_t round, int step);
cudaError_t tc_local_steps(mavg_ctx* c, int64_t round);      // all K of them

// Fused last layer on CUDA cores (tail_fused.cu): forward, loss, dZ_L, dgrad through the layer
// and the bias steps of the last two layers, for the tensor-core path's bf16 operands.
struct TailLaunch {
  const __nv_bfloat16* a_bm;     // A_{L-1} [P, B, in]
  const __nv_bfloat16* w16;      // bf16 W_L of learner 0
  int64_t w16_stride;            // elements between learners' copies (0: shared copy)
  bool shared_w;                 // biases are read from w~ (first step of a round)
  const int32_t* labels;
  float* loss_out;
  int loss_stride;
  __nv_bfloat16* dz_t;           // out: dZ_L^T [P, C, B], and where given dZ_L [P, B, cpad]
  __nv_bfloat16* dz_bm;
  int cpad;
  __nv_bfloat16* dzp_bm;         // out: dZ_{L-1} [P, B, in] and its transpose [P, in, B]
  __nv_bfloat16* dzp_mb;
  float* part;                   // scratch of tail_fused_part_bytes()
  MomArgs mom;
};
bool tail_fused_supported(const mavg_config* cfg);
size_t tail_fused_part_bytes(const mavg_config* cfg);
cudaError_t tail_fused_prepare();
cudaError_t launch_tail_fused(mavg_ctx* c, const TailLaunch& t);    // the products, dZ, partial sums
cudaError_t launch_tail_finish(mavg_ctx* c, const TailLaunch& t);   // bias steps and loss from the partials

void tc_reset_counters(mavg_ctx* c);          // after an abandoned device-side wait
bool tc_factored(const mavg_ctx* c);
bool tc_rebuilt(const mavg_ctx* c);
void tc_step_plan(mavg_ctx* c, int32_t* out);  // entries of mavg_plan_entry
// State of the learners' bf16 copies between calls: which copy of the doubled layer is current, or
// kW16Stale: none (factored steps keep none; the next step that reads them writes them anew).
constexpr int kW16Stale = -1;
int tc_get_w16_cur(mavg_ctx* c);
void tc_set_w16_cur(mavg_ctx* c, int cur);

inline bool use_tensor_cores(const mavg_config* cfg) { return cfg->gemm_bf16 == 1; }

}  // namespace mavg
