// Factored local steps of the tensor-core MLP path (factored.cu).
//
// Within a round every learner starts from w~, so its weights after k steps are
//   W_l(k) = W~_l - gamma sum_{i<k} dZ_l(i)^T A_{l-1}(i),
// and the products of step k can be taken from w~ and the factors without forming W_l(k):
//   forward   Z = A W~^T - gamma sum_i (A A(i)^T) dZ(i)
//   dgrad     dA = dZ W~  - gamma sum_i (dZ dZ(i)^T) A(i)
// The hidden layers' weights are formed once, at the end of the call.
#pragma once
#include <cuda.h>

#include <string>
#include <vector>

#include "common.cuh"

namespace mavg {

// Byte offsets of the path's scratch.  Rows of a learner are ordered (step, slot): K * B of them.
struct FacLayout {
  int64_t kb = 0;                            // rows of a learner: fac_steps() * B
  int64_t s_ld = 0;                          // row length of the Gram arrays: kb rounded up to 64
  size_t h[MAVG_MAX_LAYERS] = {};            // A_l, l = 0..L-1: bf16 [P, kb, d_l]
  size_t g[MAVG_MAX_LAYERS + 1] = {};        // dZ_l, l = 1..L-1: bf16 [P, kb, d_l]
  // X W~_1^T, fp32 [kb, d_1] per learner, and -gamma X X^T below the step diagonal, bf16 [kb, s_ld] per
  // learner.  Where they fit they lie in the learner's rows of the replica array, on W_1, which no
  // factored step reads or writes before the last (in_rows; zbase and s1 are then byte offsets in a row).
  bool in_rows = false;
  size_t zbase = 0, s1 = 0;
  size_t s[2] = {0, 0};                      // one step's -gamma A A(i)^T and -gamma dZ dZ(i)^T: bf16 [P, B, s_ld]
  size_t labels = 0;                         // int32 [K, P, B]
  size_t w_lo[MAVG_MAX_LAYERS] = {};         // low parts of w~'s hidden layers, l = 1..L-1: bf16 [d_l, d_{l-1}]
  // rebuilt steps: the learners' weights, l = 1..L: bf16 [P, d_l, d_{l-1}].  The rows above are [steps, P, B, d_l] there,
  // dZ_L's among them (padded to 8 classes)
  size_t w_own[MAVG_MAX_LAYERS + 1] = {};
  size_t act_t[MAVG_MAX_LAYERS] = {}, dz_t = 0;   // A_l, l = 1..L-1, of the step at hand, and a dZ_l: bf16 [P, d_l, B]
  size_t end = 0;
};

// Learners per block, columns per learner and block, column tiles per learner (more than 1 with nl 1 only).
// own_gram: the product may form its Gram rows itself.
struct FacCols { int nl = 1, cols = 0, c_tiles = 1; bool own_gram = false; };

struct FacState {
  FacLayout lay;
  int K = 0;                                 // steps the scratch has room for
  int row_tile = 0;                          // rows of X per tile where all steps' rows are one operand
  char *z_ptr = nullptr, *s1_ptr = nullptr;  // zbase and s1 of learner 0; strides in elements
  int64_t z_stride = 0, s1_stride = 0;
  // How the columns of the forward product of layer l, the data gradient through it and the Gram
  // products are cut; the first two's batch operands (box 64 x cols x nl) and Gram operands (64 x cols)
  FacCols fwd[MAVG_MAX_LAYERS + 1], dgrad[MAVG_MAX_LAYERS + 1], gram;
  CUtensorMap in[MAVG_MAX_LAYERS + 1], dz_in[MAVG_MAX_LAYERS + 1];
  CUtensorMap s_f[MAVG_MAX_LAYERS + 1], s_d[MAVG_MAX_LAYERS + 1];
  // Rebuilt steps: the learners' weights (boxes of 64 x 128, 64 x 64, and to store 32 x 128) and each step's batch operands:
  // A_{l-1} and dZ_l of step k at [(k - 1) (MAVG_MAX_LAYERS + 1) + l].  fwd1, dgrad1: cuts of the first step's products, with
  // w~; own_fwd (of the first step at [1]), own_dgrad: the products are k_fac_product's, not the plain form's launches
  FacCols fwd1[MAVG_MAX_LAYERS + 1], dgrad1[MAVG_MAX_LAYERS + 1];
  bool own_fwd[2][MAVG_MAX_LAYERS + 1] = {}, own_dgrad[MAVG_MAX_LAYERS + 1] = {};
  int runs[MAVG_MAX_LAYERS + 1] = {};        // partial sums of a forward product after the first step's (0, 1: none)
  CUtensorMap w_own[MAVG_MAX_LAYERS + 1], w_own_mn[MAVG_MAX_LAYERS + 1], w_own_st[MAVG_MAX_LAYERS + 1];
  std::vector<CUtensorMap> step_in, step_dz;
  CUtensorMap w_lo[MAVG_MAX_LAYERS];         // low parts of w~'s hidden layers, box 64 x 128
  // Row arrays [P, kb, d_l]: A_l (h) and dZ_l (g) with boxes of 64 x 64 rows (_mn: features are the MMA's
  // row dimension, rows the contraction), 64 x 128 (_k) and 64 x gram.cols (_b; A_0: 64 x row_tile).
  CUtensorMap h_mn[MAVG_MAX_LAYERS], g_mn[MAVG_MAX_LAYERS + 1];
  CUtensorMap h_k[MAVG_MAX_LAYERS], g_k[MAVG_MAX_LAYERS];
  CUtensorMap h_b[MAVG_MAX_LAYERS], g_b[MAVG_MAX_LAYERS];
};

// The most steps of a call that a handle's calls may take in this form (0: never; at most the K it was made
// for), and the scratch for them from `base` on.  fac_reserved: the calls as the handle is made take it, so the
// workspace size has room for it (up to ten times the plain form's for long rounds of narrow models).
int fac_steps(const mavg_config* cfg);
bool fac_reserved(const mavg_config* cfg);
FacLayout fac_layout(const mavg_config* cfg, size_t base);
struct TcState;
// A tensor map or kernel attribute that is refused leaves the handle the plain form.
void fac_setup(mavg_ctx* c, TcState* st);
// The steps of a call that starts from w~ take the factored form.
bool fac_usable(const mavg_ctx* c);
cudaError_t fac_local_steps(mavg_ctx* c, int64_t round);

// The same of rebuilt steps (rebuild.cuh), which calls take that are not factored: the weights of every step are formed anew
// from w~, u as the call found it and the rows of all steps so far.
int reb_steps(const mavg_config* cfg);
bool reb_riding(const mavg_config* cfg);       // also where the plain form's forward products ride on its weight gradients
bool reb_reserved(const mavg_config* cfg);
FacLayout reb_layout(const mavg_config* cfg, size_t base);
void reb_setup(mavg_ctx* c, TcState* st);
bool reb_usable(const mavg_ctx* c);
cudaError_t reb_local_steps(mavg_ctx* c, int64_t round);

}  // namespace mavg
