// Learner level of Algorithm 1 with the stochastic gradient replaced by seeded variates:
//   w^j <- w^j - gamma g(seed, n, j, k, i),  k = 1..K,
// g an Irwin-Hall(4) variate of standard deviation sigma built from one SplitMix64 stream value
// (see mavg.h).  The K steps are applied in order to a value held in registers, so one pass over
// the replicas (8 bytes per element and learner) serves the whole round; the per-step rounding is
// the same as K separate passes.  The first pass after a (re-)broadcast reads w~ in place of
// every w^j ("set w^j = w~"), so the P copies need not exist before it.
#include "common.cuh"

namespace mavg {
namespace {

// The variate of element i at a step with key `key`: mix64(key + (i+1) G), its four 16-bit lanes
// summed, minus 131070, times c (mavg.h).  What bounds the pass is the integer pipes: about 25
// instructions of arithmetic per variate (29.3 executed, keys and loop included) -- a 64-bit addition, three xor-shifts of 4, two 64 x 64 -> 64 bit
// products of 3 multiply-adds, two dot products, three float operations -- of which the shifts and
// logic operations (ALU pipe) and the multiply-adds (FMA pipe, 64-bit ones at a quarter of the
// rate) are about 24 cycles per warp each.  Hence the 64-bit value is kept as two words:
//  - the carry of the addition is a compare and a predicated increment, which the scheduler may
//    place on either pipe, where a 64-bit add occupies the multiply pipe for four cycles;
//  - the lane sum starts from the bits of 2^23, so that the sum's bits already are the float
//    2^23 + sum and one exact subtraction takes the place of an integer-to-float conversion.
// With four steps unrolled, 5.12e8 x 12.8 variates in 6.16 ms against 6.71 ms for the plain
// 64-bit form (n = 6.4 M, P = 16, K = 64: 0.98e12 -> 1.06e12 variates/s).
struct U64 { uint32_t lo, hi; };

__device__ __forceinline__ U64 split(uint64_t v) { return {(uint32_t)v, (uint32_t)(v >> 32)}; }

__device__ __forceinline__ U64 add(U64 a, uint64_t b) {
  const uint32_t bl = (uint32_t)b;
  U64 r{a.lo + bl, a.hi + (uint32_t)(b >> 32)};
  if (r.lo < bl) r.hi += 1u;
  return r;
}
template <int S>
__device__ __forceinline__ U64 xor_shift(U64 z) {   // z ^ (z >> S), S < 32
  return {z.lo ^ __funnelshift_r(z.lo, z.hi, S), z.hi ^ (z.hi >> S)};
}
template <uint64_t C>
__device__ __forceinline__ U64 mul(U64 z) {
  const uint64_t p = (uint64_t)z.lo * (uint32_t)C;
  return {(uint32_t)p, z.hi * (uint32_t)C + (z.lo * (uint32_t)(C >> 32) + (uint32_t)(p >> 32))};
}
__device__ __forceinline__ float variate(U64 z, float c) {
  z = mul<0xBF58476D1CE4E5B9ull>(xor_shift<30>(z));
  z = mul<0x94D049BB133111EBull>(xor_shift<27>(z));
  z = xor_shift<31>(z);
  const uint32_t s = __dp2a_lo(z.hi, 0x0101u, __dp2a_lo(z.lo, 0x0101u, 0x4B000000u));
  return (__uint_as_float(s) - (8388608.f + 131070.f)) * c;
}

// One local step on four consecutive elements, the first of which has counter c0 = (i+1) G.
template <bool MOM>
__device__ __forceinline__ void local_step4(float4& w, float4& u, uint64_t key, uint64_t c0,
                                            float c, float gamma, float beta) {
  const U64 z = add(split(key), c0);
  const float g0 = variate(z, c), g1 = variate(add(z, kGamma), c);
  const float g2 = variate(add(z, 2 * kGamma), c), g3 = variate(add(z, 3 * kGamma), c);
  if (MOM) {
    msgd(w.x, u.x, g0, gamma, beta);
    msgd(w.y, u.y, g1, gamma, beta);
    msgd(w.z, u.z, g2, gamma, beta);
    msgd(w.w, u.w, g3, gamma, beta);
  } else {
    w.x = fmaf(-gamma, g0, w.x);
    w.y = fmaf(-gamma, g1, w.y);
    w.z = fmaf(-gamma, g2, w.z);
    w.w = fmaf(-gamma, g3, w.w);
  }
}
template <bool MOM, int U = 4>
__device__ __forceinline__ void local_steps4(float4& w, float4& u, const uint64_t* keys, int K,
                                             uint64_t c0, float c, float gamma, float beta) {
#pragma unroll U
  for (int k = 0; k < K; ++k) local_step4<MOM>(w, u, keys[k], c0, c, gamma, beta);
}
// The same on one element (the ragged end of the vector).
template <bool MOM>
__device__ __forceinline__ void local_steps1(float& w, float& u, const uint64_t* keys, int K,
                                             uint64_t c0, float c, float gamma, float beta) {
  for (int k = 0; k < K; ++k) {
    const float g = variate(add(split(keys[k]), c0), c);
    if (MOM) msgd(w, u, g, gamma, beta);
    else w = fmaf(-gamma, g, w);
  }
}

// grid = (x, P); dynamic shared memory holds the K step keys of learner blockIdx.y.
// MOM: learner-level momentum, u^j read (unless mom.read_u == 0) and written once per pass like w^j.
// U: steps unrolled, 4 (40 registers, six blocks on an SM) or, for one or two steps, where HBM counts as much as
// the variates, 1 (32 registers, all eight): n = 25.6 M, P = 16, K = 1 570 us against 670, K = 2 982 against
// 992, K = 3 1402 against 1380.
template <bool MOM, int U>
__global__ void __launch_bounds__(256, U == 1 ? 8 : 6)
k_pseudograd_steps(float* rep, int64_t stride, const float* src, int64_t src_stride, int64_t n,
                   int K, uint64_t seed, int64_t round, int k_first, float c, float gamma,
                   const MomArgs mom) {
  extern __shared__ uint64_t keys[];
  const int j = blockIdx.y;
  const uint64_t lk = learner_key(seed, kTagPseudoGrad, (uint64_t)round, (uint64_t)j);
  for (int k = threadIdx.x; k < K; k += blockDim.x) keys[k] = fold(lk, (uint64_t)(k_first + k));
  __syncthreads();
  float* row = rep + (size_t)j * stride;
  float4* row4 = reinterpret_cast<float4*>(row);
  const float* in = src + (size_t)j * src_stride;
  const float4* in4 = reinterpret_cast<const float4*>(in);
  const int64_t n4 = n >> 2;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  float* urow = MOM ? mom.u + (size_t)j * mom.u_stride : nullptr;
  float4* urow4 = reinterpret_cast<float4*>(urow);
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += step) {
    float4 w = src_stride ? __ldcs(in4 + q) : __ldg(in4 + q);
    float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MOM && mom.read_u) u = __ldcs(urow4 + q);
    local_steps4<MOM, U>(w, u, keys, K, (uint64_t)(4 * q + 1) * kGamma, c, gamma, mom.beta);
    __stcs(row4 + q, w);
    if (MOM) __stcs(urow4 + q, u);
  }
  if (blockIdx.x == 0 && threadIdx.x < (n & 3)) {
    const int64_t i = (n4 << 2) + threadIdx.x;
    float w = in[i];
    float u = (MOM && mom.read_u) ? urow[i] : 0.f;
    local_steps1<MOM>(w, u, keys, K, (uint64_t)(i + 1) * kGamma, c, gamma, mom.beta);
    row[i] = w;
    if (MOM) urow[i] = u;
  }
}

// A whole round: the K local steps of all P learners and the meta-update.  A thread takes four
// elements through learner 0's K steps, then learner 1's, ..., adds the differences w^j - w~ in
// the same ascending order as the meta-update kernels and finishes the update itself, so the
// replicas are not read back: per element (4P + 16) bytes where the two passes move (8P + 16)
// with deferred copies (the learners' models are written) and (12P + 16) without (only the P
// copies of the new w~ are).  Bounds: at K = 1 HBM (2.05 GB = 0.31 ms at n = 25.6 M, P = 16) and the
// variates (0.38 ms) about equally, the variates beyond.  Measured there, deferred copies: K = 1
// 492 us a round against 887 for the two passes, K = 64 25.5 ms against 25.8.
// One quad per thread and no loop over the grid: the blocks' ends are spread over the launch.  The
// last n % 4 elements have a block of their own, so that their serial P x K steps run beside the
// rest.  K1: K = 1, the loop over the learners is unrolled instead of the one over the steps.
// Dynamic shared memory holds the P x K step keys.
template <bool MOM, bool K1>
__global__ void __launch_bounds__(256)
k_pseudograd_round(float* rep, int64_t stride, bool from_global, float* __restrict__ gw,
                   float* __restrict__ gv, int64_t n, int P, int K, uint64_t seed, int64_t round,
                   float c, float gamma, float mu, float zeta, float inv_p, bool read_v, bool bcast,
                   const MomArgs mom) {
  extern __shared__ uint64_t keys[];
  for (int t = threadIdx.x; t < P * K; t += blockDim.x)
    keys[t] = fold(learner_key(seed, kTagPseudoGrad, (uint64_t)round, (uint64_t)(t / K)),
                   (uint64_t)(t % K + 1));
  __syncthreads();
  const int64_t n4 = n >> 2;
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n4) {
    const float4 wt = __ldcs(reinterpret_cast<const float4*>(gw) + q);
    const uint64_t c0 = (uint64_t)(4 * q + 1) * kGamma;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll K1 ? 4 : 1
    for (int j = 0; j < P; ++j) {
      float4* row4 = reinterpret_cast<float4*>(rep + (size_t)j * stride) + q;
      float4* u4 = MOM ? reinterpret_cast<float4*>(mom.u + (size_t)j * mom.u_stride) + q : nullptr;
      float4 w = from_global ? wt : __ldcs(row4);
      float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
      if (MOM && mom.read_u) u = __ldcs(u4);
      if (K1) local_step4<MOM>(w, u, keys[j], c0, c, gamma, mom.beta);
      else local_steps4<MOM>(w, u, keys + j * K, K, c0, c, gamma, mom.beta);
      acc.x += w.x - wt.x;
      acc.y += w.y - wt.y;
      acc.z += w.z - wt.z;
      acc.w += w.w - wt.w;
      if (!bcast) __stcs(row4, w);
      if (MOM) __stcs(u4, u);
    }
    float4 vt = make_float4(0.f, 0.f, 0.f, 0.f);
    if (read_v) vt = __ldcs(reinterpret_cast<const float4*>(gv) + q);
    float4 vn, wn;
    vn.x = fmaf(mu, vt.x, zeta * (acc.x * inv_p));
    vn.y = fmaf(mu, vt.y, zeta * (acc.y * inv_p));
    vn.z = fmaf(mu, vt.z, zeta * (acc.z * inv_p));
    vn.w = fmaf(mu, vt.w, zeta * (acc.w * inv_p));
    wn.x = wt.x + vn.x; wn.y = wt.y + vn.y; wn.z = wt.z + vn.z; wn.w = wt.w + vn.w;
    __stcs(reinterpret_cast<float4*>(gv) + q, vn);
    __stcs(reinterpret_cast<float4*>(gw) + q, wn);
    if (bcast)
      for (int j = 0; j < P; ++j) __stcs(reinterpret_cast<float4*>(rep + (size_t)j * stride) + q, wn);
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x < (n & 3)) {
    const int64_t i = (n4 << 2) + threadIdx.x;
    const float wt = gw[i];
    float acc = 0.f;
    for (int j = 0; j < P; ++j) {
      float* wp = rep + (size_t)j * stride + i;
      float* up = MOM ? mom.u + (size_t)j * mom.u_stride + i : nullptr;
      float w = from_global ? wt : *wp, u = (MOM && mom.read_u) ? *up : 0.f;
      local_steps1<MOM>(w, u, keys + j * K, K, (uint64_t)(i + 1) * kGamma, c, gamma, mom.beta);
      acc += w - wt;
      if (!bcast) *wp = w;
      if (MOM) *up = u;
    }
    const float vn = fmaf(mu, read_v ? gv[i] : 0.f, zeta * (acc * inv_p));
    const float wn = wt + vn;
    gv[i] = vn;
    gw[i] = wn;
    if (bcast)
      for (int j = 0; j < P; ++j) rep[(size_t)j * stride + i] = wn;
  }
}

float variate_scale(const mavg_ctx* c) {
  const double var_lane = (65536.0 * 65536.0 - 1.0) / 12.0;
  return (float)((double)c->cfg.pseudo_grad_sigma / sqrt(4.0 * var_lane));
}

constexpr int kMaxRoundKeys = 4096;   // P x K step keys of a fused round: 32 KB of shared memory

// Blocks of 64 threads in a fused round, where the vector gives every SM only a few blocks of 256.
bool small_blocks(const mavg_ctx* c) { return (c->cfg.n >> 2) < (int64_t)c->sm_count * 2048; }

}  // namespace

cudaError_t launch_pseudograd_steps(mavg_ctx* c, int64_t round) {
  const int64_t n = c->cfg.n;
  const int P = c->cfg.P, K = c->cfg.K;
  const float scale = variate_scale(c);
  constexpr int kMaxFused = 2048;  // step keys per launch (16 KB of shared memory)
  int64_t blocks_x = ((n >> 2) + 255) / 256;
  int64_t cap = ((int64_t)c->sm_count * 8 + P - 1) / P;
  if (blocks_x > cap) blocks_x = cap;
  if (blocks_x < 1) blocks_x = 1;
  for (int k0 = 0; k0 < K; k0 += kMaxFused) {
    int kc = K - k0 < kMaxFused ? K - k0 : kMaxFused;
    dim3 grid((unsigned)blocks_x, (unsigned)P);
    const bool from_global = c->replicas_equal_global;
    const MomArgs mom = mom_args(c, from_global);
    auto kernel = mom.u ? (kc <= 2 ? k_pseudograd_steps<true, 1> : k_pseudograd_steps<true, 4>)
                        : (kc <= 2 ? k_pseudograd_steps<false, 1> : k_pseudograd_steps<false, 4>);
    prof_begin(c, MAVG_K_PSEUDOGRAD);
    kernel<<<grid, 256, (size_t)kc * sizeof(uint64_t), c->stream>>>(
        c->buf.replicas, c->buf.replica_stride, from_global ? c->buf.global_w : c->buf.replicas,
        from_global ? 0 : c->buf.replica_stride, n, kc, c->cfg.seed, round, k0 + 1, scale,
        c->cfg.local_lr, mom);
    prof_end(c);
    c->replicas_equal_global = false;
    c->replicas_materialized = true;
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The fused round has n / 4 threads, each with P x K serial steps, where the local steps on their own have
// P times as many: with more steps per learner the vector has to be longer for it to pay.  Learner momentum
// adds a read per learner to the serial part.  Blocks of 64 threads (launch_pseudograd_round) with more than
// 2048 step keys leave too few warps on an SM.  Measured, us a round with deferred copies, one launch / two
// (n = 76 000 is 512 per SM; the eager form differs by a few per cent in favour of one launch):
//   K = 1: n = 76 000 P = 16 6.7 / 12.7, P = 256 50 / 94; n = 303 000 P = 1000 395 / 696;
//   K = 2: n = 76 000 P = 256 103 / 95; n = 100 000 P = 64 35.2 / 35.3, P = 256 127 / 142;
//   K = 3: n = 100 000 P = 64 47 / 43; n = 152 000 P = 32 25 / 29;
//   K = 4: n = 76 000 P = 16 14.9 / 16.8, P = 64 50 / 39; n = 152 000 P = 256 228 / 258;
//   K = 8: n = 606 000 P = 16 89 / 90;  K = 24: n = 606 000 P = 16 251 / 240, n = 2.4 M 932 / 955;
//   K = 38: n = 606 000 P = 16 394 / 371, n = 909 000 575 / 554;  K = 64: n = 1.2 M P = 5 397 / 412;
//   P x K = 4096: n = 606 000, K = 256 2833 / 2440, K = 8 2986 / 2866; n = 2.4 M, K = 64 9767 / 10776;
//   with momentum, K = 1: n = 76 000 P = 64 27.1 / 27.1, P = 256 179 / 118; n = 303 000 P = 256 241 / 260;
//   K = 3: n = 76 000 P = 16 15.2 / 15.7, P = 64 51 / 39;  K = 4: n = 76 000 P = 16 18.9 / 16.8; n = 152 000
//   P = 16 22.9 / 22.9, P = 64 79 / 72; n = 303 000 P = 64 124 / 138.
// At these lines the two are within 5 % of one another but for n = 455 000, P = 32, K = 4 (83 / 76).
bool pseudograd_round_fused(const mavg_ctx* c) {
  if (c->cfg.objective != MAVG_OBJ_PSEUDOGRAD) return false;
  const int64_t n = c->cfg.n, sms = c->sm_count, K = c->cfg.K, keys = c->cfg.P * K;
  if (keys > (K <= 3 || !small_blocks(c) ? kMaxRoundKeys : kMaxRoundKeys / 2)) return false;
  if (K > 4) return n >= (K <= 24 ? 4096 : 6144) * sms;
  if (c->cfg.learner_momentum != 0.f)
    return n >= 2048 * sms || (n >= 1024 * sms && keys <= 64) ||
           (n >= 512 * sms && keys <= (K == 4 ? 32 : 48));
  return n >= (K == 1 ? 512 : K == 2 ? 640 : 1024) * sms || (n >= 512 * sms && keys <= 64);
}

cudaError_t launch_pseudograd_round(mavg_ctx* c, int64_t round) {
  const int64_t n4 = c->cfg.n >> 2;
  const int threads = small_blocks(c) ? 64 : 256;
  const unsigned grid = (unsigned)((n4 + threads - 1) / threads + ((c->cfg.n & 3) ? 1 : 0));
  const size_t smem = (size_t)c->cfg.P * c->cfg.K * sizeof(uint64_t);
  const bool from_global = c->replicas_equal_global;
  const bool bcast = !c->cfg.defer_broadcast;
  const MomArgs mom = mom_args(c, from_global);
  auto kernel = mom.u ? (c->cfg.K == 1 ? k_pseudograd_round<true, true> : k_pseudograd_round<true, false>)
                      : (c->cfg.K == 1 ? k_pseudograd_round<false, true> : k_pseudograd_round<false, false>);
  prof_begin(c, MAVG_K_PSEUDOGRAD);
  kernel<<<grid, threads, smem, c->stream>>>(
      c->buf.replicas, c->buf.replica_stride, from_global, c->buf.global_w, c->buf.momentum,
      c->cfg.n, c->cfg.P, c->cfg.K, c->cfg.seed, round, variate_scale(c), c->cfg.local_lr,
      c->cfg.mu, c->cfg.block_lr, 1.0f / (float)c->cfg.P, c->cfg.mu != 0.f, bcast, mom);
  prof_end(c);
  c->replicas_equal_global = true;
  c->replicas_materialized = bcast;
  return cudaGetLastError();
}

}  // namespace mavg
