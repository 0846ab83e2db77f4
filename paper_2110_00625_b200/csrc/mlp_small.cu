// Small models on the CUDA cores: all K local steps of a learner in one launch.  A learner's weights,
// minibatch and activations fit in an SM's shared memory, so a step is a few microseconds of
// work where a launch per product leaves a chain of latencies.  A learner is a cluster of S
// blocks, each holding a copy of the weights:
//   - forward, loss and data gradients are split by batch rows (groups of four);
//   - what the weight gradients need of a row -- its activations and dZ -- is written to every
//     block of the cluster as it is produced;
//   - weight gradients, bias gradients and the SGD step are split by output rows of a layer, the
//     updated weights again written to every block.
// Two cluster barriers per step.  Arithmetic: fp32 FMAs, operands rounded to bf16 first with QUANT.
// Bound by the latency of dependent instructions: 32-64-10, P = 4, K = 4, B = 32 takes 6.2 us a step, of which the forward
// products, loss and data gradient are 3.5 and the weight gradients 1.2, the rest barriers.  Logits, loss and dZ of a row
// stay in one warp (two phases and a barrier before), and the weight gradients of all layers are one list of tasks for all
// twelve warps, biases behind them (8 us a step with a phase per layer and per bias): rounds of that model 50 -> 44 us,
// of 24 models drawn around it 1.11 times faster in the geometric mean.
#include <algorithm>

#include "mlp.cuh"
#include "tc_ptx.cuh"

namespace mavg {
namespace {

__device__ __forceinline__ float qbf(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
template <bool QUANT>
__device__ __forceinline__ float operand(float v) { return QUANT ? qbf(v) : v; }
template <bool QUANT>
__device__ __forceinline__ float4 operand4(float4 v) {
  return make_float4(operand<QUANT>(v.x), operand<QUANT>(v.y), operand<QUANT>(v.z), operand<QUANT>(v.w));
}

constexpr int kCompute = 256, kGather = 128;   // threads: 8 warps compute, 4 fetch the next minibatch
constexpr int kWarps = (kCompute + kGather) / 32;
constexpr size_t kSmallSmem = 220 * 1024;

// Shared memory, offsets in floats.  Activations and dZ are [feature][pitch] with the batch row
// innermost, so that a thread takes four rows per load; pitch / 4 is odd, which keeps 16-byte reads
// along the features free of bank conflicts.  W_l is [out][in | 1]: odd rows, for reads along
// either dimension.
struct SmallLayout {
  int pitch;
  int x[2], label[2], loss;
  int w[MAVG_MAX_LAYERS + 1], b[MAVG_MAX_LAYERS + 1];
  int a[MAVG_MAX_LAYERS + 1], dz[MAVG_MAX_LAYERS + 1];
  size_t floats;
};

struct SmallArgs {
  SmallLayout s;
  int P, B, K, L, splits;
  int dims[MAVG_MAX_LAYERS + 1];
  uint32_t inv[MAVG_MAX_LAYERS + 1];       // ceil(2^32 / dims): quotients without a division
  int w_off[MAVG_MAX_LAYERS + 1], b_off[MAVG_MAX_LAYERS + 1];   // in a replica
  const float* src; int64_t src_stride;    // weights before the first step (w~: stride 0)
  float* rep; int64_t rep_stride;
  const void* x; int x_bf16;
  const int32_t* y; int64_t S;
  uint64_t seed; int64_t round;
  float gamma;
  MomArgs mom;
  float* losses;                           // [P, K]
};

__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// *dst = v in every block of the cluster, of which this thread takes the ranks first, first + step, ...
__device__ __forceinline__ void put(float* dst, float v, int splits, int first = 0, int step = 1) {
  if (splits == 1) { if (first == 0) *dst = v; return; }
  const uint32_t at = tc::smem_u32(dst);
  for (int q = first; q < splits; q += step) st_cluster(tc::mapa_u32(at, q), v);
}
__device__ __forceinline__ void put4(float* dst, float4 v, int splits, int first = 0, int step = 1) {
  if (splits == 1) { if (first == 0) *reinterpret_cast<float4*>(dst) = v; return; }
  const uint32_t at = tc::smem_u32(dst);
  for (int q = first; q < splits; q += step) tc::st_cluster_f4(tc::mapa_u32(at, q), v.x, v.y, v.z, v.w);
}
// e / d for e d < 2^32, inv = ceil(2^32 / d)  (d = 1: inv is 0)
__device__ __forceinline__ int quotient(int e, uint32_t inv) {
  return inv ? (int)__umulhi((uint32_t)e, inv) : e;
}
template <int THREADS, int ID>
__device__ __forceinline__ void barrier() {
  asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
}
__device__ __forceinline__ void fma4(float4& s, float4 a, float b) {
  s.x = fmaf(a.x, b, s.x); s.y = fmaf(a.y, b, s.y);
  s.z = fmaf(a.z, b, s.z); s.w = fmaf(a.w, b, s.w);
}

// The minibatch of `step`, transposed, by the gather warps.  The learner's samples are
// [lo, lo + len), `key` its index stream (mavg.h).
template <bool QUANT>
__device__ __forceinline__ void gather(const SmallArgs& g, float* sm, uint64_t key, int64_t lo,
                                       uint64_t len, int step, int t) {
  const int buf = step & 1, d = g.dims[0];
  int32_t* label = reinterpret_cast<int32_t*>(sm + g.s.label[buf]);
  int32_t* index = label + g.s.pitch;
  const uint64_t step_key = fold(key, (uint64_t)step);
  for (int b = t; b < g.B; b += kGather)
    index[b] = (int32_t)(lo + (int64_t)(((fold(step_key, (uint64_t)b) >> 32) * len) >> 32));
  barrier<kGather, 2>();
  float* x = sm + g.s.x[buf];
  int32_t y = 0;                                 // the label of row t travels beside the inputs
  if (t < g.B) y = g.y[index[t]];
  const int count = g.B * d;
  for (int e0 = t; e0 < count; e0 += 8 * kGather) {
    float v[8];
    int to[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = min(e0 + u * kGather, count - 1), b = quotient(e, g.inv[0]), i = e - b * d;
      const size_t at = (size_t)index[b] * d + i;
      v[u] = g.x_bf16 ? __bfloat162float(((const __nv_bfloat16*)g.x)[at]) : operand<QUANT>(((const float*)g.x)[at]);
      to[u] = i * g.s.pitch + b;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + u * kGather < count) x[to[u]] = v[u];
  }
  if (t < g.B) label[t] = y;
  for (int b = t + kGather; b < g.B; b += kGather) label[b] = g.y[index[b]];
}

// out(j, rows) = sum_k A(k, rows) W(j, k) for the block's batch rows; A and out are [feature][pitch],
// W(j, k) = w[j * sj + k * sk].  A task is R groups of four rows of one j (lanes along j); where
// there are fewer tasks than threads, `lanes` neighbouring lanes share one and split the sum.
enum Stage { FWD_HIDDEN = 0, FWD_LAST = 1, DGRAD = 2 };
template <bool QUANT, int R>
__device__ __forceinline__ void product(const float* a, const float* w, int sj, int sk, int J, int Kk,
                                        uint32_t inv_j, int g0, int ng, int B, int pitch, Stage stage,
                                        const float* aux, float* out, int lanes, int splits, int t) {
  const int part = t & (lanes - 1);
  const int tasks = J * ((ng + R - 1) / R);
  for (int e0 = 0; e0 < tasks; e0 += kCompute / lanes) {
    const int e = e0 + t / lanes;               // whole warps take part in the shuffles below
    const int ec = min(e, tasks - 1);
    const int jr = quotient(ec, inv_j), j = ec - jr * J;
    const int gr = g0 + jr * R;
    const float* ar = a + 4 * gr;
    const float* wj = w + j * sj;
    const int more = (R == 2 && jr * R + 1 < ng) ? 4 : 0;   // no second group: the first again
    float4 s[R];
#pragma unroll
    for (int q = 0; q < R; ++q) s[q] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int k = part; k < Kk; k += lanes) {
      const float wv = operand<QUANT>(wj[k * sk]);
#pragma unroll
      for (int q = 0; q < R; ++q) {
        float4 v = *reinterpret_cast<const float4*>(ar + k * pitch + q * more);
        if (stage == DGRAD) v = operand4<QUANT>(v);          // dZ is kept unrounded
        fma4(s[q], v, wv);
      }
    }
    for (int o = lanes / 2; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < R; ++q) {
        s[q].x += __shfl_xor_sync(0xffffffffu, s[q].x, o);
        s[q].y += __shfl_xor_sync(0xffffffffu, s[q].y, o);
        s[q].z += __shfl_xor_sync(0xffffffffu, s[q].z, o);
        s[q].w += __shfl_xor_sync(0xffffffffu, s[q].w, o);
      }
    if (e >= tasks) continue;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (q && !more) break;
      const int at = j * pitch + 4 * (gr + q);
      float4 v = s[q];
      if (stage == DGRAD) {                                  // ReLU'(0) = 0
        const float4 m = *reinterpret_cast<const float4*>(aux + at);
        v = make_float4(m.x > 0.f ? v.x : 0.f, m.y > 0.f ? v.y : 0.f, m.z > 0.f ? v.z : 0.f,
                        m.w > 0.f ? v.w : 0.f);
        put4(out + at, v, splits, part, lanes);
      } else {
        const float b = aux[j];
        v = make_float4(v.x + b, v.y + b, v.z + b, v.w + b);
        if (stage == FWD_LAST) {
          if (part == 0) *reinterpret_cast<float4*>(out + at) = v;   // logits stay in this block
        } else {
          const int left = B - 4 * (gr + q);   // rows beyond the batch stay zero, whatever the weights are
          put4(out + at, operand4<QUANT>(make_float4(v.x > 0.f ? v.x : 0.f, v.y > 0.f && left > 1 ? v.y : 0.f,
                                                     v.z > 0.f && left > 2 ? v.z : 0.f,
                                                     v.w > 0.f && left > 3 ? v.w : 0.f)),
               splits, part, lanes);
        }
      }
    }
  }
}

// Loss and dZ_L of the block's rows from the logits, a warp per row, in place.
__device__ __forceinline__ void softmax_rows(const SmallArgs& g, float* sm, const int32_t* label,
                                             int g0, int ng, int warp, int lane) {
  const int C = g.dims[g.L], B = g.B, pitch = g.s.pitch, splits = g.splits;
  const float inv_b = 1.0f / (float)B;
  for (int b = 4 * g0 + warp; b < 4 * (g0 + ng); b += kCompute / 32) {
    float* z = sm + g.s.dz[g.L] + b;
    if (b >= B) {
      for (int c = lane; c < C; c += 32) put(z + c * pitch, 0.f, splits);
      continue;
    }
    const int yb = label[b];
    const float zy = z[yb * pitch];
    float m = z[(lane < C ? lane : 0) * pitch];
    for (int c = lane + 32; c < C; c += 32) m = fmaxf(m, z[c * pitch]);
    for (int q = 16; q > 0; q >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, q));
    float se = 0.f;
    for (int c = lane; c < C; c += 32) se += expf(z[c * pitch] - m);
    for (int q = 16; q > 0; q >>= 1) se += __shfl_xor_sync(0xffffffffu, se, q);
    const float lse = m + logf(se);
    for (int c = lane; c < C; c += 32)
      put(z + c * pitch, (expf(z[c * pitch] - lse) - (c == yb ? 1.f : 0.f)) * inv_b, splits);
    if (lane == 0) {
      if (splits == 1) sm[g.s.loss + b] = lse - zy;
      else st_cluster(tc::mapa_u32(tc::smem_u32(sm + g.s.loss + b), 0), lse - zy);
    }
  }
}

// Logits, loss and dZ_L of the block's rows for up to 32 classes, a warp per row and without a barrier between: `width`
// lanes (a power of two) have a class each, and 32 / width groups of them share the inputs and later the copies.
template <bool QUANT>
__device__ __forceinline__ void last_rows(const SmallArgs& g, float* sm, const float* a, const int32_t* label, int g0, int ng,
                                          int warp, int lane) {
  const int C = g.dims[g.L], in = g.dims[g.L - 1], B = g.B, pitch = g.s.pitch, splits = g.splits;
  const int width = C <= 4 ? 4 : C <= 8 ? 8 : C <= 16 ? 16 : 32, parts = 32 / width;
  const int c = lane & (width - 1), part = lane / width;
  const float* w = sm + g.s.w[g.L] + min(c, C - 1) * (in | 1);
  const float bias = sm[g.s.b[g.L] + min(c, C - 1)], inv_b = 1.0f / (float)B;
  for (int b = 4 * g0 + warp; b < 4 * (g0 + ng); b += kCompute / 32) {
    float* out = sm + g.s.dz[g.L] + c * pitch + b;
    float d = 0.f;
    if (b < B) {
      float s = 0.f;
#pragma unroll 8
      for (int k = part; k < in; k += parts) s = fmaf(a[k * pitch + b], operand<QUANT>(w[k]), s);
      for (int o = width; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float z = c < C ? s + bias : -INFINITY;
      float m = z;
      for (int o = width / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      float se = c < C ? expf(z - m) : 0.f;
      for (int o = width / 2; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
      const float lse = m + logf(se);
      const bool mine = c == label[b];
      d = (expf(z - lse) - (mine ? 1.f : 0.f)) * inv_b;
      if (mine && part == 0) {
        if (splits == 1) sm[g.s.loss + b] = lse - z;
        else st_cluster(tc::mapa_u32(tc::smem_u32(sm + g.s.loss + b), 0), lse - z);
      }
    }
    if (c < C) put(out, d, splits, part, parts);
  }
}

template <bool QUANT>
__global__ void __launch_bounds__(kCompute + kGather)
k_small_steps(const __grid_constant__ SmallArgs g) {
  extern __shared__ __align__(16) float sm[];
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();
  const int splits = g.splits, p = blockIdx.x / splits, rank = blockIdx.x % splits;
  const int t = threadIdx.x, pitch = g.s.pitch, L = g.L, B = g.B;
  const int warp = t / 32, lane = t % 32;
  const bool computes = t < kCompute;
  const int groups = (B + 3) / 4;
  const int g0 = groups * rank / splits, ng = groups * (rank + 1) / splits - g0;
  const float inv_b = 1.0f / (float)B;
  // the block's share of the weight gradients: tasks of the layers up to l, output rows that share a task, the first row
  // and how many
  __shared__ int task_end[MAVG_MAX_LAYERS + 1], share[MAVG_MAX_LAYERS + 1], row0[MAVG_MAX_LAYERS + 1], row_end[MAVG_MAX_LAYERS + 1];
  if (t == 0) {
    task_end[0] = row_end[0] = 0;
    for (int l = 1; l <= L; ++l) {
      const int in = g.dims[l - 1], out = g.dims[l], o0 = out * rank / splits, rows = out * (rank + 1) / splits - o0;
      // four output rows share the reads of A where that leaves every thread something to do
      const int per = rows * in >= 4 * kCompute ? 4 : 1;
      row0[l] = o0;
      row_end[l] = row_end[l - 1] + rows;
      share[l] = per;
      task_end[l] = task_end[l - 1] + (rows + per - 1) / per * in;
    }
  }
  uint64_t key = 0, len = 0;
  int64_t lo = 0;
  if (!computes) {
    key = learner_key(g.seed, kTagBatch, (uint64_t)g.round, (uint64_t)p);
    lo = shard_begin(p, g.P, g.S);
    len = (uint64_t)(shard_begin(p + 1, g.P, g.S) - lo);
  }

  if (computes) {
    // the whole model, sixteen parameters of a thread in flight
    const float* src = g.src + (size_t)p * g.src_stride;
    const int n = g.b_off[L] + g.dims[L];
    for (int e0 = t; e0 < n; e0 += 16 * kCompute) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = e0 + u * kCompute < n ? src[e0 + u * kCompute] : 0.f;
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int e = e0 + u * kCompute;
        if (e >= n) break;
        int l = 1;
        while (e >= g.b_off[l] + g.dims[l]) ++l;
        if (e >= g.b_off[l]) {
          sm[g.s.b[l] + e - g.b_off[l]] = v[u];
        } else {
          const int o = quotient(e - g.w_off[l], g.inv[l - 1]), i = e - g.w_off[l] - o * g.dims[l - 1];
          sm[g.s.w[l] + o * (g.dims[l - 1] | 1) + i] = v[u];
        }
      }
    }
    // rows of the last group beyond the batch: zero inputs (their dZ is zero as well)
    for (int e = t; e < g.dims[0] * 4; e += kCompute) {
      const int b = groups * 4 - 4 + e % 4;
      if (b >= B) sm[g.s.x[0] + e / 4 * pitch + b] = sm[g.s.x[1] + e / 4 * pitch + b] = 0.f;
    }
  } else {
    gather<QUANT>(g, sm, key, lo, len, 1, t - kCompute);
  }
  tc::cluster_sync_all();

  for (int step = 1; step <= g.K; ++step) {
    const float* x = sm + g.s.x[step & 1];
    if (computes) {
      const int32_t* label = reinterpret_cast<const int32_t*>(sm + g.s.label[step & 1]);
      // stages 1..L: forward products; then the loss; then L-1 data gradients, layer L first
      for (int st = 1; st <= 2 * L - 1; ++st) {
        const bool fwd = st <= L;
        if (st == L && g.dims[L] <= 32) {
          last_rows<QUANT>(g, sm, L == 1 ? x : sm + g.s.a[L - 1], label, g0, ng, warp, lane);
          barrier<kCompute, 1>();
          continue;
        }
        const int l = fwd ? st : 2 * L + 1 - st;
        const int in = g.dims[l - 1], out = g.dims[l], J = fwd ? out : in, Kk = fwd ? in : out;
        const float* a = !fwd ? sm + g.s.dz[l] : l == 1 ? x : sm + g.s.a[l - 1];
        const float* aux = fwd ? sm + g.s.b[l] : sm + g.s.a[l - 1];
        float* to = !fwd ? sm + g.s.dz[l - 1] : l < L ? sm + g.s.a[l] : sm + g.s.dz[L];
        const Stage stage = !fwd ? DGRAD : l < L ? FWD_HIDDEN : FWD_LAST;
        const int sj = fwd ? in | 1 : 1, sk = fwd ? 1 : in | 1;
        if (J * ng >= 4 * kCompute) {
          product<QUANT, 2>(a, sm + g.s.w[l], sj, sk, J, Kk, g.inv[fwd ? l : l - 1], g0, ng, B, pitch, stage, aux, to, 1, splits, t);
        } else {
          int lanes = 1;
          while (lanes < 16 && J * ng * lanes * 2 <= kCompute && lanes * 4 <= Kk) lanes *= 2;
          product<QUANT, 1>(a, sm + g.s.w[l], sj, sk, J, Kk, g.inv[fwd ? l : l - 1], g0, ng, B, pitch, stage, aux, to, lanes, splits, t);
        }
        barrier<kCompute, 1>();
        if (st == L) {
          softmax_rows(g, sm, label, g0, ng, warp, lane);
          barrier<kCompute, 1>();
        }
      }
      tc::cluster_arrive();
      tc::cluster_wait();
    } else {
      // the gather warps' own results are needed at the end of the step only
      tc::cluster_arrive();
      if (step < g.K) gather<QUANT>(g, sm, key, lo, len, step + 1, t - kCompute);
      tc::cluster_wait();
    }

    const bool last = step == g.K;
    // weight gradients and steps of all layers, by all twelve warps
    MomArgs mom = g.mom;
    if (step > 1) mom.read_u = 1;
    float* rep = g.rep + (size_t)p * g.rep_stride;
    float* u = mom.u ? mom.u + (size_t)p * mom.u_stride : nullptr;
    for (int e = t; e < task_end[L]; e += kCompute + kGather) {
      int l = 1;
      while (e >= task_end[l]) ++l;
      const int in = g.dims[l - 1], per = share[l], rows = row_end[l] - row_end[l - 1], o0 = row0[l];
      const float* a = l == 1 ? x : sm + g.s.a[l - 1];
      const float* dz = sm + g.s.dz[l];
      const int el = e - task_end[l - 1], er = quotient(el, g.inv[l - 1]), i = el - er * in, o = o0 + er * per;
      float s[4] = {0.f, 0.f, 0.f, 0.f};
      if (per == 4) {
        const int left = o0 + rows - 1 - o;          // rows beyond the last repeat it
        const float* d[4] = {dz + o * pitch, dz + (o + min(1, left)) * pitch,
                             dz + (o + min(2, left)) * pitch, dz + (o + min(3, left)) * pitch};
#pragma unroll 2
        for (int q = 0; q < groups; ++q) {
          const float4 av = *reinterpret_cast<const float4*>(a + i * pitch + 4 * q);
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const float4 dv = operand4<QUANT>(*reinterpret_cast<const float4*>(d[h] + 4 * q));
            s[h] = fmaf(dv.x, av.x, s[h]); s[h] = fmaf(dv.y, av.y, s[h]);
            s[h] = fmaf(dv.z, av.z, s[h]); s[h] = fmaf(dv.w, av.w, s[h]);
          }
        }
      } else {
        const float *ar = a + i * pitch, *dr = dz + o * pitch;
#pragma unroll 4
        for (int q = 0; q < groups; ++q) {
          const float4 av = *reinterpret_cast<const float4*>(ar + 4 * q);
          const float4 dv = operand4<QUANT>(*reinterpret_cast<const float4*>(dr + 4 * q));
          s[0] = fmaf(dv.x, av.x, s[0]); s[0] = fmaf(dv.y, av.y, s[0]);
          s[0] = fmaf(dv.z, av.z, s[0]); s[0] = fmaf(dv.w, av.w, s[0]);
        }
      }
      float* w = sm + g.s.w[l];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (h >= per || o + h >= o0 + rows) break;
        float* wp = w + (o + h) * (in | 1) + i;
        const int off = g.w_off[l] + (o + h) * in + i;
        float v;
        local_update(&v, *wp, u ? u + off : nullptr, mom.read_u, s[h], g.gamma, mom.beta);
        if (last) rep[off] = v;
        else put(wp, v, splits);
      }
    }
    // bias steps (from the unrounded dZ), a warp per output, last warp first: its tasks above may be fewer
    for (int e = kWarps - 1 - warp; e < row_end[L]; e += kWarps) {
      int l = 1;
      while (e >= row_end[l]) ++l;
      const int o = row0[l] + e - row_end[l - 1];
      const float* dz = sm + g.s.dz[l] + o * pitch;
      float s = 0.f;
      for (int b = lane; b < B; b += 32) s += dz[b];
      for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
      if (lane == 0) {
        float v;
        local_update(&v, sm[g.s.b[l] + o], u ? u + g.b_off[l] + o : nullptr, mom.read_u, s, g.gamma, mom.beta);
        if (last) rep[g.b_off[l] + o] = v;
        else put(sm + g.s.b[l] + o, v, splits);
      }
      __syncwarp();
    }
    if (rank == 0 && warp == 0) {
      float s = 0.f;
      for (int b = lane; b < B; b += 32) s += sm[g.s.loss + b];
      for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
      if (lane == 0) g.losses[(size_t)p * g.K + step - 1] = s * inv_b;
    }
    __syncwarp();
    tc::cluster_sync_all();
  }
}

SmallLayout layout(const mavg_config* cfg) {
  SmallLayout s{};
  s.pitch = (cfg->B + 3) / 4 * 4;
  if (s.pitch / 4 % 2 == 0) s.pitch += 4;
  size_t off = 0;
  auto take = [&](size_t floats) { const size_t r = off; off += (floats + 3) / 4 * 4; return (int)std::min<size_t>(r, 1 << 30); };
  for (int i = 0; i < 2; ++i) {
    s.x[i] = take((size_t)cfg->dims[0] * s.pitch);
    s.label[i] = take(2 * (size_t)s.pitch);       // labels and indices
  }
  s.loss = take(s.pitch);
  for (int l = 1; l <= cfg->n_layers; ++l) {
    s.w[l] = take((size_t)cfg->dims[l] * (cfg->dims[l - 1] | 1));
    s.b[l] = take(cfg->dims[l]);
    if (l < cfg->n_layers) s.a[l] = take((size_t)cfg->dims[l] * s.pitch);
    s.dz[l] = take((size_t)cfg->dims[l] * s.pitch);
  }
  s.floats = off;
  return s;
}

cudaLaunchConfig_t launch_config(const mavg_ctx* c, int splits, cudaLaunchAttribute (&at)[2]) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = dim3((unsigned)(c->cfg.P * splits));
  lc.blockDim = dim3(kCompute + kGather);
  lc.dynamicSmemBytes = layout(&c->cfg).floats * sizeof(float);
  lc.stream = c->stream;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)splits;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  return lc;
}

}  // namespace

// Layout that fits at all; small_setup decides whether the path is taken.
static bool small_fits(const mavg_config* cfg) {
  return cfg->gemm_bf16 != 1 && layout(cfg).floats * sizeof(float) <= kSmallSmem;
}

bool small_always(const mavg_config* cfg) { return cfg->n <= 4096 && small_fits(cfg); }

// Splits: the widest cluster that every block still has a group of rows for and of which the GPU holds
// all P at once (a cluster's blocks share one GPC, so that is fewer than SMs / S).
// The path is taken for models of at most 4096 parameters and, up to what shared memory holds, where
// at least four blocks share a learner and a block's products are at most 110 000 multiply-adds each.
// Measured against a launch per product, 150 models with K = 1, 4 or 8 and P = 1 .. 300: up to 4096 parameters 1.18 .. 4.3
// times as fast (32-64-10, K = 4, B = 32, us a round: P = 4 32 / 75, P = 100 78 / 165, P = 300 179 / 423); beyond, in fp32
// 1.00 .. 2.6 (80-128-16, B = 32, P = 4 55 / 83; B = 48, P = 16, 74 600 a block, 95 / 94); with bf16 operands, whose
// launches have a plane to each operand, 1.03 .. 1.6 up to 25 000 a block and 0.76 .. 1.25 above (52-112-126-10, P = 8,
// K = 4, B = 20 148 / 112).  What the lines leave to the launches would be 0.60 .. 2.3 with one to three blocks a learner
// (80-128-128-16, B = 16, P = 300 800 / 569; 78-57-13, P = 123, K = 8, B = 61 251 / 575) and 1.2 beyond 110 000
// (80-128-128-16, B = 32, P = 4 107 / 129).
// A device or driver that refuses one of the calls here leaves the handle the launch per product.
void small_setup(mavg_ctx* c) {
  const mavg_config& cfg = c->cfg;
  c->small_splits = 0;
  if (!small_fits(&cfg)) return;
  auto kernel = cfg.gemm_bf16 ? k_small_steps<true> : k_small_steps<false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem);
  int splits = 1;
  for (int s = 8; s > 1 && e == cudaSuccess; s /= 2) {
    if (s > (cfg.B + 3) / 4) continue;
    cudaLaunchAttribute at[2];
    const cudaLaunchConfig_t lc = launch_config(c, s, at);
    int resident = 0;
    e = cudaOccupancyMaxActiveClusters(&resident, kernel, &lc);
    if (e == cudaSuccess && resident >= cfg.P) { splits = s; break; }
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  if (small_always(&cfg) || (splits >= 4 && cfg.n * cfg.B <= (int64_t)110000 * splits)) c->small_splits = splits;
}

cudaError_t small_local_steps(mavg_ctx* c, int64_t round) {
  const mavg_config& cfg = c->cfg;
  SmallArgs g{};
  g.s = layout(&cfg);
  g.P = cfg.P; g.B = cfg.B; g.K = cfg.K; g.L = cfg.n_layers; g.splits = c->small_splits;
  for (int l = 0; l <= g.L; ++l)
    g.inv[l] = (uint32_t)((((uint64_t)1 << 32) + cfg.dims[l] - 1) / cfg.dims[l]);   // 0 for a width of 1
  g.dims[0] = cfg.dims[0];
  for (int l = 1; l <= g.L; ++l) {
    g.dims[l] = cfg.dims[l];
    g.w_off[l] = (int)c->layers[l - 1].w_off;
    g.b_off[l] = (int)c->layers[l - 1].b_off;
  }
  g.src = starts_from_global(c) ? c->buf.global_w : c->buf.replicas;
  g.src_stride = starts_from_global(c) ? 0 : c->buf.replica_stride;
  g.rep = c->buf.replicas; g.rep_stride = c->buf.replica_stride;
  g.x = cfg.x; g.x_bf16 = cfg.x_dtype == MAVG_X_BF16;
  g.y = cfg.y; g.S = cfg.n_samples;
  g.seed = cfg.seed; g.round = round;
  g.gamma = cfg.local_lr;
  g.mom = mom_args(c, c->replicas_equal_global);
  g.losses = (float*)ws_ptr(c, c->ws.losses);
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t lc = launch_config(c, g.splits, at);
  prof_begin(c, MAVG_K_WGRAD_SGD);
  cudaError_t e = cudaLaunchKernelEx(&lc, cfg.gemm_bf16 ? k_small_steps<true> : k_small_steps<false>, g);
  prof_end(c);
  c->replicas_equal_global = false;
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace mavg
