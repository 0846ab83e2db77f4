// CUDA-core MLP learner step, batched over the P learners (blockIdx.z).
//   forward   Z_l = A_{l-1} W_l^T + b_l,  A_l = act(Z_l)          (A_0 = gathered minibatch)
//   backward  dA_{l-1} = (dZ_l W_l) .* [A_{l-1} > 0];  dW_l = dZ_l^T A_{l-1};  db_l = colsum dZ_l
//   SGD       W_l <- W_l - gamma dW_l, b_l <- b_l - gamma db_l    (Algorithm 1's local update)
// fp32 FMAs.  With QUANT every matrix-product operand is first rounded to bf16
// (nearest-even), which makes this path compute the same thing as the tensor-core path, and the products run
// on warp-level MMAs (fp32 sums); it is the path for true fp32 models and for layer widths the tensor-core
// path does not cover.
// A step is L-1 forward launches, one for the whole last layer up to its data gradient (which
// also gathers the next step's minibatch), L-2 data gradients and one for the weight gradients,
// bias gradients and SGD steps of all layers.  While a deferred re-broadcast is outstanding the first
// step of a round reads the weights from w~ and writes the results to the replicas, so its P copies
// are never needed.
#include <algorithm>

#include "mlp.cuh"
#include "tc_ptx.cuh"

namespace mavg {
namespace {

__device__ __forceinline__ float qbf(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
template <bool QUANT>
__device__ __forceinline__ float operand(float v) { return QUANT ? qbf(v) : v; }

// ------------------------------------------------------------------------------ matrix products
// C(m,n) = sum_k A(m,k) B(n,k): one 64 x 64 tile per block of 128 threads, 8 x 4 outputs each.
// Bound: the FMA pipe and the register ports that feed it (a product of ordinary size keeps its
// operands in the L2).  Slabs of 16 k go through registers into two shared-memory buffers, so the
// loads of a slab overlap the products of the one before; both operands are stored k-major, the
// operands of k + 1 are read while k is multiplied, and an fma.f32x2 does the FMAs of two rows in
// one issue slot, which leaves slots for the reads.  Where the tiles would leave SMs idle the
// contraction is split over the blocks of a cluster, which add their partial tiles in rank order
// through distributed shared memory.
// First layer of a 3072-512-512-10 model, P = 4, B = 100: 53 us forward (21 us of FMAs at the peak
// rate, padding of the batch to 128 included), weight gradients of all layers 55 us.  Measured on the
// same case and not better: 8 x 8 outputs per thread (51 and 60 us, whole round 693 us against
// 590: half as many warps), the same with one-element FMAs (76), and a ring of asynchronous copies in
// the operands' own orientation (58, and twice as slow for rows that do not start on 16 bytes).
constexpr int BM = 64, BN = 64, BK = 16, kThreads = 128;
constexpr int kPitchA = BM + 4, kPitchB = BN + 4;
constexpr int kMaxSplit = 8;

enum Epi { EPI_FWD = 0, EPI_DGRAD = 1, EPI_WGRAD_SGD = 2 };

// FWD:   A = activations [M, K], B = W [N, K];       C = A_l (hidden) or the logits; aux = bias [N]
// DGRAD: A = dZ [M, K],          B = W [K, N];       C = dZ of the layer below; aux = A_{l-1} [M, N]
// WGRAD: A = dZ [K, M],          B = A_{l-1} [K, N]; C = W [M, N], aux = W before the step
struct GemmArgs {
  const float* A; int64_t a_batch;
  const float* B; int64_t b_batch;
  int M, N, K;
  float* C; int64_t c_batch;
  const float* aux; int64_t aux_batch;
  int vec_a, vec_b, vec_c;  // rows of the operand start on 16 bytes and hold whole groups of 4
  int k_per_split;
  int hidden;           // FWD: apply ReLU (and the operand rounding of the next products)
  // WGRAD: bias after the step, before it, and what the local update needs
  float* bias; const float* bias_in;
  float gamma;
  MomArgs mom;          // momentum slots at mom.u[p*u_stride + u_off (+ the bias offset ub_off)]
  int64_t u_off, ub_off;
};

struct __align__(16) Slab { float a[BK][kPitchA], b[BK][kPitchB]; };
union __align__(16) GemmShared {
  Slab slab[2];
  float c[BM][kPitchB];  // partial tile of a split contraction
};

// A ROWS x 16 piece of an operand through registers.  KC: memory is [row, k] (k contiguous), else
// [k, row].  rows and k_end bound the operand; what lies outside is zero.  The way a thread's
// elements lie depends on `vec` alone (uniform): groups of four or single elements.
template <int ROWS, bool KC>
struct Piece {
  static constexpr int N = ROWS * BK / kThreads;   // elements per thread
  float r[N];
  __device__ __forceinline__ void load(const float* __restrict__ p, int ld, int vec, int row0,
                                       int rows, int k0, int k_end) {
    const int t = threadIdx.x;
    if (vec) {
#pragma unroll
      for (int e = 0; e < N / 4; ++e) {
        const int row = row0 + (KC ? t / 4 + 32 * e : (t % (ROWS / 4)) * 4);
        const int k = k0 + (KC ? (t % 4) * 4 : t / (ROWS / 4) + e * (kThreads * 4 / ROWS));
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < rows && k < k_end)
          v = *reinterpret_cast<const float4*>(p + (KC ? (size_t)row * ld + k : (size_t)k * ld + row));
        r[4 * e] = v.x; r[4 * e + 1] = v.y; r[4 * e + 2] = v.z; r[4 * e + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < N; ++e) {
        const int row = row0 + (KC ? t / 16 + 8 * e : t % ROWS);
        const int k = k0 + (KC ? t % 16 : t / ROWS + e * (kThreads / ROWS));
        r[e] = (row < rows && k < k_end) ? p[KC ? (size_t)row * ld + k : (size_t)k * ld + row] : 0.f;
      }
    }
  }
  template <int PITCH>
  __device__ __forceinline__ void store(float (*s)[PITCH], int vec) const {
    const int t = threadIdx.x;
    if (vec) {
#pragma unroll
      for (int e = 0; e < N / 4; ++e) {
        if (KC) {
#pragma unroll
          for (int i = 0; i < 4; ++i) s[(t % 4) * 4 + i][t / 4 + 32 * e] = r[4 * e + i];
        } else {
          *reinterpret_cast<float4*>(&s[t / (ROWS / 4) + e * (kThreads * 4 / ROWS)][(t % (ROWS / 4)) * 4]) =
              make_float4(r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]);
        }
      }
    } else {
#pragma unroll
      for (int e = 0; e < N; ++e) {
        if (KC) s[t % 16][t / 16 + 8 * e] = r[e];
        else s[t / ROWS + e * (kThreads / ROWS)][t % ROWS] = r[e];
      }
    }
  }
};

__device__ __forceinline__ uint64_t dup2(float v) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ float half_of(uint64_t v, int hi) {
  return __uint_as_float((uint32_t)(hi ? v >> 32 : v));
}

// acc[i][j] holds rows 8 ty + 2 i, + 1 of column 4 tx + j
struct Fragment { ulonglong2 a0, a1; float4 b; };
__device__ __forceinline__ void read(Fragment& f, const Slab& s, int k) {
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  f.a0 = *reinterpret_cast<const ulonglong2*>(&s.a[k][8 * ty]);
  f.a1 = *reinterpret_cast<const ulonglong2*>(&s.a[k][8 * ty + 4]);
  f.b = *reinterpret_cast<const float4*>(&s.b[k][4 * tx]);
}
__device__ __forceinline__ void multiply(const Slab& s, uint64_t (&acc)[4][4]) {
  Fragment f[2];
  read(f[0], s, 0);
#pragma unroll
  for (int k = 0; k < BK; ++k) {
    if (k + 1 < BK) read(f[(k + 1) & 1], s, k + 1);
    const Fragment& c = f[k & 1];
    const uint64_t a[4] = {c.a0.x, c.a0.y, c.a1.x, c.a1.y};
    const float b[4] = {c.b.x, c.b.y, c.b.z, c.b.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint64_t bb = dup2(b[j]);
#pragma unroll
      for (int i = 0; i < 4; ++i) fma2(acc[i][j], a[i], bb);
    }
  }
}

// ---- bf16 operands: the same tile on warp-level MMAs, 4 warps of 32 x 32 each.  They take operands from any row
// length and start, which tiled copies do not (B200's rate for them, 144 TFLOP/s measured, is twice the FMA
// pipe's; as sums of three bf16 numbers fp32 operands would need six of them: 76 us for the 53 of the first
// layer above).  Bound by the way through registers and the latency of a few slabs: 1000-333-100, P = 6, B = 50:
// forward product of layer 1 14 us (19 with FMAs), weight gradients of
// both layers 16 us (26, of which a last wave that was nearly empty and four loads at a time in the epilogue).
// A slab's sum starts from zero and is added to the tile's in fp32, rounded to nearest: the tensor cores cut a
// sum off where they add to it.
constexpr int QK = 32;                             // k per slab
// An operand's slab: [64 rows][32 k] in rows of 40 elements, or [32 k][64 rows] in rows of 72: eight
// consecutive rows start in different banks.
constexpr int kPitchK = QK + 8, kPitchR = BM + 8;
constexpr int kSlab = BM * kPitchK;                // elements, the larger of the two
static_assert(QK * kPitchR <= kSlab && BM == BN, "");
union __align__(16) MmaShared {
  __nv_bfloat16 slab[2][2][kSlab];                 // buffer, operand
  float c[BM][kPitchB];
};

// A 64 x 32 piece of an operand through registers.  KC: memory is [row, k] (k contiguous), else
// [k, row].  rows and k_end bound the operand; what lies outside is zero.  The way a thread's
// elements lie depends on `vec` alone (uniform): groups of four or single elements.
template <bool KC>
struct MmaPiece {
  static constexpr int N = BM * QK / kThreads;   // elements per thread
  float r[N];
  __device__ __forceinline__ void load(const float* __restrict__ p, int ld, int vec, int row0,
                                       int rows, int k0, int k_end) {
    const int t = threadIdx.x;
    if (vec) {
#pragma unroll
      for (int e = 0; e < N / 4; ++e) {
        const int row = row0 + (KC ? t / 8 + 16 * e : (t % 16) * 4);
        const int k = k0 + (KC ? (t % 8) * 4 : t / 16 + 8 * e);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (row < rows && k < k_end)
          v = *reinterpret_cast<const float4*>(p + (KC ? (size_t)row * ld + k : (size_t)k * ld + row));
        r[4 * e] = v.x; r[4 * e + 1] = v.y; r[4 * e + 2] = v.z; r[4 * e + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < N; ++e) {
        const int row = row0 + (KC ? t / 32 + 4 * e : t % 64);
        const int k = k0 + (KC ? t % 32 : t / 64 + 2 * e);
        r[e] = (row < rows && k < k_end) ? p[KC ? (size_t)row * ld + k : (size_t)k * ld + row] : 0.f;
      }
    }
  }
  __device__ __forceinline__ void store(__nv_bfloat16* s, int vec) const {
    const int t = threadIdx.x;
    if (vec) {
#pragma unroll
      for (int e = 0; e < N / 4; ++e) {
        const int at = KC ? (t / 8 + 16 * e) * kPitchK + (t % 8) * 4 : (t / 16 + 8 * e) * kPitchR + (t % 16) * 4;
        __nv_bfloat162 h[2] = {__floats2bfloat162_rn(r[4 * e], r[4 * e + 1]), __floats2bfloat162_rn(r[4 * e + 2], r[4 * e + 3])};
        *reinterpret_cast<uint2*>(s + at) = *reinterpret_cast<uint2*>(h);
      }
    } else {
#pragma unroll
      for (int e = 0; e < N; ++e)
        s[KC ? (t / 32 + 4 * e) * kPitchK + t % 32 : (t / 64 + 2 * e) * kPitchR + t % 64] = __float2bfloat16_rn(r[e]);
    }
  }
};

// 16 rows x 16 k of the MMA's row operand, 16 columns x 16 k (two of its column operands) from a plane.
template <bool KC>
__device__ __forceinline__ void row_operand(uint32_t (&r)[4], const __nv_bfloat16* pl, int row, int k) {
  const int i = threadIdx.x % 32 / 8, j = threadIdx.x % 8;
  if (KC) tc::ldsm_x4(r, pl + (row + (i & 1) * 8 + j) * kPitchK + k + (i >> 1) * 8);
  else tc::ldsm_x4_t(r, pl + (k + (i >> 1) * 8 + j) * kPitchR + row + (i & 1) * 8);
}
template <bool KC>
__device__ __forceinline__ void col_operands(uint32_t (&r)[4], const __nv_bfloat16* pl, int row, int k) {
  const int i = threadIdx.x % 32 / 8, j = threadIdx.x % 8;
  if (KC) tc::ldsm_x4(r, pl + (row + (i >> 1) * 8 + j) * kPitchK + k + (i & 1) * 8);
  else tc::ldsm_x4_t(r, pl + (k + (i & 1) * 8 + j) * kPitchR + row + (i >> 1) * 8);
}
// One slab of the tile.  acc[mt][nt]: 16 x 8 results at rows 32 wm + 16 mt, columns 32 wn + 8 nt; mts, nps: how
// many 16-row and 16-column groups of the warp's lie inside the result.
// FRESH: the slab's sum on its own first.  Not for weight gradients over batches of up to kChainRows samples, whose
// chains are short (the sums apart need the registers of a fifth block on the SM: 3000-801-99, P = 8, B = 128 513 us
// for two steps, 582 with spills).  A chain's cut-offs all go the same way, an fp32 sum's roundings either way: relative
// to 2^-24 of a sum of like terms, root mean square, chain / fp32 sum / FRESH: 1000 samples 7.5 / 9.2 / 1.7; 3000
// samples 133 / 14 / 2.5; 12000 samples 1082 / 30 / 5.0.
template <bool A_KC, bool B_KC, bool FRESH>
__device__ __forceinline__ void multiply_mma(const __nv_bfloat16* a, const __nv_bfloat16* b, int mts, int nps,
                                             float (&acc)[2][4][4]) {
  const int warp = threadIdx.x / 32, wm = warp & 1, wn = warp >> 1;
  float own[2][4][4] = {};
  float (&d)[2][4][4] = FRESH ? own : acc;
#pragma unroll
  for (int k = 0; k < QK; k += 16) {
    uint32_t fa[2][4];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) row_operand<A_KC>(fa[mt], a, 32 * wm + 16 * mt, k);
#pragma unroll
    for (int np = 0; np < 2; ++np) {
      if (np >= nps) break;
      uint32_t fb[4];
      col_operands<B_KC>(fb, b, 32 * wn + 16 * np, k);
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        if (mt >= mts) break;
        tc::mma_bf16(d[mt][2 * np], fa[mt], fb[0], fb[1]);
        tc::mma_bf16(d[mt][2 * np + 1], fa[mt], fb[2], fb[3]);
      }
    }
  }
  if constexpr (FRESH) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[mt][nt][i] += own[mt][nt][i];
  }
}

// Four finished sums C(m, n .. n+3): the layer's tail and the store.
template <bool QUANT, int EPI>
__device__ __forceinline__ void emit(const GemmArgs& g, int p, int m, int n, float (&v)[4]) {
  if (m >= g.M || n >= g.N) return;
  const size_t ci = (size_t)m * g.N + n;
  float* C = g.C + (size_t)p * g.c_batch + ci;
  const float* aux = g.aux + (size_t)p * g.aux_batch + (EPI == EPI_FWD ? (size_t)n : ci);
  float x[4] = {0.f, 0.f, 0.f, 0.f};
  if (g.vec_c && EPI != EPI_FWD) {       // the bias vector may start anywhere
    const float4 t = *reinterpret_cast<const float4*>(aux);
    x[0] = t.x; x[1] = t.y; x[2] = t.z; x[3] = t.w;
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (n + i < g.N) x[i] = aux[i];
  }
  float* U = (EPI == EPI_WGRAD_SGD && g.mom.u)
                 ? g.mom.u + (size_t)p * g.mom.u_stride + g.u_off + ci : nullptr;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (EPI == EPI_FWD) {
      v[i] += x[i];
      if (g.hidden) v[i] = operand<QUANT>(v[i] > 0.f ? v[i] : 0.f);
    } else if (EPI == EPI_DGRAD) {
      v[i] = x[i] > 0.f ? v[i] : 0.f;    // ReLU'(0) = 0
    } else if (U && n + i < g.N) {
      float u = g.mom.read_u ? U[i] : 0.f;
      msgd(x[i], u, v[i], g.gamma, g.mom.beta);
      U[i] = u;
      v[i] = x[i];
    } else {
      v[i] = fmaf(-g.gamma, v[i], x[i]);
    }
  }
  if (g.vec_c) {
    *reinterpret_cast<float4*>(C) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (n + i < g.N) C[i] = v[i];
  }
}

// The blocks of a cluster have left their partial tiles in c: this block finishes 64 / splits rows of the tile.
template <bool QUANT, int EPI>
__device__ __forceinline__ void finish_split(const GemmArgs& g, int m0, int n0, int p, int rank, int splits,
                                             float (*c)[kPitchB]) {
  tc::cluster_sync_all();
  for (int t = threadIdx.x; t < BM / splits * (BN / 4); t += kThreads) {
    const int m = rank * (BM / splits) + t / (BN / 4), n = 4 * (t % (BN / 4));
    const uint32_t own = tc::smem_u32(&c[m][n]);
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    for (int q = 0; q < splits; ++q) {
      float4 x;
      asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w)
                   : "r"(tc::mapa_u32(own, q)) : "memory");
      v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
    }
    emit<QUANT, EPI>(g, p, m0 + m, n0 + n, v);
  }
  __syncwarp();
  tc::cluster_sync_all();   // a peer may still be reading this block's partial tile
}

template <int EPI>
__device__ __forceinline__ void fma_tile(const GemmArgs& g, int m0, int n0, int p, int rank,
                                         int splits, GemmShared& sh) {
  constexpr bool A_KC = EPI != EPI_WGRAD_SGD, B_KC = EPI == EPI_FWD;
  const float* A = g.A + (size_t)p * g.a_batch;
  const float* B = g.B + (size_t)p * g.b_batch;
  const int lda = A_KC ? g.K : g.M, ldb = B_KC ? g.K : g.N;
  const int k_begin = rank * g.k_per_split;
  const int k_end = min(g.K, k_begin + g.k_per_split);
  uint64_t acc[4][4] = {};
  Piece<BM, A_KC> pa;
  Piece<BN, B_KC> pb;
  if (k_begin < k_end) {
    pa.load(A, lda, g.vec_a, m0, g.M, k_begin, k_end);
    pb.load(B, ldb, g.vec_b, n0, g.N, k_begin, k_end);
    pa.store(sh.slab[0].a, g.vec_a);
    pb.store(sh.slab[0].b, g.vec_b);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = k_begin; k0 < k_end; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < k_end;
    if (more) {
      pa.load(A, lda, g.vec_a, m0, g.M, k0 + BK, k_end);
      pb.load(B, ldb, g.vec_b, n0, g.N, k0 + BK, k_end);
    }
    multiply(sh.slab[buf], acc);
    if (more) {
      pa.store(sh.slab[buf ^ 1].a, g.vec_a);
      pb.store(sh.slab[buf ^ 1].b, g.vec_b);
    }
    __syncthreads();
  }
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  if (splits == 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) v[j] = half_of(acc[i / 2][j], i & 1);
      emit<false, EPI>(g, p, m0 + 8 * ty + i, n0 + 4 * tx, v);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
    *reinterpret_cast<float4*>(&sh.c[8 * ty + i][4 * tx]) =
        make_float4(half_of(acc[i / 2][0], i & 1), half_of(acc[i / 2][1], i & 1),
                    half_of(acc[i / 2][2], i & 1), half_of(acc[i / 2][3], i & 1));
  finish_split<false, EPI>(g, m0, n0, p, rank, splits, sh.c);
}

template <int EPI, bool FRESH>
__device__ __forceinline__ void mma_tile(const GemmArgs& g, int m0, int n0, int p, int rank, int splits,
                                         MmaShared& sh) {
  constexpr bool A_KC = EPI != EPI_WGRAD_SGD, B_KC = EPI == EPI_FWD;
  const float* A = g.A + (size_t)p * g.a_batch;
  const float* B = g.B + (size_t)p * g.b_batch;
  const int lda = A_KC ? g.K : g.M, ldb = B_KC ? g.K : g.N;
  const int k_begin = rank * g.k_per_split;
  const int k_end = min(g.K, k_begin + g.k_per_split);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, wm = warp & 1, wn = warp >> 1;
  const int mts = (g.M - m0 - 32 * wm + 15) / 16, nps = (g.N - n0 - 32 * wn + 15) / 16;
  float acc[2][4][4] = {};
  MmaPiece<A_KC> pa;
  MmaPiece<B_KC> pb;
  if (k_begin < k_end) {
    pa.load(A, lda, g.vec_a, m0, g.M, k_begin, k_end);
    pb.load(B, ldb, g.vec_b, n0, g.N, k_begin, k_end);
    pa.store(sh.slab[0][0], g.vec_a);
    pb.store(sh.slab[0][1], g.vec_b);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = k_begin; k0 < k_end; k0 += QK, buf ^= 1) {
    const bool more = k0 + QK < k_end;
    if (more) {
      pa.load(A, lda, g.vec_a, m0, g.M, k0 + QK, k_end);
      pb.load(B, ldb, g.vec_b, n0, g.N, k0 + QK, k_end);
    }
    multiply_mma<A_KC, B_KC, FRESH>(sh.slab[buf][0], sh.slab[buf][1], mts, nps, acc);
    if (more) {
      pa.store(sh.slab[buf ^ 1][0], g.vec_a);
      pb.store(sh.slab[buf ^ 1][1], g.vec_b);
    }
    __syncthreads();
  }
  // through shared memory, so that a thread finishes four neighbours of a row
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        *reinterpret_cast<float2*>(&sh.c[32 * wm + 16 * mt + lane / 4 + 8 * h][32 * wn + 8 * nt + 2 * (lane % 4)]) =
            make_float2(acc[mt][nt][2 * h], acc[mt][nt][2 * h + 1]);
  __syncthreads();
  if (splits > 1) {
    finish_split<true, EPI>(g, m0, n0, p, rank, splits, sh.c);
    return;
  }
#pragma unroll
  for (int i = 0; i < BM * (BN / 4) / kThreads; ++i) {
    const int t = threadIdx.x + i * kThreads;
    const float4 x = *reinterpret_cast<const float4*>(&sh.c[t / (BN / 4)][4 * (t % (BN / 4))]);
    float v[4] = {x.x, x.y, x.z, x.w};
    emit<true, EPI>(g, p, m0 + t / (BN / 4), n0 + 4 * (t % (BN / 4)), v);
  }
}

template <bool QUANT> struct TileShared { using type = GemmShared; };
template <> struct TileShared<true> { using type = MmaShared; };
template <bool QUANT, int EPI, bool FRESH = true>
__device__ __forceinline__ void gemm_tile(const GemmArgs& g, int m0, int n0, int p, int rank, int splits,
                                          typename TileShared<QUANT>::type& sh) {
  if constexpr (QUANT) mma_tile<EPI, FRESH>(g, m0, n0, p, rank, splits, sh);
  else fma_tile<EPI>(g, m0, n0, p, rank, splits, sh);
}

// Forward and data gradient: grid (splits x row tiles x column tiles, 1, P), clusters of `splits`.
template <bool QUANT, int EPI>
__global__ void __launch_bounds__(kThreads, 4)
k_simt_gemm(const __grid_constant__ GemmArgs g, int splits) {
  __shared__ typename TileShared<QUANT>::type sh;
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();
  const int rank = blockIdx.x % splits, tile = blockIdx.x / splits;
  const int n_tiles = (g.N + BN - 1) / BN;
  gemm_tile<QUANT, EPI>(g, tile / n_tiles * BM, tile % n_tiles * BN, blockIdx.z, rank, splits, sh);
}

// Weight gradients + SGD of all layers in one launch: grid (tiles of layer 1, 2, ..., 1, P).  The
// blocks of a layer's first column tile also take the bias step (ascending batch, unrounded dZ),
// and the first block of a learner adds up its row losses.
struct WgradArgs {
  GemmArgs g[MAVG_MAX_LAYERS];
  int tile0[MAVG_MAX_LAYERS + 1];
  int L;
  const float* row_loss;   // [P, B]
  float* loss_out;
  int loss_stride;
};
// FRESH (bf16 operands): see multiply_mma.
constexpr int kChainRows = 512;
template <bool QUANT, bool FRESH>
__global__ void __launch_bounds__(kThreads, QUANT && !FRESH ? 5 : 4)
k_simt_wgrad(const __grid_constant__ WgradArgs w) {
  __shared__ typename TileShared<QUANT>::type sh;
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();
  int l = 0;
  while (l + 1 < w.L && (int)blockIdx.x >= w.tile0[l + 1]) ++l;
  const GemmArgs& g = w.g[l];
  const int tile = blockIdx.x - w.tile0[l], p = blockIdx.z;
  const int n_tiles = (g.N + BN - 1) / BN;
  const int m0 = tile / n_tiles * BM, n0 = tile % n_tiles * BN;
  gemm_tile<QUANT, EPI_WGRAD_SGD, FRESH>(g, m0, n0, p, 0, 1, sh);
  const int o = m0 + threadIdx.x;
  if (n0 == 0 && threadIdx.x < BM && o < g.M) {
    const float* d = g.A + (size_t)p * g.a_batch + o;
    float s = 0.f;
#pragma unroll 16
    for (int b = 0; b < g.K; ++b) s += d[(size_t)b * g.M];
    float* ub = g.mom.u ? g.mom.u + (size_t)p * g.mom.u_stride + g.ub_off + o : nullptr;
    local_update(g.bias + (size_t)p * g.c_batch + o, g.bias_in[(size_t)p * g.aux_batch + o], ub,
                 g.mom.read_u, s, g.gamma, g.mom.beta);
  }
  if (blockIdx.x == 0 && threadIdx.x >= kThreads - 32) {
    const int lane = threadIdx.x % 32;
    float s = 0.f;
    for (int b = lane; b < g.K; b += 32) s += w.row_loss[(size_t)p * g.K + b];
    for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
    if (lane == 0) w.loss_out[(size_t)p * w.loss_stride] = s / (float)g.K;
  }
}

// ------------------------------------------------------------------------- minibatch and loss
struct GatherArgs {
  const void* x; int x_bf16;
  const int32_t* y;
  uint64_t seed; int64_t round; const int64_t* round_ptr;
  int step, P, B, d;
  int64_t S;
  float* out;            // [P, B, d]
  int32_t* labels;       // [P, B]
};

// One sampled row: index, label and the row itself.
template <bool QUANT>
__device__ __forceinline__ void gather_row(const GatherArgs& g, int row) {
  __shared__ int32_t sidx;
  if (threadIdx.x == 0) {
    const int64_t round = g.round_ptr ? *g.round_ptr : g.round;
    sidx = sample_index(g.seed, round, row / g.B, g.step, row % g.B, g.P, g.S);
    g.labels[row] = g.y[sidx];
  }
  __syncthreads();
  const size_t src = (size_t)sidx * g.d;
  float* dst = g.out + (size_t)row * g.d;
  if (g.x_bf16) {
    const __nv_bfloat16* x = (const __nv_bfloat16*)g.x + src;
    for (int i = threadIdx.x; i < g.d; i += blockDim.x) dst[i] = __bfloat162float(x[i]);
  } else if (g.d % 4 == 0) {
    const float4* x = reinterpret_cast<const float4*>((const float*)g.x + src);
    for (int i = threadIdx.x; i < g.d / 4; i += blockDim.x) {
      const float4 v = x[i];
      reinterpret_cast<float4*>(dst)[i] = make_float4(operand<QUANT>(v.x), operand<QUANT>(v.y),
                                                      operand<QUANT>(v.z), operand<QUANT>(v.w));
    }
  } else {
    const float* x = (const float*)g.x + src;
    for (int i = threadIdx.x; i < g.d; i += blockDim.x) dst[i] = operand<QUANT>(x[i]);
  }
}

template <bool QUANT>
__global__ void __launch_bounds__(256) k_simt_gather(const __grid_constant__ GatherArgs g) {
  tc::grid_launch_dependents();
  tc::grid_dependency_wait();
  gather_row<QUANT>(g, blockIdx.x);
}

// Softmax of one row z (C logits in shared or global memory) by a warp: writes dz and returns the loss.
template <typename Put>
__device__ __forceinline__ float softmax_row(const float* z, int C, int label, float inv_b, Put put) {
  const int lane = threadIdx.x % 32;
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
// 11 here).  The layer's weights are brought into shared memory at once, which exposes one
// trip to the L2 where reading them class by class exposed a dozen.  For the logits a warp takes
// two rows and every fourth group of four classes (lanes along the input width); for the data
// gradient a thread takes two columns of the input and four rows.
// Dynamic shared memory: dZ [C][8], logits [8][C], the rows of A_{L-1} [8][in], W_L [C][in].
// With bf16 operands the two products are warp-level MMAs on bf16 copies (mma_tail): their reads of shared
// memory were what bounded the launch (333 x 100, P = 6, B = 50: 24 us, 13 now).
struct TailArgs {
  const float* a;                          // A_{L-1} [P, B, in]
  const float* w; const float* b; int64_t w_batch;
  const int32_t* labels;
  int P, B, in, C, row_blocks;
  float* row_loss;                         // [P, B]
  float* dz;                               // [P, B, C]
  float* dzp;                              // dZ_{L-1} [P, B, in], null for a one-layer model
  bool mma;                                // bf16 operands on warp-level MMAs (mma_tail)
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
  const float* W = t.w + (size_t)p * t.w_batch;
  const float* bias = t.b + (size_t)p * t.w_batch;
  const int n16 = ((c16 + 16) * ip + 16 * dp) / 8;
  for (int i = threadIdx.x; i < n16; i += kTailThreads) reinterpret_cast<uint4*>(w)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  // rows of `in` floats, contiguous from src on, to rows of ip
  auto fill = [&](__nv_bfloat16* dst, const float* __restrict__ src, int count) {
    const int head = min(count, (int)((16 - ((uintptr_t)src & 15)) & 15) / 4), n4 = (count - head) / 4;
    const float4* s4 = reinterpret_cast<const float4*>(src + head);
    for (int i0 = threadIdx.x; i0 < n4; i0 += 8 * kTailThreads) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (i0 + u * kTailThreads < n4) v[u] = s4[i0 + u * kTailThreads];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = i0 + u * kTailThreads;
        if (i >= n4) break;
        const int at = head + 4 * i;
        int r = at / in, k = at - r * in;
        const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          dst[r * ip + k] = __float2bfloat16_rn(x[j]);
          if (++k == in) { k = 0; ++r; }
        }
      }
    }
    const int rest = count - head - 4 * n4, x = threadIdx.x;
    if (x < head) dst[x / in * ip + x % in] = __float2bfloat16_rn(src[x]);
    if (x < rest) {
      const int at = head + 4 * n4 + x;
      dst[at / in * ip + at % in] = __float2bfloat16_rn(src[at]);
    }
  };
  fill(w, W, C * in);
  fill(a, t.a + ((size_t)p * t.B + r0) * in, rows * in);
  __syncthreads();
  const int i8 = lane / 8, j8 = lane % 8, qr = lane / 4, qc = 2 * (lane % 4);
  for (int nt = warp; nt < (C + 7) / 8; nt += kTailThreads / 32) {
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = 0; k0 < in16; k0 += 64) {            // 64 inputs' sum on its own: see multiply_mma
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      for (int k = k0; k < min(in16, k0 + 64); k += 16) {
        uint32_t fa[4], fb[2];
        tc::ldsm_x4(fa, a + ((i8 & 1) * 8 + j8) * ip + k + (i8 >> 1) * 8);
        tc::ldsm_x2(fb, w + (size_t)(nt * 8 + j8) * ip + k + (i8 & 1) * 8);
        tc::mma_bf16(d, fa, fb[0], fb[1]);
      }
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
    });
    if (lane == 0) t.row_loss[row] = loss;
  }
  if (!t.dzp) return;
  __syncthreads();
  for (int nt = warp; nt < (in + 7) / 8; nt += kTailThreads / 32) {
    float s[2] = {0.f, 0.f};
    for (int k0 = 0; k0 < c16; k0 += 64) {             // 64 classes' sum on its own, likewise
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      for (int k = k0; k < min(c16, k0 + 64); k += 16) {
        uint32_t fa[4], fb[2];
        tc::ldsm_x4(fa, dq + ((i8 & 1) * 8 + j8) * dp + k + (i8 >> 1) * 8);
        tc::ldsm_x2_t(fb, w + (size_t)(k + (i8 & 1) * 8 + j8) * ip + nt * 8);
        tc::mma_bf16(d, fa, fb[0], fb[1]);
      }
      s[0] += d[0];
      s[1] += d[1];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = nt * 8 + qc + h;
      if (qr < rows && i < in)                         // ReLU'(0) = 0
        t.dzp[((size_t)p * t.B + r0 + qr) * in + i] = __bfloat162float(a[qr * ip + i]) > 0.f ? s[h] : 0.f;
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
  const float* arow = t.a + ((size_t)p * t.B + r0) * in;
  float* w = a + kTailRows * in;
  copy_floats<QUANT>(w, W, C * in);
  copy_floats<false>(a, arow, rows * in);
  for (int i = rows * in + threadIdx.x; i < kTailRows * in; i += kTailThreads) a[i] = 0.f;
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
        if (rh + r < rows)
          t.dzp[((size_t)p * t.B + r0 + rh + r) * in + i] = a[(rh + r) * in + i] > 0.f ? s[h][r] : 0.f;
    }
  }
}

// Loss and dZ_L from the logits, for last layers too large for k_simt_tail.  Blocks 0..P-1: a learner's B
// rows, a warp per row; the remaining blocks gather the next step's minibatch.
template <bool QUANT>
__global__ void __launch_bounds__(1024)
k_simt_loss(const float* __restrict__ logits, const int32_t* __restrict__ labels, int P, int B, int C,
            float* __restrict__ row_loss, float* __restrict__ dz,
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
    });
    if (threadIdx.x % 32 == 0) row_loss[row] = loss;
  }
}

// ---------------------------------------------------------------------------------- host side
struct SimtBuffers {
  float* xg[2];                     // [P, B, d0], alternate steps
  int32_t* labels[2];               // [P, B]
  float* row_loss;                  // [P, B]
  float* a[MAVG_MAX_LAYERS + 1];    // a[l]  [P, B, d_l]: A_l, l < L; a[L]: the logits
  float* dz[MAVG_MAX_LAYERS + 1];   // dz[l] [P, B, d_l]
};

size_t carve(const mavg_config* cfg, char* base, SimtBuffers* sb) {
  const size_t rows = (size_t)cfg->P * cfg->B;
  size_t off = 0;
  auto take = [&](size_t words) {
    char* p = base + off;
    off += (words * 4 + 255) / 256 * 256;
    return p;
  };
  for (int i = 0; i < 2; ++i) {
    sb->xg[i] = (float*)take(rows * cfg->dims[0]);
    sb->labels[i] = (int32_t*)take(rows);
  }
  sb->row_loss = (float*)take(rows);
  for (int l = 1; l <= cfg->n_layers; ++l) {
    sb->a[l] = (float*)take(rows * cfg->dims[l]);
    sb->dz[l] = (float*)take(rows * cfg->dims[l]);
  }
  return off;
}

// Every launch of the chain may begin while its predecessor finishes; the kernels wait for it
// before they touch memory.
template <typename... Params, typename... Args>
cudaError_t launch(mavg_ctx* c, int cls, void (*kernel)(Params...), dim3 grid, int threads,
                   int cluster, size_t smem, Args... args) {
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

// The dense rows of `len` elements at p can be copied in groups of four.
bool vec4(const float* p, int64_t batch, int len) {
  return (uintptr_t)p % 16 == 0 && batch % 4 == 0 && len % 4 == 0;
}

int tiles_of(const GemmArgs& g) { return ((g.M + BM - 1) / BM) * ((g.N + BN - 1) / BN); }

// Forward / data gradient.  The contraction is halved until there are two blocks per SM, but a
// block keeps at least 64 of it (four slabs).
template <bool QUANT, int EPI>
cudaError_t launch_gemm(mavg_ctx* c, int cls, GemmArgs g) {
  const int P = c->cfg.P, tiles = tiles_of(g);
  int splits = 1;
  while (splits < kMaxSplit && (int64_t)tiles * P * splits < 2 * c->sm_count && g.K >= 128 * splits)
    splits *= 2;
  g.k_per_split = ((g.K + splits - 1) / splits + BK - 1) / BK * BK;
  return launch(c, cls, k_simt_gemm<QUANT, EPI>, dim3((unsigned)(tiles * splits), 1, (unsigned)P),
                kThreads, splits, 0, g, splits);
}

// Last layer in one launch (k_simt_tail) where its weights fit in an SM's shared memory.
constexpr size_t kTailSmem = 200 * 1024;
size_t tail_smem(int in, int C, bool quant) {
  if (quant)
    return ((size_t)((C + 15) / 16 * 16 + 16) * bf_pitch(in) + (size_t)16 * bf_pitch(C)) * 2 +
           (size_t)kTailRows * C * sizeof(float);
  return ((size_t)kTailRows * in + 2 * (size_t)kTailRows * C + (size_t)in * C) * sizeof(float);
}
bool use_tail(int in, int C) { return tail_smem(in, C, false) <= kTailSmem; }

// Every kernel of a step asks for the same split of the SM's memory: a launch that needs another
// split than the kernel before it has to wait until the SM is empty.
template <bool QUANT>
cudaError_t set_attributes() {
  const void* kernels[] = {
      (const void*)k_simt_gemm<QUANT, EPI_FWD>, (const void*)k_simt_gemm<QUANT, EPI_DGRAD>,
      (const void*)k_simt_wgrad<QUANT, false>, (const void*)k_simt_wgrad<QUANT, QUANT>, (const void*)k_simt_gather<QUANT>,
      (const void*)k_simt_loss<QUANT>, (const void*)k_simt_tail<QUANT>};
  for (const void* k : kernels) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
  }
  return cudaFuncSetAttribute(k_simt_tail<QUANT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kTailSmem);
}

template <bool QUANT>
cudaError_t step_impl(mavg_ctx* c, int64_t round, int step) {
  const mavg_config& cfg = c->cfg;
  const int P = cfg.P, B = cfg.B, L = cfg.n_layers;
  SimtBuffers sb;
  carve(&cfg, ws_ptr(c, c->ws.act), &sb);
  const int cur = step & 1;
  GatherArgs ga{};
  ga.x = cfg.x; ga.x_bf16 = cfg.x_dtype == MAVG_X_BF16;
  ga.y = cfg.y; ga.seed = cfg.seed; ga.round = round;
  ga.round_ptr = c->capturing ? (const int64_t*)(ws_ptr(c, c->ws.status) + 64) : nullptr;
  ga.step = step; ga.P = P; ga.B = B; ga.d = cfg.dims[0]; ga.S = cfg.n_samples;
  ga.out = sb.xg[cur]; ga.labels = sb.labels[cur];
  GatherArgs next = ga;
  next.step = step + 1; next.out = sb.xg[cur ^ 1]; next.labels = sb.labels[cur ^ 1];
  const int gather_rows = step < cfg.K ? P * B : 0;
  cudaError_t e;
  if (step == 1 &&
      (e = launch(c, MAVG_K_BATCH, k_simt_gather<QUANT>, dim3((unsigned)(P * B)), 256, 1, 0, ga)) != cudaSuccess)
    return e;
  // the weights before this step
  float* rep = c->buf.replicas;
  const int64_t rs = c->buf.replica_stride;
  const float* win = starts_from_global(c) ? c->buf.global_w : rep;
  const int64_t ws = starts_from_global(c) ? 0 : rs;
  const MomArgs mom = mom_args(c, c->replicas_equal_global);
  auto a_in = [&](int l) { return l == 1 ? sb.xg[cur] : sb.a[l - 1]; };
  const MlpLayer& top = c->layers[L - 1];
  const bool tail = use_tail(top.in, top.out);
  for (int l = 1; l <= (tail ? L - 1 : L); ++l) {
    const MlpLayer& ly = c->layers[l - 1];
    GemmArgs g{};
    g.A = a_in(l); g.a_batch = (int64_t)B * ly.in;
    g.B = win + ly.w_off; g.b_batch = ws;
    g.M = B; g.N = ly.out; g.K = ly.in;
    g.C = sb.a[l]; g.c_batch = (int64_t)B * ly.out;
    g.aux = win + ly.b_off; g.aux_batch = ws;
    g.vec_a = vec4(g.A, g.a_batch, g.K);
    g.vec_b = vec4(g.B, g.b_batch, g.K);
    g.vec_c = vec4(g.C, g.c_batch, g.N);
    g.hidden = l < L;
    if ((e = launch_gemm<QUANT, EPI_FWD>(c, MAVG_K_FWD, g)) != cudaSuccess) return e;
  }
  if (tail) {
    TailArgs t{};
    t.a = a_in(L); t.w = win + top.w_off; t.b = win + top.b_off; t.w_batch = ws;
    t.labels = sb.labels[cur];
    t.P = P; t.B = B; t.in = top.in; t.C = top.out; t.row_blocks = (B + kTailRows - 1) / kTailRows;
    t.row_loss = sb.row_loss; t.dz = sb.dz[L];
    if (L >= 2) t.dzp = sb.dz[L - 1];
    // few classes on very wide rows: their padding to 16 would not fit
    t.mma = QUANT && tail_smem(t.in, t.C, true) <= kTailSmem;
    if ((e = launch(c, MAVG_K_LOSS, k_simt_tail<QUANT>, dim3((unsigned)(P * t.row_blocks + gather_rows)),
                    kTailThreads, 1, tail_smem(t.in, t.C, t.mma), t, next)) != cudaSuccess)
      return e;
  } else {
    if ((e = launch(c, MAVG_K_LOSS, k_simt_loss<QUANT>, dim3((unsigned)(P + gather_rows)), 1024, 1, 0,
                    (const float*)sb.a[L], (const int32_t*)sb.labels[cur], P, B, top.out, sb.row_loss,
                    sb.dz[L], next)) != cudaSuccess)
      return e;
  }
  for (int l = tail ? L - 1 : L; l >= 2; --l) {
    const MlpLayer& ly = c->layers[l - 1];
    GemmArgs g{};
    g.A = sb.dz[l]; g.a_batch = (int64_t)B * ly.out;
    g.B = win + ly.w_off; g.b_batch = ws;
    g.M = B; g.N = ly.in; g.K = ly.out;
    g.C = sb.dz[l - 1]; g.c_batch = (int64_t)B * ly.in;
    g.aux = sb.a[l - 1]; g.aux_batch = g.c_batch;
    g.vec_a = vec4(g.A, g.a_batch, g.K);
    g.vec_b = vec4(g.B, g.b_batch, g.N);
    g.vec_c = vec4(g.C, g.c_batch, g.N);
    if ((e = launch_gemm<QUANT, EPI_DGRAD>(c, MAVG_K_DGRAD, g)) != cudaSuccess) return e;
  }
  WgradArgs w{};
  w.L = L;
  for (int l = 1; l <= L; ++l) {
    const MlpLayer& ly = c->layers[l - 1];
    GemmArgs& g = w.g[l - 1];
    g.A = sb.dz[l]; g.a_batch = (int64_t)B * ly.out;
    g.B = a_in(l); g.b_batch = (int64_t)B * ly.in;
    g.M = ly.out; g.N = ly.in; g.K = g.k_per_split = B;
    g.C = rep + ly.w_off; g.c_batch = rs;
    g.aux = win + ly.w_off; g.aux_batch = ws;
    g.vec_a = vec4(g.A, g.a_batch, g.M);
    g.vec_b = vec4(g.B, g.b_batch, g.N);
    g.vec_c = vec4(g.C, g.c_batch, g.N) && vec4(g.aux, g.aux_batch, g.N);
    g.bias = rep + ly.b_off; g.bias_in = win + ly.b_off;
    g.gamma = cfg.local_lr;
    g.mom = mom; g.u_off = ly.w_off; g.ub_off = ly.b_off;
    w.tile0[l] = w.tile0[l - 1] + tiles_of(g);
  }
  w.row_loss = sb.row_loss;
  w.loss_out = (float*)ws_ptr(c, c->ws.losses) + (step - 1);
  w.loss_stride = cfg.K;
  return launch(c, MAVG_K_WGRAD_SGD, B > kChainRows ? k_simt_wgrad<QUANT, QUANT> : k_simt_wgrad<QUANT, false>,
                dim3((unsigned)w.tile0[L], 1, (unsigned)P), kThreads, 1, 0, w);
}

}  // namespace

size_t simt_workspace_bytes(const mavg_config* cfg, size_t base, size_t* act_off) {
  *act_off = base;
  SimtBuffers sb;
  return base + carve(cfg, nullptr, &sb);
}

cudaError_t simt_setup(mavg_ctx* c) {
  return c->cfg.gemm_bf16 ? set_attributes<true>() : set_attributes<false>();
}

cudaError_t simt_step(mavg_ctx* c, int64_t round, int step) {
  return c->cfg.gemm_bf16 ? step_impl<true>(c, round, step) : step_impl<false>(c, round, step);
}

}  // namespace mavg
