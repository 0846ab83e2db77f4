// Rebuilt local steps: a learner's hidden weights after k steps, formed anew from w~, the momentum buffer the call found
// and the rows of the k steps' factors, instead of being read, stepped and written back every step.  With w~ the same for
// all learners and the rows a few MB, a step moves 2 bytes per weight (the bf16 copy that the next step's products read)
// and 4 more with learner momentum (u as it was before the call), where stepping in place moves 10 and 18.  The steps are
// taken one after the other in fp32, each from its own gradient's sum, and the weights are rounded to bf16 at every step: the
// plain form's numbers, to the bit.
//
// 3072-2048-2048-2048-10, P = 8, B = 64, momentum (14.7 M weights a learner), step 1 .. 4 of 4: 145, 164, 194 us against 116 us
// for the 0.76 GB of steps 1 .. 3 at the copy rate, and 386 against 222 (1.47 GB: W and u go out); the round takes 1447 us,
// 1928 with the steps in place.  What bounds steps 1 .. 3 is what an SM takes in from the L2, about 49 GB/s: 32 KB of operands
// per tile and step so far beside 64 KB of u, 95, 127 and 158 us.  The last step waits for its stores and, with all of
// tensor memory taken by one learner's four gradients, for the next learner's.  Registers: four steps' accumulators of
// 8 columns at once spilled (166, 184, 236 and 437 us), two at once do not.  Measured and worse: more groups, or eight
// warps a group; storing from registers (296 .. 560 us: half-empty sectors); deeper rings with two operand stages; in the
// last step pieces of 16 columns, two in turn (400); the copies in and out by warps of their own (137, 151, 238 and 423).
// Without momentum an accumulator is read and given back at a time (two at a time: 1.04 times as long over 25 shapes).  All
// steps' gradients in one accumulator took 0.76 to 1 of the time but rounded the weights once, and not at every step.
#pragma once
#include <cuda.h>

#include "gemm_unit.cuh"
#include "wgrad_tc.cuh"

namespace mavg {
namespace rebuild {

using namespace tc;
using namespace gemm;

constexpr int kGroups = 4;                        // of four epilogue warps: one for each piece of a tile
constexpr int kThreads = (2 + 4 * kGroups) * 32;  // warp 0: TMA producer, 1: MMA issuer, the rest: epilogue
constexpr int kBN = 128;                          // input columns of a tile
constexpr int kPiece = 32;                        // columns of a piece: 16 KB of fp32, rows of 128 bytes, 128-byte swizzle
constexpr int kPieceBytes = kBM * kPiece * 4;
constexpr int kStageBytes = 2 * kATileBytes;
// Shared memory: operand stages and, per epilogue group, buffers for pieces on their way in (w~, u) and one to store from.
// What leaves with LAST takes fp32 pieces of W, and u where it came in, so one piece less comes in ahead.
constexpr int stages_of(bool last) { return last ? 3 : 2; }
constexpr int ring_of(bool last) { return last ? 1 : 2; }
constexpr int out_bytes(bool last) { return last ? kPieceBytes : kPieceBytes / 2; }
constexpr int group_bytes(bool last) { return ring_of(last) * kPieceBytes + out_bytes(last); }
constexpr size_t smem_of(bool last) { return (size_t)stages_of(last) * kStageBytes + kGroups * group_bytes(last) + 1024; }
static_assert(smem_of(false) <= 226 * 1024 && smem_of(true) <= 226 * 1024, "");
constexpr int kAccs = 512 / kBN;                  // every step's gradient has an accumulator of its own
constexpr int kMaxMomSteps = kAccs;               // with momentum all of a learner's are taken together
static_assert(kMaxMomSteps == 4, "reb_steps");
enum { ERR_REB_PRODUCER = 51, ERR_REB_MMA = 52, ERR_REB_EPILOGUE = 53 };

struct Layer { int m_tiles, n_tiles, in, first; };   // first: tiles of the layers before
struct Args {
  CUtensorMap dz[MAVG_MAX_LAYERS], a[MAVG_MAX_LAYERS];   // rows [steps P, B, d], boxes of 64 features x 64 rows
  CUtensorMap w_in[MAVG_MAX_LAYERS], u[MAVG_MAX_LAYERS];    // w~ and u, fp32 pieces
  CUtensorMap out[MAVG_MAX_LAYERS];                    // the bf16 copies, or (LAST) the fp32 masters
  Layer layer[MAVG_MAX_LAYERS];
  int n_layers, tiles, P, group;                  // tiles of a learner; learners that share a fetch of w~
  int B, steps;                                   // steps taken so far, B rows each
  int load_u;                                     // u is not zero
  float gamma, beta;
  int* status;
};
struct alignas(16) Shared {                       // (whole 16 bytes, as static shared memory is counted)
  uint64_t full[3], empty[3], acc_full[4], acc_empty[4], piece_full[kGroups][2];
  uint32_t tmem_slot;
  int abort_flag;
  int fetch_unit[kGroups], fetch_p[kGroups], fetched[kGroups];   // a group's place in its list of pieces to fetch
};

// Dynamic shared memory of a launch: at least the same share of an SM as of its tensor memory, of which a block takes all.
inline size_t launch_bytes(bool last) {
  const size_t share = tmem_share_bytes(512, sizeof(Shared));
  return smem_of(last) > share ? smem_of(last) : share;
}

// Persistent over units: a tile of 128 x 128 weights for `group` learners, whose w~ stays in the epilogue's registers (a
// fetch of w~ for every learner is 4 bytes per weight more, twice what leaves in steps 1 .. K-1 without momentum).
// LAST: the learners' own weights and u leave, else the bf16 copies of the weights.
template <bool MOM, bool LAST>
__global__ void __launch_bounds__(kThreads, 1)
k_rebuild(const __grid_constant__ Args g) {
  constexpr int kStages = stages_of(LAST);
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(16) Shared sh;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    for (int b = 0; b < 4; ++b) {
      mbar_init(&sh.acc_full[b], 1);
      mbar_init(&sh.acc_empty[b], 4 * kGroups);
    }
    for (int b = 0; b < kGroups; ++b)
      for (int s = 0; s < 2; ++s) mbar_init(&sh.piece_full[b][s], 1);
    sh.abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async();
  }
  uint32_t* tmem_slot = &sh.tmem_slot;
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = sh.tmem_slot;
  grid_launch_dependents();   // not before the tensor memory is this block's: see tc_ptx.cuh
  grid_dependency_wait();
  volatile int* abortp = &sh.abort_flag;
  const int nkb = (g.B + kBK - 1) / kBK;          // slabs of a step
  // Tensor memory as a ring of four accumulators, of which a learner takes one per step (a learner's at a time, twice
  // where they fit twice: 146, 158, 225 and 370 us, the round 1463)
  const int accs = g.steps;
  const int groups = (g.P + g.group - 1) / g.group, units = groups * g.tiles;
  // units of the same learners follow one another: their rows stay in the L2
  auto decode = [&](int unit, int& p0, int& p1, int& l, int& m0, int& n0) {
    const int gr = unit / g.tiles;
    int r = unit - gr * g.tiles;
    p0 = gr * g.group;
    p1 = min(p0 + g.group, g.P);
    l = 0;
    while (l + 1 < g.n_layers && r >= g.layer[l + 1].first) ++l;
    r -= g.layer[l].first;
    m0 = (r % g.layer[l].m_tiles) * kBM;
    n0 = (r / g.layer[l].m_tiles) * kBN;
  };

  if (warp == 0) {
    if (lane == 0) {
      int issued = 0;
      bool ok = true;
      for (int unit = blockIdx.x; unit < units && ok; unit += gridDim.x) {
        int p0, p1, l, m0, n0;
        decode(unit, p0, p1, l, m0, n0);
        for (int p = p0; p < p1 && ok; ++p)
          for (int i = 0; i < g.steps * nkb; ++i, ++issued) {
            const int s = issued % kStages, row = i % nkb * kBK, z = i / nkb * g.P + p;
            if (!(ok = mbar_wait(&sh.empty[s], ((issued / kStages) & 1) ^ 1, abortp, g.status, ERR_REB_PRODUCER))) break;
            uint8_t* sa = smem + (size_t)s * kStageBytes;
            mbar_arrive_expect_tx(&sh.full[s], (uint32_t)kStageBytes);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              tma_load_3d(sa + h * 8192, &g.dz[l], &sh.full[s], m0 + 64 * h, row, z);
              tma_load_3d(sa + kATileBytes + h * 8192, &g.a[l], &sh.full[s], n0 + 64 * h, row, z);
            }
          }
      }
      if (*abortp) drain_copies(sh.full, issued, kStages, g.status);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_f32(kBM, kBN, 1, 1);
      const uint64_t a0 = smem_desc_mn_sw128(smem_u32(smem)), b0 = smem_desc_mn_sw128(smem_u32(smem) + kATileBytes);
      int it = 0, n = 0;
      bool ok = true;
      for (int unit = blockIdx.x; unit < units && ok; unit += gridDim.x) {
        int p0, p1, l, m0, n0;
        decode(unit, p0, p1, l, m0, n0);
        for (int p = p0; p < p1 && ok; ++p)
          for (int i = 0; i < g.steps * nkb; ++i, ++it) {
            const int s = it % kStages, kb = i % nkb, b = n & 3;
            const bool first = kb == 0, last = kb == nkb - 1;
            if (first && !(ok = mbar_wait(&sh.acc_empty[b], ((n >> 2) & 1) ^ 1, abortp, g.status, ERR_REB_MMA))) break;
            if (!(ok = mbar_wait(&sh.full[s], (it / kStages) & 1, abortp, g.status, ERR_REB_MMA))) break;
            tc_fence_after_sync();
            const uint32_t off = (uint32_t)(s * kStageBytes) >> 4, d = tmem_base + (uint32_t)(b * kBN);
            // a step's last slab ends with its batch (a multiple of 16)
            const int nk = min(kBK, g.B - kb * kBK) / 16;
            for (int k = 0; k < nk; ++k)
              umma_bf16(d, a0 + off + (uint32_t)k * ((16 * 128) >> 4), b0 + off + (uint32_t)k * ((16 * 128) >> 4), idesc,
                        (uint32_t)(!first || k > 0));
            umma_commit(&sh.empty[s]);
            if (last) {
              umma_commit(&sh.acc_full[b]);
              ++n;
            }
          }
      }
    }
    __syncwarp();
  } else {
    // A group of four warps per piece.  Its first thread fetches w~ and u pieces ahead of their use and stores the finished
    // ones.  One barrier a piece: behind it the piece has been read and what is to be stored is in shared memory; before
    // the next is written, the first thread has seen the store leave it (it carries that to the barrier before the write).
    // The barriers carry a wait that was given up, so that the group leaves together.
    constexpr int kRing = MOM ? ring_of(LAST) : 1;   // (without momentum w~'s pieces alone come in)
    const int grp = (warp - 2) >> 2, q4 = warp & 3, row = q4 * 32 + lane;
    const bool leader = ((warp - 2) & 3) == 0 && lane == 0, load_u = MOM && g.load_u;
    const bool u_apart = MOM && LAST && !load_u;   // u does not come in, but leaves from the buffer for it
    uint8_t* in_buf = smem + kStages * kStageBytes + (size_t)grp * group_bytes(LAST);
    uint8_t* ob = in_buf + ring_of(LAST) * kPieceBytes;
    uint8_t* between = LAST ? ob : in_buf + kPieceBytes;   // not MOM: weights after four steps, each thread's own
    // the leader's place in the group's list of pieces: of w~ (fp == -1), then of each learner's u
    // (in shared memory: it is seldom looked at, and registers are short)
    auto fetch = [&]() {
      int fu = sh.fetch_unit[grp], fp = sh.fetch_p[grp];
      while (fu < units) {
        int p0, p1, l, m0, n0;
        decode(fu, p0, p1, l, m0, n0);
        const int c0 = n0 + grp * kPiece, of = fp, last_of = load_u ? p1 - p0 : 0;
        if (++fp >= last_of || c0 >= g.layer[l].in) { fp = -1; fu += gridDim.x; }
        if (c0 >= g.layer[l].in) continue;
        const uint32_t s = (uint32_t)sh.fetched[grp]++ % kRing;
        sh.fetch_unit[grp] = fu;
        sh.fetch_p[grp] = fp;
        mbar_arrive_expect_tx(&sh.piece_full[grp][s], kPieceBytes);
        if (of < 0) tma_load_3d(in_buf + (size_t)s * kPieceBytes, &g.w_in[l], &sh.piece_full[grp][s], c0, m0, 0);
        else tma_load_3d(in_buf + (size_t)s * kPieceBytes, &g.u[l], &sh.piece_full[grp][s], c0, m0, p0 + of);
        return;
      }
      sh.fetch_unit[grp] = fu;
    };
    if (leader) {
      sh.fetch_unit[grp] = blockIdx.x;
      sh.fetch_p[grp] = -1;
      sh.fetched[grp] = 0;
      for (int i = 0; i < kRing; ++i) fetch();
    }
    uint32_t pn = 0;                               // pieces taken in
    int n = 0;                                     // accumulators taken before this learner's
    bool failed = false, gone = false;
    auto cell = [&](uint8_t* buf, int c) { return reinterpret_cast<float4*>(buf + (size_t)row * 128 + ((c ^ (row & 7)) << 4)); };
    auto wait_piece = [&]() {
      if (!mbar_wait(&sh.piece_full[grp][pn % kRing], (pn / kRing) & 1, abortp, g.status, ERR_REB_EPILOGUE)) failed = true;
      return in_buf + (size_t)(pn % kRing) * kPieceBytes;
    };
    auto put_fp32 = [&](uint8_t* buf, int h, const float (&x)[8]) {
#pragma unroll
      for (int c = 0; c < 2; ++c) *cell(buf, 2 * h + c) = make_float4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
    };
    auto put_bf16 = [&](int h, const float (&x)[8]) {   // rows of 64 bytes, 64-byte swizzle
      uint32_t hw[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const __nv_bfloat162 t = __floats2bfloat162_rn(x[2 * j], x[2 * j + 1]);
        hw[j] = *reinterpret_cast<const uint32_t*>(&t);
      }
      *reinterpret_cast<uint4*>(ob + (size_t)row * 64 + ((h ^ ((row >> 1) & 3)) << 4)) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    };
    for (int unit = blockIdx.x; unit < units && !gone; unit += gridDim.x) {
      int p0, p1, l, m0, n0;
      decode(unit, p0, p1, l, m0, n0);
      const int c0 = grp * kPiece;
      const bool mine = n0 + c0 < g.layer[l].in;
      float w[kPiece];
      if (mine) {
        uint8_t* buf = wait_piece();
#pragma unroll
        for (int c = 0; c < kPiece / 4; ++c) {
          const float4 v = *cell(buf, c);
          w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
        }
        ++pn;
        if (leader) tma_store_wait_read<0>();      // (the store before the first write of this unit)
        if ((gone = barrier_any(failed, 2 + grp, 128))) break;
        if (leader && !u_apart) fetch();
      }
      for (int p = p0; p < p1; ++p, n += accs) {
        const uint32_t acc = tmem_base + ((uint32_t)(q4 * 32) << 16) + (uint32_t)c0;
        uint8_t* ub = in_buf;
        if (MOM) {                                 // all of the learner's accumulators together
          for (int i = n; i < n + accs; ++i)
            if (!mbar_wait(&sh.acc_full[i & 3], (i >> 2) & 1, abortp, g.status, ERR_REB_EPILOGUE)) failed = true;
          __syncwarp();
          tc_fence_after_sync();
          if (mine && load_u) ub = wait_piece();
          if (mine) {
#pragma unroll
            for (int h = 0; h < kPiece / 8; ++h) {   // 8 columns
              float x[8], v[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                x[j] = w[8 * h + j];
                v[j] = 0.f;
              }
              if (load_u) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                  const float4 t = *cell(ub, 2 * h + c);
                  v[4 * c] = t.x; v[4 * c + 1] = t.y; v[4 * c + 2] = t.z; v[4 * c + 3] = t.w;
                }
              }
#pragma unroll
              for (int i = 0; i < kMaxMomSteps; i += 2) {   // two steps at a time: more accumulators in flight do not fit the registers
                if (i >= g.steps) break;
                uint32_t r[2][8];
                tmem_ld_8cols(acc + (uint32_t)(((n + i) & 3) * kBN + 8 * h), r[0]);
                if (i + 1 < g.steps) tmem_ld_8cols(acc + (uint32_t)(((n + i + 1) & 3) * kBN + 8 * h), r[1]);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j) msgd(x[j], v[j], __uint_as_float(r[0][j]), g.gamma, g.beta);
                if (i + 1 < g.steps)
#pragma unroll
                  for (int j = 0; j < 8; ++j) msgd(x[j], v[j], __uint_as_float(r[1][j]), g.gamma, g.beta);
              }
              if (LAST) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                  *cell(ob, 2 * h + c) = make_float4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
                  *cell(ub, 2 * h + c) = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
                }
              } else {
                put_bf16(h, x);
              }
            }
          }
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0)
            for (int i = n; i < n + accs; ++i) mbar_arrive(&sh.acc_empty[i & 3]);
        } else {                                   // up to four at a time; between the fours the weights stay in shared memory
          for (int done = 0; done < accs; done += kAccs) {
            const int begin = n + done, end = n + min(done + kAccs, accs);
            for (int i = begin; i < end; ++i)
              if (!mbar_wait(&sh.acc_full[i & 3], (i >> 2) & 1, abortp, g.status, ERR_REB_EPILOGUE)) failed = true;
            __syncwarp();
            tc_fence_after_sync();
            if (mine) {
#pragma unroll
              for (int h = 0; h < kPiece / 8; ++h) {
                float x[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = w[8 * h + j];
                if (done > 0) {
#pragma unroll
                  for (int c = 0; c < 2; ++c) {
                    const float4 t = *cell(between, 2 * h + c);
                    x[4 * c] = t.x; x[4 * c + 1] = t.y; x[4 * c + 2] = t.z; x[4 * c + 3] = t.w;
                  }
                }
#pragma unroll 1
                for (int i = begin; i < end; ++i) {
                  uint32_t r[8];
                  tmem_ld_8cols(acc + (uint32_t)((i & 3) * kBN + 8 * h), r);
                  tmem_ld_wait();
#pragma unroll
                  for (int j = 0; j < 8; ++j) x[j] = fmaf(-g.gamma, __uint_as_float(r[j]), x[j]);
                }
                if (LAST) put_fp32(ob, h, x);
                else if (end < n + accs) put_fp32(between, h, x);
                else put_bf16(h, x);
              }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0)
              for (int i = begin; i < end; ++i) mbar_arrive(&sh.acc_empty[i & 3]);
          }
        }
        if (!mine) continue;                       // (a wait given up here is carried by the next barrier)
        fence_proxy_async();
        if ((gone = barrier_any(failed, 2 + grp, 128))) break;
        if (leader) {
          tma_store_3d(&g.out[l], ob, n0 + c0, m0, p);
          if (MOM && LAST) tma_store_3d(&g.u[l], ub, n0 + c0, m0, p);
          tma_store_commit();
        }
        if (load_u) ++pn;
        if (leader && load_u && !LAST) fetch();    // (its buffer has been read)
        if (leader) tma_store_wait_read<0>();
        if (leader && load_u && LAST) fetch();     // (its buffer has been stored from)
        if ((gone = barrier_any(failed, 2 + grp, 128))) break;
      }
      if (leader && mine && u_apart && !gone) fetch();
    }
    if (leader) {
      tma_store_wait_read<0>();
      if (*abortp) drain_copies(sh.piece_full[grp], sh.fetched[grp], kRing, g.status);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

}  // namespace rebuild
}  // namespace mavg
