// Backward of the masked attention, rows kernel: dQ and the row statistics.
//
// Persistent, one CTA per SM; a work item is one (b, h, query tile), handed out through a counter (late query
// tiles of a head first, heads in order, so that concurrent CTAs share a few heads' K and V in L2).
// An item follows the query tile's rounds (up to eight non-empty 16-column groups each).  Per round:
//   S  = Q K^T, dP = dO V^T   tcgen05.mma, fp32 accumulators in TMEM
//   dS = 2^(c S - r) (dP - D) by two threads per query row (32-column chunks alternate between them), written
//                             as 16-bit values over S in TMEM
//   dQ += dS K                tcgen05.mma, A = dS from TMEM, B = the same K rows read MN-major
// ONE sweep: the exponent's reference r is an online softmax's running maximum, the weights' sum l is
// collected beside it, dQ is rescaled where the reference moves (lazily, by 2^8) and divided by l at the
// end.  dS then carries the factor l, which bf16's exponent takes; fp16 cannot, so fp16 tensors sweep their
// rounds twice (kF16): S alone for r = log2 of the row's sum, then the above with that fixed reference.
//
// Warp roles (448 threads): warps 0-7 compute, 8 producer (TMA ring of K, V, bitmap), 9 issues every MMA,
// 10-13 form D_i = dO_i . O_i of the NEXT item straight from global memory and write the last item's dQ,
// -log2 sum and D.  TMEM (512 columns): S[2], dP, dQ.  The issuer runs one round ahead: S(g+1) and dP(g+1)
// are under way while the threads work on round g; dP has one buffer, which the threads release as soon as
// it is in registers.
//
// What bounds it: per round 24 products of 128 x 128 x 16 (measured 79 cycles each) and one exponential per
// score (1024 cycles).  The version it replaces had one CTA per query tile, two sweeps and every step
// waiting for the one before: 402 us on 4 x 16 heads, 4096 tokens, d = 128, 5 % kept (8 176 rounds), 110 us on
// 64 x 8 heads, 250 x 231, d = 64.
#include <math_constants.h>

#include "ap_bwd_tc.cuh"

namespace ap {
namespace bwd {

namespace {

using namespace pipe;

constexpr int kThreads = 448;
constexpr int kComputeWarps = 8;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemDp = 256, kTmemDq = 384;
constexpr int kItemRing = 8;

constexpr uint32_t kInfoSlots = 15u;
constexpr uint32_t kInfoFirst = 1u << 4;  // first round of its sweep
constexpr uint32_t kInfoLast = 1u << 5;   // last round of its sweep
constexpr uint32_t kInfoFull = 1u << 6;   // every entry kept: no bitmap was copied
constexpr uint32_t kInfoStop = 1u << 7;
constexpr uint32_t kInfoStats = 1u << 8;  // (fp16) first sweep: S only

template <int kStages>
struct Shared {
  alignas(16) uint32_t bitmap[kStages][kTile][4];
  float2 ml[4][2][kTile];       // [item % 4][column half][row]: (reference, sum)
  float xchg[2][2][kTile];      // [round % 2][column half][row]: maximum
  float dsum[2][kTile];         // D of item n at [n % 2]
  uint64_t q_full, q_empty;
  uint64_t kv_full[kStages], kv_empty[kStages];
  uint64_t s_full[2], ds_full[2], dq_done[2];
  uint64_t dp_full, dp_free;
  uint64_t o_done, o_free;      // dQ of the item complete / read out
  uint64_t ml_ready[4], d_ready[2], item_ready[kItemRing];
  uint64_t pair[4];             // the two warps that share 32 rows
  int32_t item_bh[kItemRing], item_qt[kItemRing];  // qt = -1: no more items
  uint32_t info[kStages];
  uint32_t tmem_base;
  int abort_flag;
};

template <int D, bool kSplit>
struct Cfg {
  using L = TileLayout<D, kSplit>;
  static constexpr int kStages = D == 64 ? 4 : 2;
  static constexpr int kDoOffset = L::kBytes;
  static constexpr int kStageOffset = 2 * L::kBytes;
  static constexpr int kStageBytes = 2 * L::kBytes;
  static constexpr int kOutOffset = kStageOffset + kStages * kStageBytes;  // 4 KB per epilogue warp
  static constexpr int kSharedOffset = kOutOffset + 4 * 4096;
  static constexpr int kSmemBytes = kSharedOffset + (int)sizeof(Shared<kStages>) + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory");
  static_assert(kSmemBytes > 114 * 1024, "one CTA per SM: all of TMEM is taken");
};

template <int D, bool kSplit, bool kF16>
__global__ void __launch_bounds__(kThreads, 1)
rows_kernel(const __grid_constant__ RowsMaps maps, const uint16_t *__restrict__ O, const uint16_t *__restrict__ dO,
            uint16_t *__restrict__ dQ, float *__restrict__ neg_l, float *__restrict__ stat_d, int32_t *__restrict__ next,
            const int32_t *__restrict__ round_ptr, const int32_t *__restrict__ round_rows,
            const uint8_t *__restrict__ round_info, const uint32_t *__restrict__ round_bitmap, int n_items, int H,
            int Lq, int n_qt, float scale, unsigned *err, uint32_t max_polls, int dbg_skip) {
  using C = Cfg<D, kSplit>;
  using L = TileLayout<D, kSplit>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *q_s = smem, *do_s = smem + C::kDoOffset, *stage_s = smem + C::kStageOffset;
  auto *sh = reinterpret_cast<Shared<C::kStages> *>(smem + C::kSharedOffset);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    mbar_init(&sh->q_full, 1);
    mbar_init(&sh->q_empty, 1);
    for (int i = 0; i < C::kStages; ++i) {
      mbar_init(&sh->kv_full[i], 1);
      mbar_init(&sh->kv_empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh->s_full[i], 1);
      mbar_init(&sh->ds_full[i], kComputeWarps);
      mbar_init(&sh->dq_done[i], 1);
      mbar_init(&sh->d_ready[i], 4);
    }
    for (int i = 0; i < 4; ++i) mbar_init(&sh->pair[i], 2);
    mbar_init(&sh->dp_full, 1);
    mbar_init(&sh->dp_free, kComputeWarps);
    mbar_init(&sh->o_done, 1);
    mbar_init(&sh->o_free, 4);
    for (int i = 0; i < 4; ++i) mbar_init(&sh->ml_ready[i], kComputeWarps);
    for (int i = 0; i < kItemRing; ++i) mbar_init(&sh->item_ready[i], 1);
    sh->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 9) {
    tmem_alloc(&sh->tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sh->tmem_base;
  const Waiter wait{&sh->abort_flag, err, max_polls};

  if (warp == 8) {
    // ------------------------------------------------------------ producer
    if (lane < 4) {
      prefetch_tensormap(&maps.k[lane]);
      prefetch_tensormap(&maps.v[lane]);
    } else if (lane == 4) {
      prefetch_tensormap(&maps.q);
      prefetch_tensormap(&maps.d_o);
    }
    bool ok = dbg_skip == 0;  // (test hook: nothing is copied, the other roles' waits run out)
    uint32_t g = 0, n = 0;    // rounds / non-empty items so far
    int q_armed = -1;         // item whose Q and dO were copied last
    // the next item's number is drawn while the current one is under way, its rounds looked up with it
    auto draw = [&]() {
      int x = 0;
      if (lane == 0) x = atomicAdd(next, 1);  // (every CTA begins with the item of its own number)
      return (int)gridDim.x + __shfl_sync(0xffffffffu, x, 0);
    };
    struct Item {
      int bh, qt, r0, r1;
    };
    auto look_up = [&](int k) {
      Item it{0, -1, 0, 0};
      if (k < n_items) {
        it.bh = k / n_qt;
        it.qt = n_qt - 1 - k % n_qt;
        const int lr = (it.bh % H) * n_qt + it.qt;
        it.r0 = (int)ldg_now_u32(round_ptr + lr);
        it.r1 = (int)ldg_now_u32(round_ptr + lr + 1);
      }
      return it;
    };
    Item cur = look_up((int)blockIdx.x);
    int k_next = ok ? draw() : n_items;
    while (ok && cur.qt >= 0) {
      const Item it = cur;
      cur = look_up(k_next);
      if (cur.qt >= 0) k_next = draw();
      if (it.r0 == it.r1) {  // nothing kept: dQ is zero, and no key block visits the tile
        const int rows = min(kTile, Lq - it.qt * kTile);
        uint4 *dst = reinterpret_cast<uint4 *>(dQ + ((size_t)it.bh * Lq + (size_t)it.qt * kTile) * D);
        for (int x = lane; x < rows * (D / 8); x += 32) dst[x] = make_uint4(0u, 0u, 0u, 0u);
        continue;
      }
      if (lane == 0) {
        sh->item_bh[n % kItemRing] = it.bh;
        sh->item_qt[n % kItemRing] = it.qt;
        mbar_arrive(&sh->item_ready[n % kItemRing]);
      }
      ok = wait(&sh->q_empty, (n & 1u) ^ 1u);
      if (!ok) break;
      q_armed = (int)n;
      if (lane == 0) {
        mbar_arrive_expect_tx(&sh->q_full, 2 * L::kBytes);
#pragma unroll
        for (int s = 0; s < L::kSub; ++s) {
          tma_load_3d(q_s + s * kSubBytes, &maps.q, &sh->q_full, 64 * s, it.qt * kTile, it.bh);
          tma_load_3d(do_s + s * kSubBytes, &maps.d_o, &sh->q_full, 64 * s, it.qt * kTile, it.bh);
        }
      }
      __syncwarp();
      for (int sweep = kF16 ? 0 : 1; sweep < 2 && ok; ++sweep) {
        int row = lane < 8 ? (int)ldg_now_u32(round_rows + (size_t)it.r0 * 8 + lane) : -1;
        uint32_t rinfo = ldg_now_u8(round_info + it.r0);
        for (int v = it.r0; v < it.r1; ++v, ++g) {
          const int my_row = row;
          const uint32_t my_info = rinfo;
          if (v + 1 < it.r1) {
            row = lane < 8 ? (int)ldg_now_u32(round_rows + (size_t)(v + 1) * 8 + lane) : -1;
            rinfo = ldg_now_u8(round_info + v + 1);
          }
          const int ng = (int)(my_info & 15u);
          const bool full = (my_info & 0x80u) != 0u;
          const int run = run_of_slots(lane, ng, my_row);
          const int st = (int)(g % C::kStages);
          ok = wait(&sh->kv_empty[st], ((g / C::kStages) & 1u) ^ 1u);
          if (!ok) break;
          unsigned char *k_st = stage_s + st * C::kStageBytes;
          if (lane == 0) {
            sh->info[st] = (uint32_t)ng | (v == it.r0 ? kInfoFirst : 0u) | (v + 1 == it.r1 ? kInfoLast : 0u) |
                           (full ? kInfoFull : 0u) | (sweep == 0 ? kInfoStats : 0u);
            mbar_arrive_expect_tx(&sh->kv_full[st], (uint32_t)ng * (sweep == 0 ? 16u : 32u) * D * 2u +
                                                        (full ? 0u : (uint32_t)kBitmapWords * 4u));
            if (!full)
              bulk_load(&sh->bitmap[st][0][0], round_bitmap + (size_t)v * kBitmapWords, kBitmapWords * 4, &sh->kv_full[st]);
          }
          __syncwarp();
          if (run > 0) {
            load_run<D, kSplit>(k_st, maps.k, &sh->kv_full[st], lane, my_row, run, it.bh);
            if (sweep == 1) load_run<D, kSplit>(k_st + L::kBytes, maps.v, &sh->kv_full[st], lane, my_row, run, it.bh);
          }
          __syncwarp();
        }
      }
      ++n;
    }
    if (ok) {
      const int st = (int)(g % C::kStages);
      ok = wait(&sh->kv_empty[st], ((g / C::kStages) & 1u) ^ 1u);
      if (ok && lane == 0) {
        sh->info[st] = kInfoStop;
        mbar_arrive(&sh->kv_full[st]);
        sh->item_qt[n % kItemRing] = -1;
        mbar_arrive(&sh->item_ready[n % kItemRing]);
      }
    }
    if (!ok && dbg_skip == 0 && lane == 0) {
      // winding down: wait (bounded) for the copies armed most recently
      if (q_armed >= 0) mbar_wait(&sh->q_full, (uint32_t)q_armed & 1u, 1u << 16);
      for (uint32_t a = g > (uint32_t)C::kStages ? g - C::kStages : 0; a < g; ++a)
        mbar_wait(&sh->kv_full[a % C::kStages], (a / C::kStages) & 1u, 1u << 16);
    }
  } else if (warp == 9) {
    // ------------------------------------------------------------ issuer of all products
    const uint32_t q_lo = smem_desc_lo(smem_u32(q_s), 16), do_lo = smem_desc_lo(smem_u32(do_s), 16);
    const uint32_t stage_lo = smem_desc_lo(smem_u32(stage_s), 16), stage_mn = smem_desc_lo(smem_u32(stage_s), L::kSlabStride);
    constexpr uint32_t idesc_dq = idesc_bf16_f32(128, D, false, true, kF16);
    uint32_t n_front = 0, n_back = 0;  // items started by S / by dQ
    uint32_t info_front = 0u;
    bool ok = true;
    // S and dP of round g; false at the end of the work or after an expired wait (ok tells which)
    auto front = [&](uint32_t g) {
      const int st = (int)(g % C::kStages);
      const uint32_t sb = g & 1u;
      ok = wait(&sh->kv_full[st], (g / C::kStages) & 1u);
      if (!ok) return false;
      info_front = sh->info[st];
      if (info_front & kInfoStop) return false;
      const bool stats = kF16 && (info_front & kInfoStats);
      const bool first = (info_front & kInfoFirst) != 0u, last = (info_front & kInfoLast) != 0u;
      if (first && (!kF16 || stats)) ok = wait(&sh->q_full, n_front & 1u);
      // the S buffer held dS of round g - 2 until that round's dQ += dS K was over
      if (ok && g >= 2) ok = wait(&sh->dq_done[sb], ((g >> 1) - 1u) & 1u);
      if (!ok) return false;
      tc_fence_after_sync();
      const uint32_t idesc = idesc_bf16_f32(128, 16 * (int)(info_front & kInfoSlots), false, false, kF16);
      const uint32_t k_lo = stage_lo + st * (C::kStageBytes >> 4);
      if (elect_one()) {
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t a_step = (ks / 4) * (kSubBytes >> 4) + (ks % 4) * 2;
          const uint32_t b_step = (ks / 4) * (L::kSlabStride >> 4) + (ks % 4) * 2;
          mma_ss<smem_desc_hi_sw128(1024), smem_desc_hi_sw128(L::kSbo)>(tmem + 128u * sb, q_lo + a_step, k_lo + b_step, idesc, ks > 0);
        }
        mma_commit(&sh->s_full[sb]);
      }
      __syncwarp();
      // dP of the previous round is in the threads' registers
      if (g >= 1) ok = wait(&sh->dp_free, (g - 1u) & 1u);
      if (!ok) return false;
      tc_fence_after_sync();
      if (elect_one()) {
        if (!stats) {
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t a_step = (ks / 4) * (kSubBytes >> 4) + (ks % 4) * 2;
            const uint32_t b_step = (L::kBytes >> 4) + (ks / 4) * (L::kSlabStride >> 4) + (ks % 4) * 2;
            mma_ss<smem_desc_hi_sw128(1024), smem_desc_hi_sw128(L::kSbo)>(tmem + kTmemDp, do_lo + a_step, k_lo + b_step, idesc, ks > 0);
          }
          if (last) mma_commit(&sh->q_empty);
        }
        mma_commit(&sh->dp_full);
      }
      __syncwarp();
      if (last && !stats) ++n_front;
      return true;
    };
    bool more = front(0);
    for (uint32_t g = 0; more; ++g) {
      const uint32_t info = info_front;
      more = front(g + 1);
      if (!ok) break;
      const int st = (int)(g % C::kStages);
      const uint32_t sb = g & 1u;
      const int ng = (int)(info & kInfoSlots);
      const bool stats = kF16 && (info & kInfoStats);
      const bool first = (info & kInfoFirst) != 0u, last = (info & kInfoLast) != 0u;
      // the first round of an item overwrites dQ: the previous item's must have been read
      if (first && !stats && n_back > 0) ok = wait(&sh->o_free, (n_back - 1u) & 1u);
      if (ok) ok = wait(&sh->ds_full[sb], (g >> 1) & 1u);
      if (!ok) break;
      tc_fence_after_sync();
      if (elect_one()) {
        if (!stats) {
          const uint32_t k_lo = stage_mn + st * (C::kStageBytes >> 4), a_addr = tmem + 128u * sb;
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            if (ks < ng)
              mma_ts<smem_desc_hi_sw128(L::kSbo)>(tmem + kTmemDq, a_addr + 32 * (ks >> 1) + 8 * (ks & 1),
                                                  k_lo + ks * (L::kSlotStride >> 4), idesc_dq, ks > 0 || !first);
          if (last) mma_commit(&sh->o_done);
        }
        mma_commit(&sh->kv_empty[st]);
        mma_commit(&sh->dq_done[sb]);
      }
      __syncwarp();
      if (last && !stats) ++n_back;
    }
  } else if (warp < 8) {
    // ------------------------------------------------------------ dS
    const int half = warp >> 2;            // columns: chunks half and half + 2 of every round
    const int r = (warp & 3) * 32 + lane;  // row of the query tile == TMEM lane
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const float c = scale * kLog2e, ref_slack = 8.f / c;
    // rows are shared by warps w and w + 4: maxima are exchanged between these two only
    uint32_t n_pair = 0;
    auto pair_sync = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->pair[warp & 3]);
      return wait(&sh->pair[warp & 3], n_pair++ & 1u);
    };
    float m = -CUDART_INF_F, l = 0.f, dsum = 0.f;
    float fixed = 0.f;  // (fp16) minus log2 of the row's sum
    bool started = false;
    uint32_t n = 0;
    for (uint32_t g = 0;; ++g) {
      const int st = (int)(g % C::kStages);
      const uint32_t sb = g & 1u;
      const uint32_t tmem_s = tmem + 128u * sb + lane_addr;
      if (!wait(&sh->kv_full[st], (g / C::kStages) & 1u)) break;
      const uint32_t info = sh->info[st];
      if (info & kInfoStop) break;
      const int chunks = ((int)(info & kInfoSlots) + 1) >> 1;
      const bool mine = chunks > half;  // the round reaches this thread's columns
      const bool stats = kF16 && (info & kInfoStats);
      const bool first = (info & kInfoFirst) != 0u, last = (info & kInfoLast) != 0u;
      if (first && (!kF16 || stats)) {
        m = -CUDART_INF_F;
        l = 0.f;
        started = false;
      }
      uint32_t w0 = 0xffffffffu, w1 = 0xffffffffu;
      if (!(info & kInfoFull)) {
        w0 = sh->bitmap[st][r][half];
        w1 = sh->bitmap[st][r][half + 2];
      }
      if (!wait(&sh->s_full[sb], (g >> 1) & 1u)) break;
      tc_fence_after_sync();
      uint32_t xs[64];
      float top = -CUDART_INF_F;
      if (mine) {
        // both chunks always: one the round does not reach holds stale values whose bitmap bits are zero
        tmem_ld32(tmem_s + 32 * half, &xs[0]);
        tmem_ld32(tmem_s + 32 * (half + 2), &xs[32]);
        tmem_wait_ld();
        if (!(info & kInfoFull)) {
#pragma unroll
          for (int e = 0; e < 32; ++e) xs[e] = ((w0 >> e) & 1u) ? xs[e] : 0xff800000u;
#pragma unroll
          for (int e = 0; e < 32; ++e) xs[32 + e] = ((w1 >> e) & 1u) ? xs[32 + e] : 0xff800000u;
        }
        if (!kF16 || stats) {
          float t0 = top, t1 = top, t2 = top, t3 = top;
#pragma unroll
          for (int e = 0; e < 64; e += 8) {
            t0 = fmax3(t0, __uint_as_float(xs[e]), __uint_as_float(xs[e + 1]));
            t1 = fmax3(t1, __uint_as_float(xs[e + 2]), __uint_as_float(xs[e + 3]));
            t2 = fmax3(t2, __uint_as_float(xs[e + 4]), __uint_as_float(xs[e + 5]));
            t3 = fmax3(t3, __uint_as_float(xs[e + 6]), __uint_as_float(xs[e + 7]));
          }
          top = fmaxf(fmaxf(t0, t1), fmaxf(t2, t3));
        }
      }
      float neg_ref = fixed;
      if (!kF16 || stats) {
        if (!stats) {  // one reference for the row: its two threads exchange their maxima
          sh->xchg[sb][half][r] = top;
          if (!pair_sync()) break;
          top = fmaxf(top, sh->xchg[sb][half ^ 1][r]);
        }
        const bool move = top > m + ref_slack;  // also true for the first kept entry (m = -inf)
        const float m_new = move ? top : m;
        const float m_safe = m_new == -CUDART_INF_F ? 0.f : m_new;
        const float alpha = move ? ex2_approx((m - m_safe) * c) : 1.f;
        neg_ref = -m_safe * c;
        m = m_new;
        l *= alpha;
        if (!stats && started && __any_sync(0xffffffffu, alpha != 1.f)) {
          // the same decision in both of the row's warps: each rescales half of dQ's columns
          if (!wait(&sh->dq_done[(g - 1u) & 1u], ((g - 1u) >> 1) & 1u)) break;
          tc_fence_after_sync();
#pragma unroll 1
          for (int x = 0; x < D / 64; ++x) {
            uint32_t o[32];
            const uint32_t at = tmem + kTmemDq + lane_addr + (D / 2) * half + 32 * x;
            tmem_ld32(at, o);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 32; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            tmem_st32(at, o);
          }
        }
      }
      if (mine) {
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int e = 0; e < 64; e += 2) {
          const float p0 = ex2_approx(fmaf(__uint_as_float(xs[e]), c, neg_ref));
          const float p1 = ex2_approx(fmaf(__uint_as_float(xs[e + 1]), c, neg_ref));
          if (!kF16 || stats) s0 += p0, s1 += p1;
          xs[e] = __float_as_uint(p0);
          xs[e + 1] = __float_as_uint(p1);
        }
        l += s0 + s1;
      }
      if (first && !stats) {
        if (!wait(&sh->d_ready[n & 1u], (n >> 1) & 1u)) break;
        dsum = sh->dsum[n & 1u][r];
      }
      if (!wait(&sh->dp_full, g & 1u)) break;
      if (mine && !stats) {
        tc_fence_after_sync();
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          uint32_t y[32], pk[16];
          tmem_ld32(tmem + kTmemDp + lane_addr + 32 * (half + 2 * x), y);
          tmem_wait_ld();
          if (x == 1) {  // dP is in registers: the next round's may be computed
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->dp_free);
          }
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            // a pruned entry has p = 0; a column beyond the round's slots is never read by the product
            const float d0 = __uint_as_float(xs[32 * x + 2 * e]) * (__uint_as_float(y[2 * e]) - dsum);
            const float d1 = __uint_as_float(xs[32 * x + 2 * e + 1]) * (__uint_as_float(y[2 * e + 1]) - dsum);
            pk[e] = pack2<kF16>(d0, d1);
          }
          tmem_st16(tmem_s + 32 * (half + 2 * x), pk);
        }
      } else {
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh->dp_free);
      }
      started = true;
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->ds_full[sb]);
      if (!last) continue;
      if (stats) {
        // the row's two partial (maximum, sum) pairs, merged the same way by both threads
        float2 *mine2 = &sh->ml[n & 3u][half][r], *other = &sh->ml[n & 3u][half ^ 1][r];
        *mine2 = make_float2(m, l);
        if (!pair_sync()) break;
        const float2 a = half ? *other : *mine2, b = half ? *mine2 : *other;
        const float top2 = fmaxf(a.x, b.x);
        const float sum = (a.y > 0.f ? a.y * ex2_approx((a.x - top2) * c) : 0.f) +
                          (b.y > 0.f ? b.y * ex2_approx((b.x - top2) * c) : 0.f);
        fixed = sum > 0.f ? -fmaf(top2, c, lg2_approx(sum)) : -CUDART_INF_F;
        if (!pair_sync()) break;  // read before the hand-over below writes the slot
        continue;
      }
      sh->ml[n & 3u][half][r] = kF16 ? make_float2(fixed, 0.f) : make_float2(m, l);
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->ml_ready[n & 3u]);
      ++n;
    }
  } else {
    // ------------------------------------------------------------ D of the next item, dQ of the last one
    const int wr = (warp & 3) * 32;  // this warp's 32 rows of the tile
    const uint32_t lane_addr = (uint32_t)wr << 16;
    unsigned char *out_s = smem + C::kOutOffset + (warp - 10) * 4096;
    const float c = scale * kLog2e;
    // D_i of item n's rows wr .. wr+31; false if there is no such item (or a wait has expired)
    auto form_d = [&](uint32_t n) {
      if (!wait(&sh->item_ready[n % kItemRing], (n / kItemRing) & 1u)) return false;
      const int bh = sh->item_bh[n % kItemRing], qt = sh->item_qt[n % kItemRing];
      if (qt < 0) return false;
      constexpr int kLanes = D / 8, kRows = 32 / kLanes;  // lanes per row (16 bytes each), rows per step
      const int sub = lane / kLanes, piece = lane % kLanes;
      const size_t base = ((size_t)bh * Lq + (size_t)qt * kTile) * D + piece * 8;
      const int rows = Lq - qt * kTile;
#pragma unroll 1
      for (int b = 0; b < 32 / kRows; b += 4) {
        uint4 x[4], y[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int row = wr + (b + u) * kRows + sub;
          x[u] = y[u] = make_uint4(0u, 0u, 0u, 0u);
          if (row < rows) {
            x[u] = *reinterpret_cast<const uint4 *>(dO + base + (size_t)row * D);
            y[u] = *reinterpret_cast<const uint4 *>(O + base + (size_t)row * D);
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t xw[4] = {x[u].x, x[u].y, x[u].z, x[u].w}, yw[4] = {y[u].x, y[u].y, y[u].z, y[u].w};
          float acc = 0.f;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 a = unpack2<kF16>(xw[e]), o = unpack2<kF16>(yw[e]);
            acc = fmaf(a.x, o.x, acc);
            acc = fmaf(a.y, o.y, acc);
          }
#pragma unroll
          for (int o = kLanes / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
          if (piece == 0) sh->dsum[n & 1u][wr + (b + u) * kRows + sub] = acc;
        }
      }
      __syncwarp();
      stat_d[((size_t)bh * n_qt + qt) * kTile + wr + lane] = sh->dsum[n & 1u][wr + lane];
      if (lane == 0) mbar_arrive(&sh->d_ready[n & 1u]);
      return true;
    };
    bool there = form_d(0);
    for (uint32_t n = 0; there; ++n) {
      there = form_d(n + 1);
      if (!wait(&sh->ml_ready[n & 3u], (n >> 2) & 1u)) break;
      const int bh = sh->item_bh[n % kItemRing], qt = sh->item_qt[n % kItemRing];
      const float2 a = sh->ml[n & 3u][0][wr + lane], b = sh->ml[n & 3u][1][wr + lane];
      float f, nl;
      if (kF16) {
        f = scale;
        nl = a.x;
      } else {
        const float sum = a.y + b.y;  // (one reference for both halves)
        f = sum > 0.f ? scale / sum : 0.f;
        nl = sum > 0.f ? -fmaf(a.x, c, lg2_approx(sum)) : -CUDART_INF_F;
      }
      const int i = qt * kTile + wr + lane;
      neg_l[((size_t)bh * n_qt + qt) * kTile + wr + lane] = i < Lq ? nl : -CUDART_INF_F;
      if (!wait(&sh->o_done, n & 1u)) break;
      tc_fence_after_sync();
      uint32_t pk[D / 2];
#pragma unroll
      for (int x = 0; x < D / 32; ++x) {
        uint32_t o[32];
        tmem_ld32(tmem + kTmemDq + lane_addr + 32 * x, o);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float v0 = f != 0.f ? __uint_as_float(o[2 * e]) * f : 0.f;
          const float v1 = f != 0.f ? __uint_as_float(o[2 * e + 1]) * f : 0.f;
          pk[16 * x + e] = pack2<kF16>(v0, v1);
        }
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->o_free);  // the next item may overwrite dQ
      uint16_t *rows_out = dQ + ((size_t)bh * Lq + (size_t)qt * kTile + wr) * D;
      const int n_rows = Lq - qt * kTile - wr;
#pragma unroll
      for (int x = 0; x < D / 64; ++x)
        store_rows64(out_s, lane, &pk[32 * x],
                     [&](int rr) -> uint16_t * { return rr < n_rows ? rows_out + (size_t)rr * D + 64 * x : nullptr; });
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem, kTmemCols);
}

template <int D, bool kSplit, bool kF16>
cudaError_t launch(const RowsMaps &maps, const Args &a) {
  using C = Cfg<D, kSplit>;
  auto kern = rows_kernel<D, kSplit, kF16>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorUnknown;
  const DebugKnobs knobs = debug_knobs();
  const int n_items = a.B * a.H * a.t->n_qt, grid = n_items < sms ? n_items : sms;
  kern<<<grid, kThreads, C::kSmemBytes, a.s>>>(
      maps, static_cast<const uint16_t *>(a.O), static_cast<const uint16_t *>(a.dO), static_cast<uint16_t *>(a.dQ),
      a.plan.neg_l, a.plan.dsum, a.plan.next, a.t->round_ptr, a.t->round_rows, a.t->round_info, a.t->round_bitmap,
      n_items, a.H, a.Lq, a.t->n_qt, a.scale, a.err, knobs.max_polls, knobs.skip_arrive);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rows(const RowsMaps &maps, const Args &a) {
  if (a.d == 64) return a.f16 ? launch<64, false, true>(maps, a) : launch<64, false, false>(maps, a);
  if (a.split) return a.f16 ? launch<128, true, true>(maps, a) : launch<128, true, false>(maps, a);
  return a.f16 ? launch<128, false, true>(maps, a) : launch<128, false, false>(maps, a);
}

}  // namespace bwd
}  // namespace ap
