// Backward of the masked attention, rows kernel: dQ, the row statistics and the columns kernel's (query tile, key tile) table.
//
// Persistent, one CTA per SM; a work item is one (b, h, query tile) and a block of the grid, taken over by a running
// CTA (late query tiles of a head first, heads in order, so that concurrent CTAs share a few heads' K and V in L2).
// An item follows the query tile's rounds (up to eight non-empty 16-column groups each).  Per round:
//   S  = Q K^T, dP = dO V^T   tcgen05.mma, fp32 accumulators in TMEM
//   dS = 2^(c S - r) (dP - D) by four threads per query row (a 32-column chunk each), written as 16-bit values
//                             over S in TMEM
//   dQ += dS K                tcgen05.mma, A = dS from TMEM, B = the same K rows read MN-major
// ONE sweep: the exponent's reference r is an online softmax's running maximum, the weights' sum l is
// collected beside it, dQ is rescaled where the reference moves (lazily, by 2^8) and divided by l at the
// end.  dS then carries the factor l, which bf16's exponent takes; fp16 cannot, so fp16 tensors sweep their
// rounds twice (kF16): S alone for r = log2 of the row's sum, then the above with that fixed reference.
//
// Warp roles (704 threads): warps 0-15 compute, 16 producer, 17 issues every MMA, 18-21 form D_i = dO_i . O_i of the
// NEXT item straight from global memory and write the last item's dQ, -log2 sum and D, and the item's row of the table (as a
// launch of its own in front the table took 4 of 117 us at 64 x 8 heads, 250 queries, 231 keys, forward and backward).
// Sixteen compute warps, because what a round costs a warp is mostly latency (barriers, tensor-memory loads), which
// four warps per scheduler hide better than two.  TMEM (512 columns): S[2], dP, dQ.  The issuer runs one round ahead:
// S(g+1) and dP(g+1) are under way while the threads work on round g.  Slots: V of a round is free after its dP, K
// only after its dQ, so the K that comes kRing rounds later takes V's slot and that round's V takes K's, which gives
// both copies more than a round's time to arrive.
//
// What bounds it: the threads' chain per round (S -> maximum, exchanged by the row's four warps -> exponentials ->
// dP -> dS; 1 024 cycles of exponentials, 1 536 of products at d = 128).  The version it replaces had one CTA per query
// tile, two sweeps and every step waiting for the one before: 402 us at 4 x 16 heads x 4096 x 128 (5 % kept), 143 here; 110 and
// 42 us at 64 x 8 heads, 250 queries, 231 keys (50 % kept).
#include <math_constants.h>

#include "ap_bwd_tc.cuh"

namespace ap {
namespace bwd {

namespace {

using namespace pipe;

constexpr int kComputeWarps = 16;
constexpr int kProducer = kComputeWarps, kIssuer = kComputeWarps + 1, kFinish = kComputeWarps + 2;
constexpr int kThreads = (kFinish + 4) * 32;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemDp = 256, kTmemDq = 384;
constexpr int kItemRing = 8;

constexpr uint32_t kInfoSlots = 15u;
constexpr uint32_t kInfoFirst = 1u << 4;  // first round of its sweep
constexpr uint32_t kInfoLast = 1u << 5;   // last round of its sweep
constexpr uint32_t kInfoFull = 1u << 6;   // every entry kept: no bitmap was copied
constexpr uint32_t kInfoStop = 1u << 7;
constexpr uint32_t kInfoStats = 1u << 8;  // (fp16) first sweep: S only

template <int kRing, int kQBufs>
struct Shared {
  // (one more than slots: K comes before the threads have read the last bitmap)
  alignas(16) uint32_t bitmap[kRing + 1][kTile][4];
  float2 ml[4][kTile];          // [item % 4][row]: (reference, sum)
  float top[2][4][kTile];       // [round % 2][chunk][row]: maximum
  float sum[4][kTile];          // [chunk][row]: sum at the item's end
  float dsum[2][kTile];         // D of item n at [n % 2]
  uint64_t q_full[kQBufs], do_full[kQBufs];
  uint64_t k_full[kRing], v_full[kRing];                   // per round % kRing: rows there
  uint64_t s_full[kRing], dp_full[kRing], dq_done[kRing];  // ... S / dP / dQ of the round over
  uint64_t b_full[kRing + 1];   // word and bitmap of a round there
  uint64_t ds_full[2];
  uint64_t dp_free;
  uint64_t o_free;              // dQ of the item read out
  uint64_t ml_ready[4], d_ready[2], item_ready[kItemRing];
  uint64_t quad[4];             // the four warps that share 32 rows
  TakeOver more;                // the next item
  int32_t item_bh[kItemRing], item_qt[kItemRing];  // qt = -1: no more items
  uint32_t item_last[4];        // [item % 4]: its last round
  uint32_t info[kRing + 1];
  uint32_t tmem_base;
  int abort_flag;
};

template <int D, bool kSplit>
struct Cfg {
  using L = TileLayout<D, kSplit>;
  static constexpr int kRing = D == 64 ? 3 : 2, kQBufs = D == 64 ? 2 : 1;
  using Sh = Shared<kRing, kQBufs>;
  static constexpr int kSlotOffset = kQBufs * 2 * L::kBytes;              // behind the (Q, dO) pairs
  static constexpr int kSharedOffset = kSlotOffset + kRing * 2 * L::kBytes;
  static constexpr int kSmemBytes = kSharedOffset + (int)sizeof(Sh) + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory");
  static_assert(kSmemBytes > 114 * 1024, "one CTA per SM: all of TMEM is taken");
};

// What a list row holds, for the table of the columns kernel.
struct ListRows {
  const int32_t *row_ptr, *col_idx;
  const uint8_t *flags, *groups;
  uint32_t *table;  // see Plan
  int n_kt;
};
// By one warp: list row lr of the table.
__device__ __forceinline__ void write_table(const ListRows &l, int lr, int lane) {
  uint32_t *row = l.table + (size_t)lr * l.n_kt;
  for (int kt = lane; kt < l.n_kt; kt += 32) row[kt] = 0u;
  __syncwarp();
  const int t1 = l.row_ptr[lr + 1];
  for (int t = l.row_ptr[lr] + lane; t < t1; t += 32)
    row[l.col_idx[t]] = (uint32_t)t | (((l.flags[t] & 1u) ? 0xffu : (uint32_t)l.groups[t]) << 24);
}

template <int D, bool kSplit, bool kF16>
__global__ void __launch_bounds__(kThreads, 1)
rows_kernel(const __grid_constant__ RowsMaps maps, const uint16_t *O, const uint16_t *dO,
            uint16_t *__restrict__ dQ, float *__restrict__ neg_l, float *__restrict__ stat_d,
            const int32_t *round_ptr, const int32_t *round_rows,
            const uint8_t *round_info, const uint32_t *round_bitmap, const ListRows list, int n_items,
            int H, int Lq, int n_qt, float scale, unsigned *err, uint32_t max_polls, int dbg_skip) {
  using C = Cfg<D, kSplit>;
  using L = TileLayout<D, kSplit>;
  constexpr uint32_t kRing = C::kRing, kQBufs = C::kQBufs;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // slot of a round's K (v = 0) and V (v = 1): they change places every kRing rounds
  auto slot_of = [&](uint32_t g, uint32_t v) {
    return (uint32_t)C::kSlotOffset + ((g % kRing) * 2u + (((g / kRing) & 1u) ^ v)) * (uint32_t)L::kBytes;
  };
  auto *sh = reinterpret_cast<typename C::Sh *>(smem + C::kSharedOffset);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (uint32_t i = 0; i < kQBufs; ++i) {
      mbar_init(&sh->q_full[i], 1);
      mbar_init(&sh->do_full[i], 1);
    }
    for (uint32_t i = 0; i < kRing; ++i) {
      mbar_init(&sh->k_full[i], 1);
      mbar_init(&sh->v_full[i], 1);
      mbar_init(&sh->s_full[i], 1);
      mbar_init(&sh->dp_full[i], 1);
      mbar_init(&sh->dq_done[i], 1);
    }
    for (uint32_t i = 0; i < kRing + 1; ++i) mbar_init(&sh->b_full[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh->ds_full[i], kComputeWarps);
      mbar_init(&sh->d_ready[i], 4);
    }
    mbar_init(&sh->dp_free, kComputeWarps);
    mbar_init(&sh->o_free, 4);
    for (int i = 0; i < 4; ++i) {
      mbar_init(&sh->ml_ready[i], 4);  // the warps of chunk 0
      mbar_init(&sh->quad[i], 4);
    }
    for (int i = 0; i < kItemRing; ++i) mbar_init(&sh->item_ready[i], 1);
    mbar_init(&sh->more.answered, 1);
    sh->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kProducer) {
    if (lane < 4) {
      prefetch_tensormap(&maps.k[lane]);
      prefetch_tensormap(&maps.v[lane]);
    } else if (lane == 4) {
      prefetch_tensormap(&maps.q);
      prefetch_tensormap(&maps.d_o);
    }
  }
  const uint32_t tmem = begin_with_tmem(&sh->tmem_base, kTmemCols, warp == kIssuer);
  const Waiter wait{&sh->abort_flag, err, max_polls};

  if (warp == kProducer) {
    // ------------------------------------------------------------ producer
    bool ok = dbg_skip == 0;  // (test hook: nothing is copied, the other roles' waits run out)
    uint32_t g = 0, n = 0;    // rounds / non-empty items so far
    // The next item is asked for when the current one begins (every CTA begins with the item of its own number) and looked up
    // once its second round's copies are under way: one item ahead, no more, or the last ones would pile up on the CTAs
    // that happen to be first.
    uint32_t asked = 0, heard = 0;
    bool blocks_left = true;
    auto ask = [&]() {
      if (!blocks_left) return;
      if (lane == 0) ask_block(&sh->more);
      __syncwarp();
      ++asked;
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
    // V of a round is copied one round after its K: its slot is freed later.
    bool v_pending = false, v_used = false;
    int v_row = 0, v_run = 0, v_bh = 0, v_slots = 0;
    auto load_v = [&](uint32_t at_round) {
      const uint32_t at = at_round % kRing;
      if (at_round >= kRing) ok = wait(&sh->dq_done[at], ((at_round / kRing) - 1u) & 1u);
      if (!ok) return;
      if (lane == 0) {
        if (v_used)
          mbar_arrive_expect_tx(&sh->v_full[at], (uint32_t)v_slots * 16u * D * 2u);
        else
          mbar_arrive(&sh->v_full[at]);  // (a round of the first sweep has no dP)
      }
      __syncwarp();
      if (v_used && v_run > 0)
        load_run<D, kSplit>(smem + slot_of(at_round, 1), maps.v, &sh->v_full[at], lane, v_row, v_run, v_bh);
      __syncwarp();
      v_pending = false;
    };
    int q_armed = -1, do_armed = -1;
    uint32_t last1 = 0, last2 = 0;  // last round of the item before, and of the one before that
    uint32_t published = 0;         // non-empty items announced to the finishing warps
    auto publish = [&](const Item &it) {
      if (lane == 0) {
        sh->item_bh[published % kItemRing] = it.bh;
        sh->item_qt[published % kItemRing] = it.qt;
        mbar_arrive(&sh->item_ready[published % kItemRing]);
      }
      __syncwarp();
      ++published;
    };
    auto hear = [&]() {  // (none where nothing was asked for)
      int k = -1;
      if (asked != heard) {
        ok = wait(&sh->more.answered, heard & 1u);
        if (ok) {
          ++heard;
          k = taken_block(&sh->more);
          __syncwarp();
          blocks_left = k >= 0;
        }
      }
      return look_up(k >= 0 ? k : n_items);
    };
    Item cur = look_up((int)blockIdx.x);
    while (ok && cur.qt >= 0) {
      const Item it = cur;
      ask();
      bool known = false;  // the next item
      if (it.r0 == it.r1) {  // nothing kept: dQ is zero, and no key block visits the tile
        const int rows = min(kTile, Lq - it.qt * kTile);
        uint4 *dst = reinterpret_cast<uint4 *>(dQ + ((size_t)it.bh * Lq + (size_t)it.qt * kTile) * D);
        for (int x = lane; x < rows * (D / 8); x += 32) dst[x] = make_uint4(0u, 0u, 0u, 0u);
        if (it.bh < H) write_table(list, it.bh * n_qt + it.qt, lane);
        cur = hear();
        continue;
      }
      if (published == n) publish(it);
      for (int sweep = kF16 ? 0 : 1; sweep < 2 && ok; ++sweep) {
        int row = lane < 8 ? (int)ldg_now_u32(round_rows + (size_t)it.r0 * 8 + lane) : -1;
        uint32_t rinfo = ldg_now_u8(round_info + it.r0);
        for (int v = it.r0; v < it.r1 && ok; ++v) {
          const int my_row = row;
          const uint32_t my_info = rinfo;
          if (v + 1 < it.r1) {
            row = lane < 8 ? (int)ldg_now_u32(round_rows + (size_t)(v + 1) * 8 + lane) : -1;
            rinfo = ldg_now_u8(round_info + v + 1);
          }
          const int ng = (int)(my_info & 15u);
          const bool full = (my_info & 0x80u) != 0u;
          const int run = run_of_slots(lane, ng, my_row);
          const uint32_t at = g % kRing, bat = g % (kRing + 1u);
          if (g >= kRing) ok = wait(&sh->dp_full[at], ((g / kRing) - 1u) & 1u);
          if (!ok) break;
          if (lane == 0) {
            sh->info[bat] = (uint32_t)ng | (v == it.r0 ? kInfoFirst : 0u) | (v + 1 == it.r1 ? kInfoLast : 0u) |
                            (full ? kInfoFull : 0u) | (sweep == 0 ? kInfoStats : 0u);
            mbar_arrive_expect_tx(&sh->k_full[at], (uint32_t)ng * 16u * D * 2u);
            if (full) {
              mbar_arrive(&sh->b_full[bat]);
            } else {
              mbar_arrive_expect_tx(&sh->b_full[bat], kBitmapWords * 4);
              bulk_load(&sh->bitmap[bat][0][0], round_bitmap + (size_t)v * kBitmapWords, kBitmapWords * 4,
                        &sh->b_full[bat]);
            }
          }
          __syncwarp();
          if (run > 0) load_run<D, kSplit>(smem + slot_of(g, 0), maps.k, &sh->k_full[at], lane, my_row, run, it.bh);
          __syncwarp();
          const bool opens = v == it.r0 && (!kF16 || sweep == 0);
          // Q and dO of a new item: the buffer's last readers were S and dP of an item's last round.  (A round that
          // the K copies' own waits have passed needs none; its barrier may be phases ahead by now.)
          const uint32_t qb = n % kQBufs, q_last = kQBufs == 1 ? last1 : last2;
          const bool must = opens && n >= kQBufs && q_last + kRing >= g;
          unsigned char *q_b = smem + qb * 2 * L::kBytes;
          if (opens) {
            if (must) ok = wait(&sh->s_full[q_last % kRing], (q_last / kRing) & 1u);
            if (!ok) break;
            q_armed = (int)n;
            if (lane == 0) {
              mbar_arrive_expect_tx(&sh->q_full[qb], L::kBytes);
#pragma unroll
              for (int s = 0; s < L::kSub; ++s)
                tma_load_3d(q_b + s * kSubBytes, &maps.q, &sh->q_full[qb], 64 * s, it.qt * kTile, it.bh);
            }
            __syncwarp();
          }
          if (v_pending) load_v(g - 1u);
          if (ok && opens) {
            if (must) ok = wait(&sh->dp_full[q_last % kRing], (q_last / kRing) & 1u);
            if (!ok) break;
            do_armed = (int)n;
            if (lane == 0) {
              mbar_arrive_expect_tx(&sh->do_full[qb], L::kBytes);
#pragma unroll
              for (int s = 0; s < L::kSub; ++s)
                tma_load_3d(q_b + L::kBytes + s * kSubBytes, &maps.d_o, &sh->do_full[qb], 64 * s, it.qt * kTile, it.bh);
            }
            __syncwarp();
          }
          // the item after this one, as soon as it is known (the finishing warps form its D ahead)
          if (ok && !known && (v > it.r0 || it.r0 + 1 == it.r1)) cur = hear(), known = true;
          if (known && published == n + 1u && cur.qt >= 0 && cur.r0 < cur.r1) publish(cur);
          ++g;
          v_pending = true, v_used = sweep == 1;
          v_row = my_row, v_run = run, v_bh = it.bh, v_slots = ng;
        }
      }
      ++n;
      last2 = last1;
      last1 = g - 1u;
    }
    if (ok && v_pending) load_v(g - 1u);
    if (ok) {
      const uint32_t at = g % kRing, bat = g % (kRing + 1u);
      if (g >= kRing) ok = wait(&sh->dp_full[at], ((g / kRing) - 1u) & 1u);
      if (ok && lane == 0) {
        sh->info[bat] = kInfoStop;
        mbar_arrive(&sh->b_full[bat]);
        mbar_arrive(&sh->k_full[at]);
        sh->item_qt[n % kItemRing] = -1;
        mbar_arrive(&sh->item_ready[n % kItemRing]);
      }
    }
    if (!ok && dbg_skip == 0 && lane == 0) {
      // winding down: the items left are taken and dropped (their waits would run out one after the other), then a bounded
      // wait for the copies armed most recently
      while (asked != heard && mbar_wait(&sh->more.answered, heard & 1u, 1u << 16)) {
        ++heard;
        if (taken_block(&sh->more) < 0) break;
        ask_block(&sh->more);
        ++asked;
      }
      if (q_armed >= 0) mbar_wait(&sh->q_full[q_armed % kQBufs], ((uint32_t)q_armed / kQBufs) & 1u, 1u << 16);
      if (do_armed >= 0) mbar_wait(&sh->do_full[do_armed % kQBufs], ((uint32_t)do_armed / kQBufs) & 1u, 1u << 16);
      for (uint32_t a = g > kRing ? g - kRing : 0; a <= g; ++a) {
        mbar_wait(&sh->k_full[a % kRing], (a / kRing) & 1u, 1u << 13);
        mbar_wait(&sh->v_full[a % kRing], (a / kRing) & 1u, 1u << 13);
        mbar_wait(&sh->b_full[a % (kRing + 1u)], (a / (kRing + 1u)) & 1u, 1u << 13);
      }
    }
  } else if (warp == kIssuer) {
    // ------------------------------------------------------------ issuer of all products
    const uint32_t base = smem_u32(smem);
    constexpr uint32_t idesc_dq = idesc_bf16_f32(128, D, false, true, kF16);
    uint32_t n_front = 0, n_back = 0;  // items finished by dP / by dQ
    uint32_t info_front = 0u, sweep_round = 0u;
    bool ok = true;
    // C[128 x 16 ng] = A B^T
    auto issue_abt = [&](uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, int ng) {
      const uint32_t idesc = idesc_bf16_f32(128, 16 * ng, false, false, kF16);
      const uint32_t a_lo = smem_desc_lo(a_addr, 16), b_lo = smem_desc_lo(b_addr, 16);
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks)
        mma_ss<smem_desc_hi_sw128(1024), smem_desc_hi_sw128(L::kSbo)>(
            d_tmem, a_lo + (ks / 4) * (kSubBytes >> 4) + (ks % 4) * 2, b_lo + (ks / 4) * (L::kSlabStride >> 4) + (ks % 4) * 2,
            idesc, ks > 0);
    };
    // S and dP of round g; false at the end of the work or after an expired wait (ok tells which)
    auto front = [&](uint32_t g) {
      const uint32_t at = g % kRing, ph = (g / kRing) & 1u, qb = n_front % kQBufs, q_ph = (n_front / kQBufs) & 1u;
      ok = wait(&sh->k_full[at], ph);
      if (!ok) return false;
      info_front = sh->info[g % (kRing + 1u)];
      if (info_front & kInfoStop) return false;
      const bool stats = kF16 && (info_front & kInfoStats);
      const bool opens = (info_front & kInfoFirst) && (!kF16 || stats);
      if (opens) ok = wait(&sh->q_full[qb], q_ph);
      if (!ok) return false;
      tc_fence_after_sync();
      const int ng = (int)(info_front & kInfoSlots);
      if (elect_one()) {
        // (this S buffer held dS of round g - 2, whose dQ product was issued before)
        issue_abt(tmem + 128u * (g & 1u), base + qb * 2 * L::kBytes, base + slot_of(g, 0), ng);
        mma_commit(&sh->s_full[at]);
      }
      __syncwarp();
      if (opens) ok = wait(&sh->do_full[qb], q_ph);
      if (ok) ok = wait(&sh->v_full[at], ph);
      // dP of the previous round is in the threads' registers
      if (ok && g >= 1) ok = wait(&sh->dp_free, (g - 1u) & 1u);
      if (!ok) return false;
      tc_fence_after_sync();
      if (elect_one()) {
        if (!stats) issue_abt(tmem + kTmemDp, base + qb * 2 * L::kBytes + L::kBytes, base + slot_of(g, 1), ng);
        mma_commit(&sh->dp_full[at]);
      }
      __syncwarp();
      if ((info_front & kInfoLast) && !stats) ++n_front;
      return true;
    };
    // dQ of round g
    auto back = [&](uint32_t g, uint32_t info) {
      const bool stats = kF16 && (info & kInfoStats), first = (info & kInfoFirst) != 0u;
      // The first round of an item overwrites dQ: the previous item's must have been read.  A first sweep (fp16) writes no
      // dQ, but its kRing-th round completes the barrier on which the finishing warps wait for the previous item's last dQ a
      // second time: unless they have been there, that phase is lost to them.
      sweep_round = first ? 0u : sweep_round + 1u;
      if (sweep_round == (stats ? kRing - 1u : 0u) && n_back > 0) ok = wait(&sh->o_free, (n_back - 1u) & 1u);
      if (ok) ok = wait(&sh->ds_full[g & 1u], (g >> 1) & 1u);
      if (!ok) return;
      tc_fence_after_sync();
      const int ng = (int)(info & kInfoSlots);
      if (elect_one()) {
        if (!stats) {
          const uint32_t a_addr = tmem + 128u * (g & 1u), b_lo = smem_desc_lo(base + slot_of(g, 0), L::kSlabStride);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)
            if (ks < ng)
              mma_ts<smem_desc_hi_sw128(L::kSbo)>(tmem + kTmemDq, a_addr + 32 * (ks >> 1) + 8 * (ks & 1),
                                                  b_lo + ks * (L::kSlotStride >> 4), idesc_dq, ks > 0 || !first);
        }
        mma_commit(&sh->dq_done[g % kRing]);
      }
      __syncwarp();
      if ((info & kInfoLast) && !stats) ++n_back;
    };
    bool more = front(0);
    for (uint32_t g = 0; more && ok; ++g) {
      const uint32_t info = info_front;
      // an item's Q and dO are copied when the last S and dP of the item before are over: where they are not there yet,
      // the last dQ goes first
      bool back_first = false;
      if ((info & kInfoLast) && !(kF16 && (info & kInfoStats)))
        back_first = !__all_sync(0xffffffffu, mbar_test_wait(&sh->do_full[n_front % kQBufs], (n_front / kQBufs) & 1u));
      if (back_first) back(g, info);
      if (!ok) break;
      more = front(g + 1);
      if (!ok) break;
      if (!back_first) back(g, info);
    }
  } else if (warp < kComputeWarps) {
    // ------------------------------------------------------------ dS
    const int chunk = warp >> 2;           // columns [32 chunk, 32 chunk + 32) of every round
    const int r = (warp & 3) * 32 + lane;  // row of the query tile == TMEM lane
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16, col = lane_addr + 32u * chunk;
    const float c = scale * kLog2e, ref_slack = 8.f / c;
    // rows are shared by the four warps w mod 4: they exchange maxima and sums among themselves
    uint32_t n_quad = 0;
    auto quad_sync = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->quad[warp & 3]);
      return wait(&sh->quad[warp & 3], n_quad++ & 1u);
    };
    float m = -CUDART_INF_F, l = 0.f, dsum = 0.f;
    float fixed = 0.f;  // (fp16) minus log2 of the row's sum
    bool started = false;
    uint32_t n = 0;
    for (uint32_t g = 0;; ++g) {
      const uint32_t at = g % kRing, ph = (g / kRing) & 1u, bat = g % (kRing + 1u), sb = g & 1u;
      const uint32_t tmem_s = tmem + 128u * sb + col;
      if (!wait(&sh->b_full[bat], (g / (kRing + 1u)) & 1u)) break;
      const uint32_t info = sh->info[bat];
      if (info & kInfoStop) break;
      const bool mine = (int)(info & kInfoSlots) > 2 * chunk;  // the round reaches this warp's columns
      const bool stats = kF16 && (info & kInfoStats);
      const bool first = (info & kInfoFirst) != 0u, last = (info & kInfoLast) != 0u;
      if (first && (!kF16 || stats)) {
        m = -CUDART_INF_F;
        l = 0.f;
        started = false;
      }
      const uint32_t w = (info & kInfoFull) ? 0xffffffffu : sh->bitmap[bat][r][chunk];
      if (!wait(&sh->s_full[at], ph)) break;
      tc_fence_after_sync();
      uint32_t xs[32];
      float top = -CUDART_INF_F;
      if (mine) {
        // (the second slot of a chunk may lie beyond the round: stale values, whose bitmap bits are zero)
        tmem_ld32(tmem_s, xs);
        tmem_wait_ld();
        if (!(info & kInfoFull)) {
#pragma unroll
          for (int e = 0; e < 32; ++e) xs[e] = ((w >> e) & 1u) ? xs[e] : 0xff800000u;
        }
        if (!kF16 || stats) {
          float t0 = top, t1 = top;
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            t0 = fmax3(t0, __uint_as_float(xs[e]), __uint_as_float(xs[e + 1]));
            t1 = fmax3(t1, __uint_as_float(xs[e + 2]), __uint_as_float(xs[e + 3]));
          }
          top = fmaxf(t0, t1);
        }
      }
      float neg_ref = fixed;
      if (!kF16 || stats) {
        if (!stats) {  // one reference for the row: its four threads exchange their maxima
          sh->top[sb][chunk][r] = top;
          if (!quad_sync()) break;
          top = fmaxf(fmaxf(sh->top[sb][0][r], sh->top[sb][1][r]), fmaxf(sh->top[sb][2][r], sh->top[sb][3][r]));
        }
        const bool move = top > m + ref_slack;  // also true for the first kept entry (m = -inf)
        const float m_new = move ? top : m;
        const float m_safe = m_new == -CUDART_INF_F ? 0.f : m_new;
        const float alpha = move ? ex2_approx((m - m_safe) * c) : 1.f;
        neg_ref = -m_safe * c;
        m = m_new;
        l *= alpha;
        if (!stats && started && __any_sync(0xffffffffu, alpha != 1.f)) {
          // the same decision in all of the row's warps: each rescales a quarter of dQ's columns
          if (!wait(&sh->dq_done[(g - 1u) % kRing], ((g - 1u) / kRing) & 1u)) break;
          tc_fence_after_sync();
#pragma unroll 1
          for (int x = 0; x < D / 64; ++x) {
            uint32_t o[16];
            const uint32_t o_at = tmem + kTmemDq + lane_addr + (D / 4) * chunk + 16 * x;
            tmem_ld16(o_at, o);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
            tmem_st16(o_at, o);
          }
        }
      }
      if (mine) {
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          float a0, a1;
          ffma2(a0, a1, __uint_as_float(xs[e]), __uint_as_float(xs[e + 1]), c, neg_ref, neg_ref);
          const float p0 = ex2_approx(a0), p1 = ex2_approx(a1);
          if (!kF16 || stats) fadd2(s0, s1, s0, s1, p0, p1);
          xs[e] = __float_as_uint(p0);
          xs[e + 1] = __float_as_uint(p1);
        }
        l += s0 + s1;
      }
      if (first && !stats) {
        if (!wait(&sh->d_ready[n & 1u], (n >> 1) & 1u)) break;
        dsum = sh->dsum[n & 1u][r];
      }
      if (!wait(&sh->dp_full[at], ph)) break;
      if (mine && !stats) {
        tc_fence_after_sync();
#pragma unroll
        for (int x = 0; x < 2; ++x) {  // (sixteen columns at a time: registers)
          uint32_t y[16], pk[8];
          tmem_ld16(tmem + kTmemDp + col + 16 * x, y);
          tmem_wait_ld();
          if (x == 1) {  // dP is in registers: the next round's may be computed
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->dp_free);
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            // a pruned entry has p = 0; a column beyond the round's slots is never read by the product
            float d0, d1;
            fadd2(d0, d1, __uint_as_float(y[2 * e]), __uint_as_float(y[2 * e + 1]), -dsum, -dsum);
            fmul2(d0, d1, __uint_as_float(xs[16 * x + 2 * e]), __uint_as_float(xs[16 * x + 2 * e + 1]), d0, d1);
            pk[e] = pack2<kF16>(d0, d1);
          }
          tmem_st8(tmem_s + 8 * x, pk);
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
        // the row's four partial (maximum, sum) pairs, merged the same way by its four threads
        sh->top[0][chunk][r] = m;
        sh->sum[chunk][r] = l;
        if (!quad_sync()) break;
        float top_all = sh->top[0][0][r], sum = 0.f;
#pragma unroll
        for (int q = 1; q < 4; ++q) top_all = fmaxf(top_all, sh->top[0][q][r]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float lq = sh->sum[q][r];
          if (lq > 0.f) sum += lq * ex2_approx((sh->top[0][q][r] - top_all) * c);
        }
        fixed = sum > 0.f ? -fmaf(top_all, c, lg2_approx(sum)) : -CUDART_INF_F;
        if (!quad_sync()) break;  // (read before the next item's sums are written)
        continue;
      }
      // the item's rounds are over: its (reference, sum) goes to the finishing warps
      if (!kF16) {
        sh->sum[chunk][r] = l;
        if (!quad_sync()) break;  // (the next sums are written behind the next item's first exchange)
      }
      if (chunk == 0) {
        sh->ml[n & 3u][r] = kF16 ? make_float2(fixed, 0.f)
                                 : make_float2(m, (sh->sum[0][r] + sh->sum[1][r]) + (sh->sum[2][r] + sh->sum[3][r]));
        if (threadIdx.x == 0) sh->item_last[n & 3u] = g;
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh->ml_ready[n & 3u]);
      }
      ++n;
    }
  } else {
    // ------------------------------------------------------------ D of the next item, dQ of the last one
    const int wr = (warp & 3) * 32;  // this warp's 32 rows of the tile
    const uint32_t lane_addr = (uint32_t)wr << 16;
    const bool wide = (reinterpret_cast<uintptr_t>(dQ) & 31) == 0;
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
      if (wr + lane < rows) stat_d[(size_t)bh * Lq + qt * kTile + wr + lane] = sh->dsum[n & 1u][wr + lane];
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->d_ready[n & 1u]);
      if (wr == 0 && bh < H) write_table(list, bh * n_qt + qt, lane);  // (every list row is an item of the first batch element)
      return true;
    };
    bool there = form_d(0);
    for (uint32_t n = 0; there; ++n) {
      there = form_d(n + 1);
      if (!wait(&sh->ml_ready[n & 3u], (n >> 2) & 1u)) break;
      const int bh = sh->item_bh[n % kItemRing], qt = sh->item_qt[n % kItemRing];
      const float2 a = sh->ml[n & 3u][wr + lane];
      const uint32_t g_last = sh->item_last[n & 3u];
      const float f = kF16 ? scale : a.y > 0.f ? scale / a.y : 0.f;
      const float nl = kF16 ? a.x : a.y > 0.f ? -fmaf(a.x, c, lg2_approx(a.y)) : -CUDART_INF_F;
      const int n_rows = Lq - qt * kTile - wr;  // of this warp, as far as the tensor reaches
      if (lane < n_rows) neg_l[(size_t)bh * Lq + qt * kTile + wr + lane] = nl;
      if (!wait(&sh->dq_done[g_last % kRing], (g_last / kRing) & 1u)) break;
      tc_fence_after_sync();
      uint16_t *rows_out = dQ + ((size_t)bh * Lq + (size_t)qt * kTile + wr) * D;
#pragma unroll 1
      for (int x = 0; x < D / 64; ++x) {
        uint32_t pk[32];
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          uint32_t o[16];
          tmem_ld16(tmem + kTmemDq + lane_addr + 64 * x + 16 * y, o);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float v0 = f != 0.f ? __uint_as_float(o[2 * e]) * f : 0.f;
            const float v1 = f != 0.f ? __uint_as_float(o[2 * e + 1]) * f : 0.f;
            pk[8 * y + e] = pack2<kF16>(v0, v1);
          }
        }
        if (x == D / 64 - 1) {
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh->o_free);  // the next item may overwrite dQ
        }
        if (lane < n_rows) {
          // 32-byte pieces of the lane's row, whole sectors (gathering rows of the warp through shared memory into
          // 128-byte ones took 355 instead of 346 us at 4 x 16 heads x 4096 x 128, 5 % kept, both passes)
          uint16_t *out = rows_out + (size_t)lane * D + 64 * x;
#pragma unroll
          for (int q = 0; q < 4; ++q) store_sector(out + 16 * q, pk + 8 * q, wide);
        }
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == kIssuer) tmem_dealloc(tmem, kTmemCols);
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
  // (the test hook runs on the first wave only: none of its CTAs takes over another's item)
  const int n_items = a.B * a.H * a.t->n_qt, grid = knobs.skip_arrive && n_items > sms ? sms : n_items;
  const ListRows list = {a.t->row_ptr, a.t->col_idx, a.t->flags, a.t->groups, a.plan.table, a.t->n_kt};
  return launch_early(kern, (unsigned)grid, kThreads, C::kSmemBytes, a.s, maps, static_cast<const uint16_t *>(a.O),
                      static_cast<const uint16_t *>(a.dO), static_cast<uint16_t *>(a.dQ), a.plan.neg_l, a.plan.dsum,
                      a.t->round_ptr, a.t->round_rows, a.t->round_info, a.t->round_bitmap, list, n_items, a.H, a.Lq, a.t->n_qt,
                      a.scale, a.err, knobs.max_polls, knobs.skip_arrive);
}

}  // namespace

cudaError_t launch_rows(const RowsMaps &maps, const Args &a) {
  if (a.d == 64) return a.f16 ? launch<64, false, true>(maps, a) : launch<64, false, false>(maps, a);
  if (a.split) return a.f16 ? launch<128, true, true>(maps, a) : launch<128, true, false>(maps, a);
  return a.f16 ? launch<128, false, true>(maps, a) : launch<128, false, false>(maps, a);
}

}  // namespace bwd
}  // namespace ap
