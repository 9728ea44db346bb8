// Backward of the masked attention, columns kernel: dK and dV.
//
// Persistent, one CTA per SM; a work item is one (b, h, key block) and a block of the grid, taken over by a running CTA.
// A key block is eight 16-key groups at consecutive positions of the head's KEY ORDER, so it may gather keys from several
// places; it is visited by every query tile that keeps an entry of it.  Everything is computed TRANSPOSED, keys as rows, so
// that both weights are A operands straight from TMEM.  Per visit:
//   S^T = K Q^T,  dP^T = V dO^T   tcgen05.mma
//   P^T = 2^(c S^T - L)           two threads per key row (32-query chunks alternate), 16-bit, over S^T in TMEM
//   dV += P^T dO                  A = P^T from TMEM, dO read MN-major
//   dS^T = P^T (dP^T - D)         over dP^T in TMEM
//   dK += dS^T Q
// Every dK and dV row is written once, query tiles are summed in ascending order: no atomics, bit-reproducible.
//
// The key order.  The rows kernel follows the tile list's rounds, which gather the key columns a query tile keeps;
// this kernel needs the same from the key side.  Masks of the method have a few heavy columns (attention sinks,
// strided positions) that nearly every query keeps, among bands that a few neighbouring query tiles keep; a block of
// 128 consecutive keys with one heavy column in it is visited by nearly every query tile.  So the groups of a
// head that are kept by many more query tiles than their key tile's others (more than twice the lower median of the
// tile's eight groups + 2) come last, all others before them in their natural order.  On 16 heads of 4096 tokens,
// 5 % kept, a head is left with 152 visits of its 310 stored tiles.  Every CTA works the heavy groups out for
// itself, from the (query tile, key tile) table (some 3 us; no room for them in the caller's workspace); tables beyond
// kMaxTable words or kMaxHeavy key tiles, and sequences of a few query tiles, where it cannot pay, keep the natural
// order, in which the visits are the stored tiles.
//
// Warp roles (448 threads): warps 0-7 compute, 8 producer, 9 issues every MMA, 10-13 write the last item's dK and dV
// while the next one runs.  The producer finds an item's visits in the table and copies, per visit, Q, dO, the
// queries' statistics and the visit's words of the bitmap (query-major, as the list holds them: a compute warp
// transposes its 32 x 32 blocks with shuffles while it waits for S^T).  TMEM (512 columns): S^T, dP^T, dV, dK, the
// accumulators twice at d = 64.  The two phases of a visit alternate on the threads (P, then dS), and the tensor
// cores work on the other half: dV(g), S^T(g+1) under the threads' dS(g); dK(g), dP^T(g+1) under their P(g+1).  The
// products run in order, so S^T of visit g+1 being there says that dV(g) is over and dP^T of visit g+1 that dK(g) is.
// The first frees dO's slot of visit g, which takes the Q that comes kRing visits later, the second Q's slot,
// which takes that visit's dO: both copies have a whole visit's time to arrive.
//
// What bounds it: a visit takes some 6 000 cycles at 4 x 16 heads x 4096 x 128 (5 % kept; 66 visits per SM in 190 us in a stream
// of calls, in 218 us alone with cold caches; the time between items counted in).  The threads' two phases
// account for some 2 500 (1 024 of them exponentials), the chain dV(g) -> S^T(g+1) -> P(g+1) that one S^T buffer leaves and
// the time between items of four to five visits for the rest; the products of a visit take the tensor cores 2 048 cycles at
// d = 128.  (Sixteen compute warps, one chunk per thread, were slower: 246 against 209 us.)
#include "ap_bwd_tc.cuh"

namespace ap {
namespace bwd {

namespace {

using namespace pipe;

constexpr int kComputeWarps = 8;
constexpr int kProducer = kComputeWarps, kIssuer = kComputeWarps + 1, kFinish = kComputeWarps + 2;
constexpr int kThreads = (kFinish + 4) * 32;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemDp = 128, kTmemAcc = 256;
constexpr int kItemRing = 8;
constexpr int kMaxHeavy = 2048;    // key tiles of all heads that the key order is worked out for
constexpr int kMaxTable = 1 << 16; // table words read for it by every CTA
constexpr int kMinOrderedTiles = 8;

// per-visit word: bits 0..7 the block's key groups that keep an entry
constexpr uint32_t kInfoFirst = 1u << 8;
constexpr uint32_t kInfoLast = 1u << 9;
constexpr uint32_t kInfoStop = 1u << 10;
constexpr uint32_t kInfoPlain = 1u << 11;  // the block is a key tile: its words are the tile's bitmap
constexpr uint32_t kInfoOddShift = 16;     // bits 16..23: which half of its word a gathered group is

template <int kRing>
struct Shared {
  // (one more than slots: the next copies come before the threads have finished with the last ones)
  alignas(16) uint32_t words[kRing + 1][8 * kTile];  // plain: [query][4]; gathered: [group][query], the word that holds it
  alignas(16) float neg_l[kRing + 1][kTile];
  alignas(16) float dsum[kRing + 1][kTile];
  uint32_t order[kMaxHeavy];              // [h][key tile]: bits 0..7 its heavy groups; above: light groups in the tiles below
  uint64_t b_full[kRing + 1];             // words and statistics of a visit there
  uint64_t q_full[kRing], do_full[kRing];
  uint64_t s_full[kRing], dp_full[kRing];
  uint64_t k_full[2], v_full[2];
  uint64_t p_full, ds_full;
  uint64_t dv_done[2], dv_free[2], dk_done[2], dk_free[2];  // an item's accumulators complete / read out
  uint64_t item_ready[kItemRing];
  TakeOver more;                          // the next item
  int32_t item_bh[kItemRing];             // -1: no more items
  int32_t item_group[kItemRing][8];
  uint32_t info[kRing + 1];
  uint32_t tmem_base;
  int abort_flag;
};

template <int D>
struct Cfg {
  using L = TileLayout<D, false>;
  static constexpr int kRing = D == 64 ? 3 : 2;
  using Sh = Shared<kRing>;
  static constexpr int kKvBufs = D == 64 ? 2 : 1;
  static constexpr uint32_t kAccBufs = D == 64 ? 2 : 1;
  static constexpr int kSlotOffset = kKvBufs * 2 * L::kBytes;             // behind the (K, V) pairs
  static constexpr int kOutOffset = kSlotOffset + kRing * 2 * L::kBytes;  // 2 KB per finishing warp
  static constexpr int kSharedOffset = kOutOffset + 4 * 2048;
  static constexpr int kSmemBytes = kSharedOffset + (int)sizeof(Sh) + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory");
  static_assert(kSmemBytes > 114 * 1024, "one CTA per SM: all of TMEM is taken");
};

// 4 bytes global -> shared memory, asynchronously.
__device__ __forceinline__ void cp_async4(void *smem_dst, const void *gmem_src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(smem_dst)), "l"(gmem_src) : "memory");
}

template <int D, bool kF16>
__global__ void __launch_bounds__(kThreads, 1)
cols_kernel(const __grid_constant__ ColsMaps maps, uint16_t *__restrict__ dK, uint16_t *__restrict__ dV,
            const float *neg_l, const float *stat_d,
            const uint32_t *table, const uint32_t *bitmap, int last_tile, int BH, int H, int Lq, int Lk,
            int n_qt, int n_kt, float scale, unsigned *err, uint32_t max_polls, int dbg_skip) {
  using C = Cfg<D>;
  using L = TileLayout<D, false>;
  constexpr uint32_t kRing = C::kRing, kKvBufs = C::kKvBufs;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // slot of a visit's Q (v = 0) and dO (v = 1): they change places every kRing visits
  auto slot_of = [&](uint32_t g, uint32_t v) {
    return (uint32_t)C::kSlotOffset + ((g % kRing) * 2u + (((g / kRing) & 1u) ^ v)) * (uint32_t)L::kBytes;
  };
  auto *sh = reinterpret_cast<typename C::Sh *>(smem + C::kSharedOffset);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (uint32_t i = 0; i < kRing; ++i) {
      mbar_init(&sh->q_full[i], 1);
      mbar_init(&sh->do_full[i], 1);
      mbar_init(&sh->s_full[i], 1);
      mbar_init(&sh->dp_full[i], 1);
    }
    for (uint32_t i = 0; i < kRing + 1; ++i) mbar_init(&sh->b_full[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh->k_full[i], 1);
      mbar_init(&sh->v_full[i], 1);
      mbar_init(&sh->dv_done[i], 1);
      mbar_init(&sh->dv_free[i], 4);
      mbar_init(&sh->dk_done[i], 1);
      mbar_init(&sh->dk_free[i], 4);
    }
    mbar_init(&sh->p_full, kComputeWarps);
    mbar_init(&sh->ds_full, kComputeWarps);
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
  const bool ordered = n_qt >= kMinOrderedTiles && H * n_kt <= kMaxHeavy && (int64_t)H * n_qt * n_kt <= kMaxTable;
  if (ordered) {
    for (int x = threadIdx.x; x < H * n_kt; x += kThreads) {
      const uint32_t *col = table + (size_t)(x / n_kt) * n_qt * n_kt + x % n_kt;
      uint32_t c[4] = {0u, 0u, 0u, 0u};  // query tiles per group, two 16-bit counts each
#pragma unroll 8
      for (int qt = 0; qt < n_qt; ++qt) {
        const uint32_t gm = col[(size_t)qt * n_kt] >> 24;
#pragma unroll
        for (int p = 0; p < 4; ++p) c[p] += ((gm >> (2 * p)) & 1u) | (((gm >> (2 * p + 1)) & 1u) << 16);
      }
      uint32_t heavy = 0u;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const uint32_t mine = (c[q >> 1] >> (16 * (q & 1))) & 0xffffu;
        int below = 0;  // at least four groups with a count under (mine - 2) / 2 <=> mine > 2 * lower median + 2
#pragma unroll
        for (int p = 0; p < 8; ++p) below += 2u * ((c[p >> 1] >> (16 * (p & 1))) & 0xffffu) + 2u < mine ? 1 : 0;
        heavy |= (below >= 4 ? 1u : 0u) << q;
      }
      sh->order[x] = heavy;
    }
    __syncthreads();
    for (int h = warp; h < H; h += kThreads / 32) {
      uint32_t below = 0u;
      for (int kt0 = 0; kt0 < n_kt; kt0 += 32) {
        uint32_t *mine = sh->order + h * n_kt + kt0 + lane;
        const bool there = kt0 + lane < n_kt;
        const uint32_t heavy = there ? *mine : 0xffu, light = 8u - __popc(heavy);
        uint32_t incl = light;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        if (there) *mine = heavy | (below + incl - light) << 8;
        below += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    __syncthreads();
  }
  const Waiter wait{&sh->abort_flag, err, max_polls};
  // accumulators of item n: dV at acc, dK at acc + D
  auto acc_of = [&](uint32_t n) { return tmem + kTmemAcc + (C::kAccBufs == 2u ? 128u * (n & 1u) : 0u); };

  if (warp == kProducer) {
    // ------------------------------------------------------------ producer
    bool ok = dbg_skip == 0;  // (test hook: nothing is copied, the other roles' waits run out)
    uint32_t g = 0, n = 0;    // visits / items with visits so far
    int k_armed = -1, v_armed = -1;
    uint32_t last1 = 0, last2 = 0;  // last visit of the item before, and of the one before that
    // The next item is asked for when the current one begins (every CTA begins with the item of its own number) and looked up
    // once the first visit's copies are under way: one item ahead, no more, or the last ones would pile up on the CTAs that
    // happen to be first (two ahead: 267 instead of 203 us at 310 items of 31 visits, d = 128).
    uint32_t asked = 0, heard = 0;
    bool blocks_left = true;
    auto ask = [&]() {
      if (!blocks_left) return;
      if (lane == 0) ask_block(&sh->more);
      __syncwarp();
      ++asked;
    };
    // Items: four neighbouring key blocks of a (b, h) in a row (they share query tiles, which are then read from L2
    // once for all four), the sets of four from the last to the first (the last hold the keys that most query
    // tiles keep, so the long items come first), all (b, h) of a set in a row.
    struct Item {
      int bh, block;     // block = -1: no such item
      int group;         // lanes 0..7: the block's 16-key groups
      bool plain;        // the block is a key tile
      uint32_t word[8];  // the table's words of query tile `lane` for the key tiles of the eight groups
    };
    auto load_words = [&](Item &it, int qt) {
      const uint32_t *row = table + ((size_t)(it.bh % H) * n_qt + qt) * n_kt;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q > 0 && it.plain) break;
        const int kt = __shfl_sync(0xffffffffu, it.group, q) >> 3;
        it.word[q] = qt < n_qt ? ldg_now_u32(row + kt) : 0u;
      }
    };
    auto look_up = [&](int k) {
      Item it;
      it.bh = 0, it.block = -1, it.group = 0, it.plain = true;
      if (k >= BH * n_kt) return it;
      const int set = k / (4 * BH), in_set = min(4, n_kt - 4 * set), x = k - set * 4 * BH;  // (the last set may be smaller)
      it.bh = x / in_set;
      it.block = n_kt - 1 - 4 * set - x % in_set;
      it.group = 8 * it.block + (lane & 7);
      if (ordered) {
        // lane q < 8: the group at position 8 block + q of the order, which counts the light groups first
        const uint32_t *order = sh->order + (it.bh % H) * n_kt;
        const int n_light = (int)(order[n_kt - 1] >> 8) + 8 - __popc(order[n_kt - 1] & 0xffu);
        if (n_light < 8 * n_kt) {
          const bool heavy = it.group >= n_light;
          const int pos = heavy ? it.group - n_light : it.group;  // among its kind
          auto below = [&](int kt) { return heavy ? 8 * kt - (int)(order[kt] >> 8) : (int)(order[kt] >> 8); };
          int lo = 0, hi = n_kt - 1;  // the last key tile with no more than pos of the kind below it holds the group ...
          while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (below(mid) <= pos) lo = mid; else hi = mid - 1;
          }
          uint32_t kind = heavy ? order[lo] & 0xffu : ~order[lo] & 0xffu;
          for (int skip = pos - below(lo); skip > 0; --skip) kind &= kind - 1u;  // ... as its (pos - below)-th
          it.group = 8 * lo + __ffs((int)kind) - 1;
          const int first = __shfl_sync(0xffffffffu, it.group, 0);
          it.plain = (first & 7) == 0 && __all_sync(0xffffffffu, lane >= 8 || it.group == first + lane);
        }
      }
      load_words(it, lane);
      return it;
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
      return look_up(k >= 0 ? k : BH * n_kt);
    };
    Item cur = look_up((int)blockIdx.x);
    while (ok && cur.block >= 0) {
      Item it = cur;
      ask();
      // the block's groups, wherever in their key tiles they are (the same for every lane)
      uint32_t odd = 0u, sub[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        sub[q] = (uint32_t)__shfl_sync(0xffffffffu, it.group, q) & 7u;
        odd |= (sub[q] & 1u) << q;
      }
      auto groups_of = [&]() {  // of this lane's query tile: which of the block's groups keep an entry
        if (it.plain) return it.word[0] >> 24;
        uint32_t gm = 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) gm |= ((it.word[q] >> (24 + sub[q])) & 1u) << q;
        return gm;
      };
      int qt0 = 0;
      uint32_t gm_lane = groups_of();
      uint32_t left = __ballot_sync(0xffffffffu, gm_lane != 0u);
      auto more = [&]() {  // moves on to the next 32 query tiles that hold a visit, if the current ones are used up
        while (left == 0u && qt0 + 32 < n_qt) {
          qt0 += 32;
          load_words(it, qt0 + lane);
          gm_lane = groups_of();
          left = __ballot_sync(0xffffffffu, gm_lane != 0u);
        }
        return left != 0u;
      };
      if (!more()) {  // no query keeps a key of this block
#pragma unroll 1
        for (int q = 0; q < 8; ++q) {
          const int j0 = 16 * __shfl_sync(0xffffffffu, it.group, q), rows = min(16, Lk - j0);
          uint4 *k0 = reinterpret_cast<uint4 *>(dK + ((size_t)it.bh * Lk + j0) * D);
          uint4 *v0 = reinterpret_cast<uint4 *>(dV + ((size_t)it.bh * Lk + j0) * D);
          for (int x = lane; x < rows * (D / 8); x += 32) k0[x] = v0[x] = make_uint4(0u, 0u, 0u, 0u);
        }
        cur = hear();
        continue;
      }
      if (lane == 0) sh->item_bh[n % kItemRing] = it.bh;
      if (lane < 8) sh->item_group[n % kItemRing][lane] = it.group;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->item_ready[n % kItemRing]);
      const int first_row = 16 * it.group, run = run_of_slots(lane, 8, first_row);
      bool first = true, last = false;
      while (!last) {
        const int src = __ffs((int)left) - 1, qt = qt0 + src;
        left &= left - 1u;
        const uint32_t gm = __shfl_sync(0xffffffffu, gm_lane, src);
        uint32_t pos[8];  // the groups' tiles in the list
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          // (never beyond the list, whatever a rows kernel that gave up has left in the table)
          pos[q] = min(__shfl_sync(0xffffffffu, it.word[q], src) & 0xffffffu, (uint32_t)last_tile);
          if (it.plain) break;
        }
        last = !more();
        const uint32_t at = g % kRing, bat = g % (kRing + 1u), before = g - kRing + 1u;
        // K and V of a new item: the buffer's last readers were S^T and dP^T of an item's last visit.  (A visit that the
        // waits for Q's and dO's slots have passed needs none; its barrier may be phases ahead by now.)
        const uint32_t kb = n % kKvBufs, kv_last = kKvBufs == 1 ? last1 : last2;
        const bool must = first && n >= kKvBufs && (g < kRing || kv_last + kRing > g + 1u);
        unsigned char *k_b = smem + kb * 2 * L::kBytes;
        // Q (and what the threads need) into dO's slot of visit g - kRing: dV of that visit is over when S^T of the
        // one after it is there
        if (g >= kRing) ok = wait(&sh->s_full[before % kRing], (before / kRing) & 1u);
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(&sh->q_full[at], L::kBytes);
#pragma unroll
          for (int s = 0; s < L::kSub; ++s)
            tma_load_3d(smem + slot_of(g, 0) + s * kSubBytes, &maps.q, &sh->q_full[at], 64 * s, qt * kTile, it.bh);
        }
        __syncwarp();
        {
          const int i0 = qt * kTile;
          const size_t stats = (size_t)it.bh * Lq + i0;
#pragma unroll
          for (int x = 0; x < 4; ++x) {  // (rows beyond the tensor keep nothing: their values are never used)
            const int i = 32 * x + lane;
            if (i0 + i < Lq) {
              cp_async4(&sh->neg_l[bat][i], neg_l + stats + i);
              cp_async4(&sh->dsum[bat][i], stat_d + stats + i);
            }
          }
          if (!it.plain) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if ((gm >> q) & 1u) {
                const uint32_t *tile = bitmap + (size_t)pos[q] * kBitmapWords + (sub[q] >> 1);
#pragma unroll
                for (int x = 0; x < 4; ++x) cp_async4(&sh->words[bat][kTile * q + 32 * x + lane], tile + 4 * (32 * x + lane));
              }
          }
          cp_async_arrive_on(&sh->b_full[bat]);
          __syncwarp();
          if (lane == 0) {
            sh->info[bat] = gm | (first ? kInfoFirst : 0u) | (last ? kInfoLast : 0u) | (it.plain ? kInfoPlain : 0u) |
                            (odd << kInfoOddShift);
            if (it.plain) {
              mbar_arrive_expect_tx(&sh->b_full[bat], kBitmapWords * 4u);
              bulk_load(&sh->words[bat][0], bitmap + (size_t)pos[0] * kBitmapWords, kBitmapWords * 4, &sh->b_full[bat]);
            } else {
              mbar_arrive(&sh->b_full[bat]);
            }
          }
          __syncwarp();
        }
        if (first) {
          if (must) ok = wait(&sh->s_full[kv_last % kRing], (kv_last / kRing) & 1u);
          if (!ok) break;
          k_armed = (int)n;
          if (lane == 0) mbar_arrive_expect_tx(&sh->k_full[kb], L::kBytes);
          __syncwarp();
          if (run > 0) load_run<D, false>(k_b, maps.k, &sh->k_full[kb], lane, first_row, run, it.bh);
          __syncwarp();
        }
        // dO into Q's slot of visit g - kRing: dK of that visit is over when dP^T of the one after it is there
        if (g >= kRing) ok = wait(&sh->dp_full[before % kRing], (before / kRing) & 1u);
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(&sh->do_full[at], L::kBytes);
#pragma unroll
          for (int s = 0; s < L::kSub; ++s)
            tma_load_3d(smem + slot_of(g, 1) + s * kSubBytes, &maps.d_o, &sh->do_full[at], 64 * s, qt * kTile, it.bh);
        }
        __syncwarp();
        if (first) {
          if (must) ok = wait(&sh->dp_full[kv_last % kRing], (kv_last / kRing) & 1u);
          if (!ok) break;
          v_armed = (int)n;
          if (lane == 0) mbar_arrive_expect_tx(&sh->v_full[kb], L::kBytes);
          __syncwarp();
          if (run > 0) load_run<D, false>(k_b + L::kBytes, maps.v, &sh->v_full[kb], lane, first_row, run, it.bh);
          __syncwarp();
        }
        if (first) cur = hear();
        if (!ok) break;
        first = false;
        ++g;
      }
      last2 = last1;
      last1 = g - 1u;
      if (ok) ++n;
    }
    if (ok) {
      const uint32_t bat = g % (kRing + 1u), before = g - kRing + 1u;
      if (g >= kRing) ok = wait(&sh->dp_full[before % kRing], (before / kRing) & 1u);
      if (ok && lane == 0) {
        sh->info[bat] = kInfoStop;
        mbar_arrive(&sh->b_full[bat]);
        mbar_arrive(&sh->q_full[g % kRing]);
        sh->item_bh[n % kItemRing] = -1;
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
      if (k_armed >= 0) mbar_wait(&sh->k_full[k_armed % kKvBufs], ((uint32_t)k_armed / kKvBufs) & 1u, 1u << 16);
      if (v_armed >= 0) mbar_wait(&sh->v_full[v_armed % kKvBufs], ((uint32_t)v_armed / kKvBufs) & 1u, 1u << 16);
      for (uint32_t a = g > kRing ? g - kRing : 0; a <= g; ++a) {
        mbar_wait(&sh->q_full[a % kRing], (a / kRing) & 1u, 1u << 13);
        mbar_wait(&sh->do_full[a % kRing], (a / kRing) & 1u, 1u << 13);
        mbar_wait(&sh->b_full[a % (kRing + 1u)], (a / (kRing + 1u)) & 1u, 1u << 13);
      }
    }
  } else if (warp == kIssuer) {
    // ------------------------------------------------------------ issuer of all products
    const uint32_t base = smem_u32(smem);
    constexpr uint32_t idesc_s = idesc_bf16_f32(128, 128, false, false, kF16);
    constexpr uint32_t idesc_acc = idesc_bf16_f32(128, D, false, true, kF16);
    constexpr uint32_t kHi = smem_desc_hi_sw128(1024);
    // C[128 keys x 128 queries] = A B^T
    auto issue_abt = [&](uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr) {
      const uint32_t a_lo = smem_desc_lo(a_addr, 16), b_lo = smem_desc_lo(b_addr, 16);
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        const uint32_t step = (ks / 4) * (kSubBytes >> 4) + (ks % 4) * 2;
        mma_ss<kHi, kHi>(d_tmem, a_lo + step, b_lo + step, idesc_s, ks > 0);
      }
    };
    // acc[128 keys x D] (+)= A[keys x queries, TMEM] B[queries x D]
    auto issue_acc = [&](uint32_t acc, uint32_t a_tmem, uint32_t b_addr, uint32_t info) {
      const uint32_t b_lo = smem_desc_lo(b_addr, kSubBytes);
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        mma_ts<kHi>(acc, a_tmem + 32 * (ks >> 1) + 8 * (ks & 1), b_lo + ks * 128, idesc_acc,
                    ks > 0 || !(info & kInfoFirst));
    };
    uint32_t n_front = 0, n = 0;  // items finished by dP^T / by dK
    bool ok = true;
    // S^T of visit g; false at the end of the work (or after an expired wait: !ok)
    auto scores = [&](uint32_t g, uint32_t &info) {
      const uint32_t at = g % kRing, kb = n_front % kKvBufs, bat = g % (kRing + 1u);
      ok = wait(&sh->q_full[at], (g / kRing) & 1u);
      if (ok) ok = wait(&sh->b_full[bat], (g / (kRing + 1u)) & 1u);  // (the visit's word)
      if (!ok) return false;
      info = sh->info[bat];
      if (info & kInfoStop) return false;
      if (info & kInfoFirst) ok = wait(&sh->k_full[kb], (n_front / kKvBufs) & 1u);
      if (!ok) return false;
      tc_fence_after_sync();
      if (elect_one()) {
        // (S^T's columns hold P^T of the visit before until its dV product, issued earlier, has read them)
        issue_abt(tmem, base + kb * 2 * L::kBytes, base + slot_of(g, 0));
        mma_commit(&sh->s_full[at]);
      }
      __syncwarp();
      return true;
    };
    // dP^T of visit g
    auto grads = [&](uint32_t g, uint32_t info) {
      const uint32_t at = g % kRing, kb = n_front % kKvBufs;
      ok = wait(&sh->do_full[at], (g / kRing) & 1u);
      if (ok && (info & kInfoFirst)) ok = wait(&sh->v_full[kb], (n_front / kKvBufs) & 1u);
      if (!ok) return;
      tc_fence_after_sync();
      if (elect_one()) {
        issue_abt(tmem + kTmemDp, base + kb * 2 * L::kBytes + L::kBytes, base + slot_of(g, 1));
        mma_commit(&sh->dp_full[at]);
      }
      __syncwarp();
      if (info & kInfoLast) ++n_front;
    };
    uint32_t info = 0u, info_next = 0u;
    bool more = scores(0, info);
    if (more) grads(0, info);
    for (uint32_t g = 0; more && ok; ++g) {
      const uint32_t ab = n % C::kAccBufs;
      // an item's first products overwrite accumulators that the finishing warps must have read
      const bool reuse = (info & kInfoFirst) && n >= C::kAccBufs;
      if (reuse) ok = wait(&sh->dv_free[ab], (n / C::kAccBufs - 1u) & 1u);
      if (ok) ok = wait(&sh->p_full, g & 1u);
      if (!ok) break;
      tc_fence_after_sync();
      if (elect_one()) {
        issue_acc(acc_of(n), tmem, base + slot_of(g, 1), info);
        if (info & kInfoLast) mma_commit(&sh->dv_done[ab]);
      }
      __syncwarp();
      auto finish = [&]() {  // dK
        if (reuse) ok = wait(&sh->dk_free[ab], (n / C::kAccBufs - 1u) & 1u);
        if (ok) ok = wait(&sh->ds_full, g & 1u);
        if (!ok) return;
        tc_fence_after_sync();
        if (elect_one()) {
          issue_acc(acc_of(n) + D, tmem + kTmemDp, base + slot_of(g, 0), info);
          if (info & kInfoLast) mma_commit(&sh->dk_done[ab]);
        }
        __syncwarp();
      };
      // (the last dK of an item does not wait for the next item's keys)
      const bool finish_first = (info & kInfoLast) != 0u;
      if (finish_first) finish();
      if (!ok) break;
      more = scores(g + 1, info_next);
      if (!ok) break;
      if (!finish_first) finish();
      if (!ok) break;
      if (info & kInfoLast) ++n;
      if (more) grads(g + 1, info_next);
      info = info_next;
    }
  } else if (warp < kComputeWarps) {
    // ------------------------------------------------------------ P and dS
    const int chunk0 = warp >> 2;          // queries [32 ch, 32 ch + 32) of every visit, ch = chunk0, chunk0 + 2
    const uint32_t tmem_s = tmem + ((uint32_t)((warp & 3) * 32) << 16), tmem_dp = tmem_s + kTmemDp;
    const float c = scale * kLog2e;
    // Before the transpose lane l holds query 4 (7 - l mod 8) + l / 8 of the chunk, so that a key's word holds the bits of
    // queries 4k .. 4k+3 at the tops of its bytes once it is shifted left by k: a byte permute that replicates sign
    // bits then makes the AND masks of two packed pairs.
    const int my_query = 4 * (7 - (lane & 7)) + (lane >> 3);
    auto masks = [](uint32_t w, int k, uint32_t &lo, uint32_t &hi) {
      const uint32_t t = w << k;
      asm("prmt.b32 %0, %1, 0, 0x9988;" : "=r"(lo) : "r"(t));
      asm("prmt.b32 %0, %1, 0, 0xbbaa;" : "=r"(hi) : "r"(t));
    };
    for (uint32_t g = 0;; ++g) {
      const uint32_t at = g % kRing, ph = (g / kRing) & 1u, st = g % (kRing + 1u);
      if (!wait(&sh->b_full[st], (g / (kRing + 1u)) & 1u)) break;
      const uint32_t info = sh->info[st];
      if (info & kInfoStop) break;
      uint32_t p[2][32], w[2];
      bool use[2];  // false: nothing kept in these 32 keys x 32 queries, the weights are zero
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int query = 32 * (chunk0 + 2 * x) + my_query;
        uint32_t word;
        if (info & kInfoPlain) {
          word = sh->words[st][4 * query + (warp & 3)];
        } else {
          const int qa = 2 * (warp & 3);
          const uint32_t a = sh->words[st][kTile * qa + query] >> (16 * ((info >> (kInfoOddShift + qa)) & 1u));
          const uint32_t b = sh->words[st][kTile * qa + kTile + query] >> (16 * ((info >> (kInfoOddShift + qa + 1)) & 1u));
          word = ((info >> qa) & 1u ? a & 0xffffu : 0u) | ((info >> (qa + 1)) & 1u ? b << 16 : 0u);
        }
        use[x] = __any_sync(0xffffffffu, word != 0u);
        w[x] = transpose32(word, lane);
      }
      if (!wait(&sh->s_full[at], ph)) break;
      tc_fence_after_sync();
#pragma unroll
      for (int x = 0; x < 2; ++x)
        if (use[x]) tmem_ld32(tmem_s + 32 * (chunk0 + 2 * x), p[x]);
      tmem_wait_ld();
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int ch = chunk0 + 2 * x;
        uint32_t pk[16];
        if (!use[x]) {
#pragma unroll
          for (int e = 0; e < 16; ++e) pk[e] = 0u;
          tmem_st16(tmem_s + 32 * ch, pk);
          continue;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float4 nl = *reinterpret_cast<const float4 *>(&sh->neg_l[st][32 * ch + 4 * k]);
          // (a pruned score may exceed L: masked as packed bits)
          float a0, a1, a2, a3;
          ffma2(a0, a1, __uint_as_float(p[x][4 * k]), __uint_as_float(p[x][4 * k + 1]), c, nl.x, nl.y);
          ffma2(a2, a3, __uint_as_float(p[x][4 * k + 2]), __uint_as_float(p[x][4 * k + 3]), c, nl.z, nl.w);
          const float p0 = ex2_approx(a0), p1 = ex2_approx(a1), p2 = ex2_approx(a2), p3 = ex2_approx(a3);
          uint32_t lo, hi;
          masks(w[x], k, lo, hi);
          pk[2 * k] = pack2<kF16>(p0, p1) & lo;
          pk[2 * k + 1] = pack2<kF16>(p2, p3) & hi;
          p[x][4 * k] = __float_as_uint(p0);
          p[x][4 * k + 1] = __float_as_uint(p1);
          p[x][4 * k + 2] = __float_as_uint(p2);
          p[x][4 * k + 3] = __float_as_uint(p3);
        }
        tmem_st16(tmem_s + 32 * ch, pk);
      }
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->p_full);
      if (!wait(&sh->dp_full[at], ph)) break;
      tc_fence_after_sync();
#pragma unroll
      for (int x = 0; x < 4; ++x) {  // (sixteen columns at a time: registers)
        const int ch = chunk0 + 2 * (x >> 1), q0 = 16 * (x & 1);
        uint32_t y[16], pk[8];
        if (!use[x >> 1]) {
#pragma unroll
          for (int e = 0; e < 8; ++e) pk[e] = 0u;
          // (the other eight columns of the chunk's first half are written by its other step)
          tmem_st8(tmem_dp + 32 * ch + q0 / 2, pk);
          continue;
        }
        tmem_ld16(tmem_dp + 32 * ch + q0, y);
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 dd = *reinterpret_cast<const float4 *>(&sh->dsum[st][32 * ch + q0 + 4 * k]);
          const uint32_t *pp = &p[x >> 1][q0 + 4 * k];
          float v0, v1, v2, v3;  // p (dP - D)
          ffma2(v0, v1, dd.x, dd.y, -1.f, __uint_as_float(y[4 * k]), __uint_as_float(y[4 * k + 1]));
          ffma2(v2, v3, dd.z, dd.w, -1.f, __uint_as_float(y[4 * k + 2]), __uint_as_float(y[4 * k + 3]));
          fmul2(v0, v1, __uint_as_float(pp[0]), __uint_as_float(pp[1]), v0, v1);
          fmul2(v2, v3, __uint_as_float(pp[2]), __uint_as_float(pp[3]), v2, v3);
          uint32_t lo, hi;
          masks(w[x >> 1], 4 * (x & 1) + k, lo, hi);
          pk[2 * k] = pack2<kF16>(v0, v1) & lo;
          pk[2 * k + 1] = pack2<kF16>(v2, v3) & hi;
        }
        // over the first half of the chunk's columns, which are in registers by then
        tmem_st8(tmem_dp + 32 * ch + q0 / 2, pk);
      }
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->ds_full);
    }
  } else {
    // ------------------------------------------------------------ dV and dK of the last item
    const int wr = (warp & 3) * 32;
    const uint32_t lane_addr = (uint32_t)wr << 16;
    unsigned char *out_s = smem + C::kOutOffset + (warp - kFinish) * 2048;
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      const uint32_t ab = n % C::kAccBufs;
      if (!wait(&sh->item_ready[n % kItemRing], (n / kItemRing) & 1u)) break;
      const int bh = sh->item_bh[n % kItemRing];
      if (bh < 0) break;
      const int32_t *groups = sh->item_group[n % kItemRing] + (wr >> 4);
      const int j0 = 16 * groups[0], j1 = 16 * groups[1];  // this warp's two groups of keys
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {  // dV (complete one product before dK), dK
        const float f = which ? scale : 1.f;
        uint16_t *out = (which ? dK : dV) + (size_t)bh * Lk * D;
        ok = wait(which ? &sh->dk_done[ab] : &sh->dv_done[ab], (n / C::kAccBufs) & 1u);
        if (!ok) break;
        tc_fence_after_sync();
        // everything into registers first: the next item's products may then overwrite the accumulator
        uint32_t pk[D / 2];
#pragma unroll
        for (int x = 0; x < D / 32; ++x) {
          uint32_t o[32];
          tmem_ld32(acc_of(n) + which * D + lane_addr + 32 * x, o);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e)
            pk[16 * x + e] = pack2<kF16>(__uint_as_float(o[2 * e]) * f, __uint_as_float(o[2 * e + 1]) * f);
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(which ? &sh->dk_free[ab] : &sh->dv_free[ab]);
#pragma unroll
        for (int x = 0; x < D / 32; ++x)
          store_rows(out_s, lane, &pk[16 * x], [&](int rr) -> uint16_t * {
            const int j = (rr < 16 ? j0 : j1 - 16) + rr;
            return j < Lk ? out + (size_t)j * D + 32 * x : nullptr;
          });
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == kIssuer) tmem_dealloc(tmem, kTmemCols);
}

template <int D, bool kF16>
cudaError_t launch(const ColsMaps &maps, const Args &a) {
  using C = Cfg<D>;
  auto kern = cols_kernel<D, kF16>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  const int sms = sm_count();
  if (sms <= 0) return cudaErrorUnknown;
  const DebugKnobs knobs = debug_knobs();
  // (the test hook runs on the first wave only: none of its CTAs takes over another's item)
  const int n_items = a.B * a.H * a.t->n_kt, grid = knobs.skip_arrive && n_items > sms ? sms : n_items;
  return launch_early(kern, (unsigned)grid, kThreads, C::kSmemBytes, a.s, maps, static_cast<uint16_t *>(a.dK),
                      static_cast<uint16_t *>(a.dV), a.plan.neg_l, a.plan.dsum, a.plan.table, a.t->bitmap,
                      a.t->cap > 0 ? a.t->cap - 1 : 0, a.B * a.H, a.H, a.Lq, a.Lk, a.t->n_qt, a.t->n_kt, a.scale, a.err,
                      knobs.max_polls, knobs.skip_arrive);
}

}  // namespace

cudaError_t launch_cols(const ColsMaps &maps, const Args &a) {
  if (a.d == 64) return a.f16 ? launch<64, true>(maps, a) : launch<64, false>(maps, a);
  return a.f16 ? launch<128, true>(maps, a) : launch<128, false>(maps, a);
}

}  // namespace bwd
}  // namespace ap
