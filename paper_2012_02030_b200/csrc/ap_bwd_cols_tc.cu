// Backward of the masked attention, columns kernel: dK and dV.
//
// Persistent, one CTA per SM; a work item is one (b, h, key block), handed out through a counter.  A key block is
// eight 16-key groups at consecutive positions of the head's key order (see the plan), so it may gather keys from
// several places; it is visited by every query tile that keeps an entry of it.  Everything is computed
// TRANSPOSED, keys as rows, so that both weights are A operands straight from TMEM.  Per visit:
//   S^T = K Q^T,  dP^T = V dO^T   tcgen05.mma (over the span of query groups that keep an entry)
//   P^T = 2^(c S^T - L)           two threads per key row (32-query chunks alternate), 16-bit, over S^T in TMEM
//   dV += P^T dO                  A = P^T from TMEM, dO read MN-major; steps of empty query groups are left out
//   dS^T = P^T (dP^T - D)         over dP^T in TMEM
//   dK += dS^T Q
// Every dK and dV row is written once, query tiles are summed in ascending order: no atomics, bit-reproducible.
//
// Warp roles (448 threads): warps 0-7 compute, 8 producer, 9 issues every MMA, 10-13 write the last item's dK and
// dV while the next one runs.  TMEM (512 columns): S^T, dP^T, dV, dK, the accumulators twice at d = 64.  The two
// phases of a visit alternate on the threads (P, then dS), and the tensor cores work on the other half:
// dV(g), S^T(g+1) under the threads' dS(g); dK(g), dP^T(g+1) under their P(g+1).
//
// What bounds it: four products of 128 x 128 x d per visit (measured 79 cycles per 16-deep step).  The version it
// replaces went through shared memory with P and dS and let every step wait for the one before: 589 us on
// 4 x 16 heads, 4096 tokens, d = 128, 5 % kept, 70 us on 64 x 8 heads, 250 x 231, d = 64.
#include "ap_bwd_tc.cuh"

namespace ap {
namespace bwd {

namespace {

using namespace pipe;

constexpr int kThreads = 448;
constexpr int kComputeWarps = 8;
constexpr int kMaxStages = 4;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemDp = 128, kTmemAcc = 256;
constexpr int kItemRing = 8;

// per-visit word: bits 0..7 the query groups (16 rows each) that keep an entry
constexpr uint32_t kInfoFirst = 1u << 8;
constexpr uint32_t kInfoLast = 1u << 9;
constexpr uint32_t kInfoStop = 1u << 10;

struct Shared {
  alignas(16) uint32_t bits[kMaxStages][kTile][4];  // transposed bitmap: bit q of key row k
  alignas(16) float neg_l[kMaxStages][kTile];
  alignas(16) float dsum[kMaxStages][kTile];
  uint64_t q_full[kMaxStages], q_empty[kMaxStages];    // Q, bits, statistics of a visit
  uint64_t do_full[kMaxStages], do_empty[kMaxStages];
  uint64_t kv_full[2], kv_empty[2];
  uint64_t s_full, p_full, dp_full, ds_full;
  uint64_t acc_done[2], acc_free[2];
  uint32_t info[kMaxStages];
  uint64_t item_ready[kItemRing];
  int32_t item_bh[kItemRing], item_block[kItemRing];  // block = -1: no more items
  uint32_t tmem_base;
  int abort_flag;
};

template <int D>
struct Cfg {
  using L = TileLayout<D, false>;
  static constexpr int kStages = D == 64 ? 4 : 2;
  static constexpr int kKvBufs = D == 64 ? 2 : 1;
  static constexpr uint32_t kAccBufs = D == 64 ? 2 : 1;
  static constexpr int kStageOffset = kKvBufs * 2 * L::kBytes;             // (Q, dO) pairs
  static constexpr int kOutOffset = kStageOffset + kStages * 2 * L::kBytes;  // 4 KB per epilogue warp
  static constexpr int kSharedOffset = kOutOffset + 4 * 4096;
  static constexpr int kSmemBytes = kSharedOffset + (int)sizeof(Shared) + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory");
  static_assert(kSmemBytes > 114 * 1024, "one CTA per SM: all of TMEM is taken");
};

template <int D, bool kF16>
__global__ void __launch_bounds__(kThreads, 1)
cols_kernel(const __grid_constant__ ColsMaps maps, uint16_t *__restrict__ dK, uint16_t *__restrict__ dV,
            const float *__restrict__ neg_l, const float *__restrict__ stat_d, int32_t *__restrict__ next,
            const int32_t *__restrict__ order, const int32_t *__restrict__ n_visits, const uint32_t *__restrict__ visit,
            const uint32_t *__restrict__ bits, int BH, int H, int Lk, int n_qt, int n_kt, float scale, unsigned *err,
            uint32_t max_polls, int dbg_skip) {
  using C = Cfg<D>;
  using L = TileLayout<D, false>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *stage_s = smem + C::kStageOffset;
  Shared *sh = reinterpret_cast<Shared *>(smem + C::kSharedOffset);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int i = 0; i < C::kStages; ++i) {
      mbar_init(&sh->q_full[i], 1);
      mbar_init(&sh->q_empty[i], 1);
      mbar_init(&sh->do_full[i], 1);
      mbar_init(&sh->do_empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh->kv_full[i], 1);
      mbar_init(&sh->kv_empty[i], 1);
      mbar_init(&sh->acc_done[i], 1);
      mbar_init(&sh->acc_free[i], 4);
    }
    mbar_init(&sh->s_full, 1);
    mbar_init(&sh->p_full, kComputeWarps);
    mbar_init(&sh->dp_full, 1);
    mbar_init(&sh->ds_full, kComputeWarps);
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
  // accumulators of item n: dV at acc, dK at acc + D
  auto acc_of = [&](uint32_t n) { return tmem + kTmemAcc + (C::kAccBufs == 2u ? 128u * (n & 1u) : 0u); };

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
    uint32_t g = 0, n = 0;    // visits / items with visits so far
    int kv_armed = -1;
    auto draw = [&]() {
      int x = 0;
      if (lane == 0) x = atomicAdd(next, 1);  // (every CTA begins with the item of its own number)
      return (int)gridDim.x + __shfl_sync(0xffffffffu, x, 0);
    };
    // Items: key blocks from the last to the first (the last hold the keys that most query tiles keep, see
    // the plan), all (b, h) of a block in a row: neighbouring blocks of a head, which share query tiles, run close
    // in time, and the long items come first.
    struct Item {
      int bh, block, count, group;  // group: lanes 0..7, the block's 16-key groups
    };
    auto look_up = [&](int k) {
      Item it{0, -1, 0, 0};
      if (k < BH * n_kt) {
        it.block = n_kt - 1 - k / BH;
        it.bh = k % BH;
        const int hb = (it.bh % H) * n_kt + it.block;
        it.count = (int)ldg_now_u32(n_visits + hb);
        if (lane < 8) it.group = (int)ldg_now_u32(order + (size_t)hb * 8 + lane);
      }
      return it;
    };
    Item cur = look_up((int)blockIdx.x);
    int k_next = ok ? draw() : BH * n_kt;
    while (ok && cur.block >= 0) {
      const Item it = cur;
      cur = look_up(k_next);
      if (cur.block >= 0) k_next = draw();
      const size_t hb = (size_t)(it.bh % H) * n_kt + it.block;
      if (it.count == 0) {  // no query keeps a key of this block
#pragma unroll 1
        for (int q = 0; q < 8; ++q) {
          const int j0 = 16 * __shfl_sync(0xffffffffu, it.group, q), rows = min(16, Lk - j0);
          uint4 *k0 = reinterpret_cast<uint4 *>(dK + ((size_t)it.bh * Lk + j0) * D);
          uint4 *v0 = reinterpret_cast<uint4 *>(dV + ((size_t)it.bh * Lk + j0) * D);
          for (int x = lane; x < rows * (D / 8); x += 32) k0[x] = v0[x] = make_uint4(0u, 0u, 0u, 0u);
        }
        continue;
      }
      if (lane == 0) {
        sh->item_bh[n % kItemRing] = it.bh;
        sh->item_block[n % kItemRing] = it.block;
        mbar_arrive(&sh->item_ready[n % kItemRing]);
      }
      const uint32_t *visits = visit + hb * n_qt;
      uint32_t word = ldg_now_u32(visits);
      for (int v = 0; v < it.count; ++v, ++g) {
        const uint32_t me = word;
        if (v + 1 < it.count) word = ldg_now_u32(visits + v + 1);
        const int qt = (int)(me & 0xffffffu), st = (int)(g % C::kStages);
        const uint32_t ph = ((g / C::kStages) & 1u) ^ 1u;
        unsigned char *q_st = stage_s + st * 2 * L::kBytes, *do_st = q_st + L::kBytes;
        ok = wait(&sh->do_empty[st], ph);  // (freed before Q's slot)
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(&sh->do_full[st], L::kBytes);
#pragma unroll
          for (int s = 0; s < L::kSub; ++s)
            tma_load_3d(do_st + s * kSubBytes, &maps.d_o, &sh->do_full[st], 64 * s, qt * kTile, it.bh);
        }
        ok = wait(&sh->q_empty[st], ph);
        if (!ok) break;
        if (lane == 0) {
          sh->info[st] = (me >> 24) | (v == 0 ? kInfoFirst : 0u) | (v + 1 == it.count ? kInfoLast : 0u);
          mbar_arrive_expect_tx(&sh->q_full[st], L::kBytes + kBitmapWords * 4u + 2u * kTile * 4u);
#pragma unroll
          for (int s = 0; s < L::kSub; ++s)
            tma_load_3d(q_st + s * kSubBytes, &maps.q, &sh->q_full[st], 64 * s, qt * kTile, it.bh);
          bulk_load(&sh->bits[st][0][0], bits + (hb * n_qt + v) * kBitmapWords, kBitmapWords * 4, &sh->q_full[st]);
          const size_t stats = ((size_t)it.bh * n_qt + qt) * kTile;
          bulk_load(sh->neg_l[st], neg_l + stats, kTile * 4, &sh->q_full[st]);
          bulk_load(sh->dsum[st], stat_d + stats, kTile * 4, &sh->q_full[st]);
        }
        __syncwarp();
        if (v == 0) {  // K and V (their buffer is freed last)
          const int b = (int)(n % C::kKvBufs);
          ok = wait(&sh->kv_empty[b], ((n / C::kKvBufs) & 1u) ^ 1u);
          if (!ok) break;
          kv_armed = (int)n;
          const int first = 16 * it.group, run = run_of_slots(lane, 8, first);
          if (lane == 0) mbar_arrive_expect_tx(&sh->kv_full[b], 2 * L::kBytes);
          __syncwarp();
          if (run > 0) {
            unsigned char *k_b = smem + b * 2 * L::kBytes;
            load_run<D, false>(k_b, maps.k, &sh->kv_full[b], lane, first, run, it.bh);
            load_run<D, false>(k_b + L::kBytes, maps.v, &sh->kv_full[b], lane, first, run, it.bh);
          }
          __syncwarp();
        }
      }
      if (ok) ++n;
    }
    if (ok) {
      const int st = (int)(g % C::kStages);
      ok = wait(&sh->q_empty[st], ((g / C::kStages) & 1u) ^ 1u);
      if (ok && lane == 0) {
        sh->info[st] = kInfoStop;
        mbar_arrive(&sh->q_full[st]);
        sh->item_block[n % kItemRing] = -1;
        mbar_arrive(&sh->item_ready[n % kItemRing]);
      }
    }
    if (!ok && dbg_skip == 0 && lane == 0) {
      // winding down: wait (bounded) for the copies armed most recently
      if (kv_armed >= 0) mbar_wait(&sh->kv_full[kv_armed % C::kKvBufs], ((uint32_t)kv_armed / C::kKvBufs) & 1u, 1u << 16);
      for (uint32_t a = g >= (uint32_t)C::kStages ? g - C::kStages + 1u : 0; a <= g; ++a) {
        mbar_wait(&sh->do_full[a % C::kStages], (a / C::kStages) & 1u, 1u << 14);
        mbar_wait(&sh->q_full[a % C::kStages], (a / C::kStages) & 1u, 1u << 14);
      }
    }
  } else if (warp == 9) {
    // ------------------------------------------------------------ issuer of all products
    const uint32_t base = smem_u32(smem), stage_addr = smem_u32(stage_s);
    constexpr uint32_t idesc_acc = idesc_bf16_f32(128, D, false, true, kF16);
    bool ok = true;
    uint32_t n_front = 0, n = 0;  // items started by S^T / by dV
    // span of query groups of a visit: S^T and dP^T are computed over it
    auto first_group = [](uint32_t info) { return (uint32_t)__ffs((int)(info & 0xffu)) - 1u; };
    auto span = [&](uint32_t info) { return 32u - (uint32_t)__clz((int)(info & 0xffu)) - first_group(info); };
    // C[128 keys x queries] = A B^T over the visit's span
    auto issue_abt = [&](uint32_t d_tmem, uint32_t a_addr, uint32_t b_addr, uint32_t info) {
      const uint32_t g0 = first_group(info), idesc = idesc_bf16_f32(128, 16 * (int)span(info), false, false, kF16);
      const uint32_t a_lo = smem_desc_lo(a_addr, 16), b_lo = smem_desc_lo(b_addr + g0 * 2048u, 16), d = d_tmem + 16u * g0;
      constexpr uint32_t kHi = smem_desc_hi_sw128(1024);
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        const uint32_t step = (ks / 4) * (kSubBytes >> 4) + (ks % 4) * 2;
        mma_ss<kHi, kHi>(d, a_lo + step, b_lo + step, idesc, ks > 0);
      }
    };
    // acc[128 keys x D] (+)= A[keys x queries, TMEM] B[queries x D], steps of empty query groups left out
    auto issue_acc = [&](uint32_t acc, uint32_t a_tmem, uint32_t b_addr, uint32_t info) {
      uint32_t started = (info & kInfoFirst) ? 0u : 1u;
      const uint32_t b_lo = smem_desc_lo(b_addr, kSubBytes);
#pragma unroll
      for (int ks = 0; ks < 8; ++ks)
        if ((info >> ks) & 1u) {
          mma_ts<smem_desc_hi_sw128(1024)>(acc, a_tmem + 32 * (ks >> 1) + 8 * (ks & 1), b_lo + ks * 128, idesc_acc, started);
          started = 1u;
        }
    };
    // S^T of visit g; false at the end of the work (or after an expired wait: !ok)
    auto scores = [&](uint32_t g, uint32_t &info) {
      const int st = (int)(g % C::kStages);
      ok = wait(&sh->q_full[st], (g / C::kStages) & 1u);
      if (!ok) return false;
      info = sh->info[st];
      if (info & kInfoStop) return false;
      const int b = (int)(n_front % C::kKvBufs);
      if (info & kInfoFirst) ok = wait(&sh->kv_full[b], (n_front / C::kKvBufs) & 1u);
      if (!ok) return false;
      tc_fence_after_sync();
      if (elect_one()) {
        // (S^T's columns hold P^T of the visit before until its dV product, issued earlier, has read them)
        issue_abt(tmem, base + b * 2 * L::kBytes, stage_addr + st * 2 * L::kBytes, info);
        mma_commit(&sh->s_full);
      }
      __syncwarp();
      return true;
    };
    // dP^T of visit g
    auto grads = [&](uint32_t g, uint32_t info) {
      const int st = (int)(g % C::kStages), b = (int)(n_front % C::kKvBufs);
      ok = wait(&sh->do_full[st], (g / C::kStages) & 1u);
      if (!ok) return;
      tc_fence_after_sync();
      if (elect_one()) {
        issue_abt(tmem + kTmemDp, base + b * 2 * L::kBytes + L::kBytes, stage_addr + st * 2 * L::kBytes + L::kBytes, info);
        mma_commit(&sh->dp_full);
        if (info & kInfoLast) mma_commit(&sh->kv_empty[b]);
      }
      __syncwarp();
      if (info & kInfoLast) ++n_front;
    };
    uint32_t info = 0u, info_next = 0u;
    bool more = scores(0, info);
    if (more) grads(0, info);
    for (uint32_t g = 0; more && ok; ++g) {
      const int st = (int)(g % C::kStages);
      const uint32_t q_addr = stage_addr + st * 2 * L::kBytes, acc = acc_of(n);
      const uint32_t ab = C::kAccBufs == 2u ? (n & 1u) : 0u;
      // an item's first products overwrite accumulators that the epilogue must have read
      if ((info & kInfoFirst) && n >= C::kAccBufs) ok = wait(&sh->acc_free[ab], (n / C::kAccBufs - 1u) & 1u);
      if (ok) ok = wait(&sh->p_full, g & 1u);
      if (!ok) break;
      tc_fence_after_sync();
      if (elect_one()) {
        issue_acc(acc, tmem, q_addr + L::kBytes, info);
        mma_commit(&sh->do_empty[st]);
      }
      __syncwarp();
      more = scores(g + 1, info_next);
      if (!ok) break;
      ok = wait(&sh->ds_full, g & 1u);
      if (!ok) break;
      tc_fence_after_sync();
      if (elect_one()) {
        issue_acc(acc + D, tmem + kTmemDp, q_addr, info);
        mma_commit(&sh->q_empty[st]);
        if (info & kInfoLast) mma_commit(&sh->acc_done[ab]);
      }
      __syncwarp();
      if (info & kInfoLast) ++n;
      if (more) grads(g + 1, info_next);
      info = info_next;
    }
  } else if (warp < 8) {
    // ------------------------------------------------------------ P and dS
    const int half = warp >> 2;            // query chunks half and half + 2
    const int r = (warp & 3) * 32 + lane;  // key row of the block == TMEM lane
    const uint32_t tmem_s = tmem + ((uint32_t)((warp & 3) * 32) << 16), tmem_dp = tmem_s + kTmemDp;
    const float c = scale * kLog2e;
    for (uint32_t g = 0;; ++g) {
      const int st = (int)(g % C::kStages);
      if (!wait(&sh->q_full[st], (g / C::kStages) & 1u)) break;
      const uint32_t info = sh->info[st];
      if (info & kInfoStop) break;
      // chunks with a kept entry; the products read nothing of the others
      const bool use[2] = {((info >> (2 * half)) & 3u) != 0u, ((info >> (2 * half + 4)) & 3u) != 0u};
      float p[64];
      if (!wait(&sh->s_full, g & 1u)) break;
      tc_fence_after_sync();
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (!use[x]) continue;  // (the same for the whole warp)
        const int ch = half + 2 * x;
        const uint32_t w = sh->bits[st][r][ch];
        uint32_t s[32], pk[16];
        tmem_ld32(tmem_s + 32 * ch, s);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          const float4 nl = *reinterpret_cast<const float4 *>(&sh->neg_l[st][32 * ch + e]);
          const float l4[4] = {nl.x, nl.y, nl.z, nl.w};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            // queries of a group outside the visit's span hold stale scores: their bits are zero
            const float v = ex2_approx(fmaf(__uint_as_float(s[e + u]), c, l4[u]));
            p[32 * x + e + u] = ((w >> (e + u)) & 1u) ? v : 0.f;
          }
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) pk[e] = pack2<kF16>(p[32 * x + 2 * e], p[32 * x + 2 * e + 1]);
        tmem_st16(tmem_s + 32 * ch, pk);
      }
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->p_full);
      if (!wait(&sh->dp_full, g & 1u)) break;
      tc_fence_after_sync();
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (!use[x]) continue;
        const int ch = half + 2 * x;
        uint32_t y[32], pk[16];
        tmem_ld32(tmem_dp + 32 * ch, y);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
          const float4 dd = *reinterpret_cast<const float4 *>(&sh->dsum[st][32 * ch + e]);
          const float d4[4] = {dd.x, dd.y, dd.z, dd.w};
          float v[4];  // (a column outside the visit's span is never read by the product)
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            v[u] = p[32 * x + e + u] * (__uint_as_float(y[e + u]) - d4[u]);
          }
          pk[e / 2] = pack2<kF16>(v[0], v[1]);
          pk[e / 2 + 1] = pack2<kF16>(v[2], v[3]);
        }
        tmem_st16(tmem_dp + 32 * ch, pk);
      }
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh->ds_full);
    }
  } else {
    // ------------------------------------------------------------ dK and dV of the last item
    const int wr = (warp & 3) * 32;
    const uint32_t lane_addr = (uint32_t)wr << 16;
    unsigned char *out_s = smem + C::kOutOffset + (warp - 10) * 4096;
    for (uint32_t n = 0;; ++n) {
      const uint32_t ab = C::kAccBufs == 2u ? (n & 1u) : 0u;
      if (!wait(&sh->item_ready[n % kItemRing], (n / kItemRing) & 1u)) break;
      const int bh = sh->item_bh[n % kItemRing], block = sh->item_block[n % kItemRing];
      if (block < 0) break;
      if (!wait(&sh->acc_done[ab], (n / C::kAccBufs) & 1u)) break;
      tc_fence_after_sync();
      const int32_t *groups = order + ((size_t)(bh % H) * n_kt + block) * 8 + (wr >> 4);
      const int j0 = 16 * groups[0], j1 = 16 * groups[1];  // this warp's two groups of keys
      uint32_t pk[D / 2];
#pragma unroll 1
      for (int which = 0; which < 2; ++which) {  // dV, dK
        const float f = which ? scale : 1.f;
#pragma unroll
        for (int x = 0; x < D / 32; ++x) {
          uint32_t o[32];
          tmem_ld32(acc_of(n) + which * D + lane_addr + 32 * x, o);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e)
            pk[16 * x + e] = pack2<kF16>(__uint_as_float(o[2 * e]) * f, __uint_as_float(o[2 * e + 1]) * f);
        }
        if (which == 1) {
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh->acc_free[ab]);
        }
        uint16_t *out = (which ? dK : dV) + (size_t)bh * Lk * D;
#pragma unroll
        for (int x = 0; x < D / 64; ++x)
          store_rows64(out_s, lane, &pk[32 * x], [&](int rr) -> uint16_t * {
            const int j = (rr < 16 ? j0 : j1 - 16) + rr;
            return j < Lk ? out + (size_t)j * D + 64 * x : nullptr;
          });
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem, kTmemCols);
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
  const int n_items = a.B * a.H * a.t->n_kt, grid = n_items < sms ? n_items : sms;
  kern<<<grid, kThreads, C::kSmemBytes, a.s>>>(
      maps, static_cast<uint16_t *>(a.dK), static_cast<uint16_t *>(a.dV), a.plan.neg_l, a.plan.dsum, a.plan.next + 1,
      a.plan.order, a.plan.n_visits, a.plan.visit, a.plan.bits, a.B * a.H, a.H, a.Lk, a.t->n_qt, a.t->n_kt, a.scale,
      a.err, knobs.max_polls, knobs.skip_arrive);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_cols(const ColsMaps &maps, const Args &a) {
  if (a.d == 64) return a.f16 ? launch<64, true>(maps, a) : launch<64, false>(maps, a);
  return a.f16 ? launch<128, true>(maps, a) : launch<128, false>(maps, a);
}

}  // namespace bwd
}  // namespace ap
