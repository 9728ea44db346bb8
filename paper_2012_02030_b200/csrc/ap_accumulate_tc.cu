// Eq. 1 as a running sum for bf16 and fp16 tensors, on the tcgen05 tensor cores.
//
// One CTA owns one (head, 128-row query tile) and adds, for up to 16 samples b per launch,
// the normalised softmax rows to the accumulator.  A softmax row needs its
// maximum and its sum of exponentials over ALL keys before any entry can be
// normalised, and the sum over b needs each sample normalised separately, so
// the CTA sweeps its key tiles twice:
//   sweep 1  for every key tile kt, for every b:  S = Q_b K_b(kt)^T  (tcgen05.mma,
//            operands staged by TMA, accumulator in TMEM) -> per-row running
//            maximum and sum of exp2 of the scaled, biased logits
//   sweep 2  the same visits again: p = exp2(logit - max - log2 sum) is the
//            normalised weight; the sum over b is kept in TMEM and added to the
//            accumulator once per key tile (one global update per entry and
//            call instead of one per sample).
// The bias tile of a key tile is staged once per sweep and key tile by TMA (fp32,
// 128-byte swizzle, so that a thread reads its own row without bank conflicts),
// copied to registers and reused for all b.  Samples are added in ascending b by
// a fixed thread and every accumulator entry receives exactly one addition per CTA that
// owns it, so results are reproducible bit for bit.  Shapes with few (head, query tile)
// pairs would leave most SMs idle; for them a launch's samples are cut into chunks, one
// CTA per (chunk, head, query tile), and the chunks' sums are added to the accumulator
// in ascending chunk order: per key tile a counter in global memory says how many warps
// of lower chunks have finished their addition, and a CTA waits (bounded) for its turn
// before it issues its own.  Where the accumulator's rows are
// 16-byte multiples that addition is a TMA reduction: each softmax warp stages its
// 32 rows x 32 columns in shared memory (16 columns at a time, 64-byte swizzle) and one lane issues
// cp.reduce.async.bulk.tensor ... add, which updates whole 128-byte lines in L2;
// a lane per row adding 16 bytes at a time would touch 32 lines per instruction.  Inside
// a tile that straddles the edge of a causal domain the reduction adds exact zeros to the
// entries outside the domain (boxes wholly outside are skipped).  Other shapes keep the
// per-row red.global.add.
//
// Warp roles (576 threads, one CTA per SM; kGroups = 4): warps 0-15 softmax; thread (wg, r) with wg = warp / 4 owns row r of
// the tile and columns [32 wg, 32 wg + 32) of every key tile; warp 16 TMA producer; warp 17 MMA issuer and TMEM owner.  With
// kGroups = 2 eight softmax warps take 64 columns per thread, which leaves room for the statistics of 32 samples.  S is
// double-buffered in TMEM (2 x 128 columns) so the MMA of the next visit runs under the softmax of the current one; a
// visit's 32 columns are copied to registers in one go and S is handed back before the arithmetic starts.  TMEM columns
// 256-383 hold the running sum over b, columns 384-511 the per-sample (maximum, sum) pairs of the four column quarters,
// which a thread reads back for its own row (lane) at the start of sweep 2.  Every mbarrier wait is bounded.
//
// What bounds it: the threads' chain per visit (S -> maximum -> exponentials, 1 024 cycles of them, -> sums: some 1 850
// cycles) and, at d = 128, the 64 KB of operands and the bias that a visit brings.  Sixteen softmax warps instead of eight
// with 64 columns each hide the chain's latency better (77 against 84 us at 16 x 16 heads x 512, causal; the same at 4096).
#include <math_constants.h>

#include <atomic>

#include "ap_common.cuh"
#include "ap_sm100.cuh"

namespace ap {

namespace {

using namespace sm100;

constexpr int kSubBytes = 128 * 128;
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSumCol = 256;    // running sum over b: 128 columns
constexpr uint32_t kStatsCol = 384;  // (max, sum) pairs: as many columns per group of columns as it has, 2 per sample
constexpr int kBiasBytes = 128 * 128 * 4;  // one fp32 bias tile: 4 boxes of 128 rows x 32 columns
constexpr int kRedBytes = 32 * 64;         // per softmax warp: 32 rows x 16 fp32 columns on their way to the accumulator
constexpr float kLog2e = 1.4426950408889634f;

template <int D>
struct Cfg {
  static constexpr int kSub = D / 64;
  static constexpr int kTileBytes = kSub * kSubBytes;    // one operand tile (Q or K)
  static constexpr int kStages = D == 64 ? 4 : 2;        // (Q, K) pairs in flight
  static constexpr int kBiasOffset = 2 * kStages * kTileBytes;
  static constexpr int kRedOffset = kBiasOffset + kBiasBytes;
  static constexpr int kBarOffset = kRedOffset + 16 * kRedBytes;
  static constexpr int kSmemBytes = kBarOffset + 256 + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "within the shared memory of one CTA");
};

// kGroups groups of four softmax warps share a key tile's columns.
template <int kGroups>
struct Roles {
  static constexpr int kSoftmaxWarps = 4 * kGroups, kProducer = kSoftmaxWarps, kIssuer = kSoftmaxWarps + 1;
  static constexpr int kThreads = (kSoftmaxWarps + 2) * 32;
  // registers are handed out to whole sets of four warps (sixteen softmax warps: 20 warps' worth, 96 each)
  static constexpr int kRegThreads = (kSoftmaxWarps + 4) * 32;
  static constexpr int kCols = 128 / kGroups;   // of a thread
  static constexpr int kMaxB = 64 / kGroups;    // samples per CTA (what the spare tensor-memory columns hold)
};

struct Barriers {
  uint64_t s_full[2], s_empty[2];
  uint64_t in_full[4], in_empty[4];
  uint64_t sweep1_done;  // all softmax warps have stored their sweep-1 statistics
  uint64_t stats_read;   // ... and have read them
  uint64_t bias_full, bias_empty;
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Turn counters of the chunked launches: one word per (head, query tile, key tile), zeroed before every
// such launch.  Calls take the sets in rotation: two launches that share one must not overlap on the GPU (see ap.h).
constexpr size_t kTurnWords = 8192;
constexpr int kTurnSets = 8;
constexpr int kMinChunk = 2;  // samples per CTA at least
__device__ unsigned g_turn[kTurnSets][kTurnWords];

unsigned *turn_words() {
  static std::atomic<unsigned> next{0};
  static unsigned *base[16] = {nullptr};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 16) return nullptr;
  if (!base[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_turn) != cudaSuccess) return nullptr;
    base[dev] = static_cast<unsigned *>(p);
  }
  return base[dev] + (size_t)(next.fetch_add(1) % kTurnSets) * kTurnWords;
}

// Key tiles of a query tile (memory: keys before the segment under a causal mask; -1: no mask).
__host__ __device__ inline int key_tiles(int qt, int n_kt, int memory) {
  if (memory < 0) return n_kt;
  const int n = (qt * kTile + kTile - 1 + memory) / kTile + 1;
  return n < n_kt ? n : n_kt;
}
// Chunks that a query tile's B samples are cut into, for about `visits` visits each: at least kMinChunk samples a chunk,
// at most max_b.
__host__ __device__ inline int chunks_of(int visits, int n_k, int B, int max_b) {
  int per = visits / n_k;
  per = per < kMinChunk ? kMinChunk : per > max_b ? max_b : per;
  return (B + per - 1) / per;
}

// dbg_skip != 0 (test hook): the copies of the first visit are never issued, so the MMA issuer's
// first wait runs out and the CTA leaves through its error path.
// kChunked: the instantiation for launches whose samples are cut into chunks (see below); a
// separate one so that its extra code costs the plain launches nothing.
template <int D, bool kChunked, int kGroups>
__global__ void __launch_bounds__(Roles<kGroups>::kRegThreads, 1)
accumulate_tc_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                     const __grid_constant__ CUtensorMap map_bias, const __grid_constant__ CUtensorMap map_acc,
                     int bias_by_tma, int acc_by_tma, float *__restrict__ acc, const float *bias, int b0,
                     int Bc_all, int chunk_visits, unsigned *__restrict__ turn, int H, int Lq, int Lk, int n_qt,
                     int n_kt, int causal, int f16, float scale_log2, unsigned *err, uint32_t max_polls, int dbg_skip) {
  using C = Cfg<D>;
  constexpr int kSoftmaxWarps = Roles<kGroups>::kSoftmaxWarps, kProducer = Roles<kGroups>::kProducer,
                kIssuer = Roles<kGroups>::kIssuer, kCols = Roles<kGroups>::kCols, kMaxB = Roles<kGroups>::kMaxB;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *smem =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *bias_s = smem + C::kBiasOffset;
  Barriers *bars = reinterpret_cast<Barriers *>(smem + C::kBarOffset);

  // Small shapes have fewer (head, query tile) pairs than the GPU has SMs; the launch's samples are
  // then cut into chunks of about chunk_visits (sample, key tile) visits, one CTA per (chunk, head, query tile), and the
  // chunks' sums are added to the accumulator in ascending order of the chunks (turn[], see below), so that
  // the result does not depend on which CTA finishes first.  Lower chunks have lower block indices.
  // late query tiles (most key tiles under a causal mask) first
  int qt = n_qt - 1 - (int)blockIdx.x / H, h = (int)blockIdx.x % H, chunk = 0, Bc = Bc_all;
  if (kChunked) {
    int left = (int)blockIdx.x;
    for (qt = n_qt - 1; qt > 0; --qt) {
      const int here = H * chunks_of(chunk_visits, key_tiles(qt, n_kt, causal ? Lk - Lq : -1), Bc_all, kMaxB);
      if (left < here) break;
      left -= here;
    }
    // the samples of a query tile are dealt out evenly over its chunks
    const int chunks = chunks_of(chunk_visits, key_tiles(qt, n_kt, causal ? Lk - Lq : -1), Bc_all, kMaxB);
    h = left % H;
    chunk = left / H;
    const int first = chunk * Bc_all / chunks;
    Bc = (chunk + 1) * Bc_all / chunks - first;
    b0 += first;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // causal: row i looks at keys j <= i + (Lk - Lq), i.e. Lk - Lq memory keys, then its own segment
  const int off = causal ? Lk - Lq : 0;
  const int n_k = key_tiles(qt, n_kt, causal ? off : -1);
  const int visits_per_sweep = n_k * Bc;
  const int n_visits = 2 * visits_per_sweep;

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars->s_full[s], 1);
      mbar_init(&bars->s_empty[s], kSoftmaxWarps);  // one arrival per softmax warp
    }
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&bars->in_full[s], 1);
      mbar_init(&bars->in_empty[s], 1);
    }
    mbar_init(&bars->sweep1_done, kSoftmaxWarps);
    mbar_init(&bars->stats_read, kSoftmaxWarps);
    mbar_init(&bars->bias_full, 1);
    mbar_init(&bars->bias_empty, kSoftmaxWarps);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (threadIdx.x == 32 * kProducer) {
    prefetch_tensormap(&map_q);
    prefetch_tensormap(&map_k);
    if (bias_by_tma) prefetch_tensormap(&map_bias);
  }
  const uint32_t tmem = begin_with_tmem(&bars->tmem_base, kTmemCols, warp == kIssuer);
  volatile int *abort_flag = &bars->abort_flag;
  const Waiter wait{abort_flag, err, max_polls};

  if (warp == kProducer) {
    // ------------------------------------------------------------ TMA producer
    {
      if (lane == 0) {
      }
      int v = 0, bias_loads = 0;
      for (; v < n_visits; ++v) {
        const int st = v % C::kStages;
        const uint32_t ph = (uint32_t)(v / C::kStages) & 1u;
        const int vv = v % visits_per_sweep;
        const int kt = vv / Bc, b = b0 + vv % Bc;
        if (bias_by_tma && v % Bc == 0) {
          // bias tile of the key tile whose visits start here; the buffer is free once all
          // softmax threads have copied the previous tile to registers
          const int tl = v / Bc;
          if (!wait(&bars->bias_empty, ((uint32_t)tl & 1u) ^ 1u)) break;
          if (lane == 0) {
            mbar_arrive_expect_tx(&bars->bias_full, kBiasBytes);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              tma_load_3d(bias_s + q * (kBiasBytes / 4), &map_bias, &bars->bias_full, kt * kTile + 32 * q, qt * kTile, h);
          }
          __syncwarp();
          bias_loads = tl + 1;
        }
        if (!wait(&bars->in_empty[st], ph ^ 1u)) break;
        if (dbg_skip != 0 && v == 0) continue;
        unsigned char *q_s = smem + (2 * st) * C::kTileBytes, *k_s = q_s + C::kTileBytes;
        if (lane == 0) {
          mbar_arrive_expect_tx(&bars->in_full[st], 2 * C::kTileBytes);
#pragma unroll
          for (int s = 0; s < C::kSub; ++s) {
            tma_load_3d(q_s + s * kSubBytes, &map_q, &bars->in_full[st], 64 * s, qt * kTile, b * H + h);
            tma_load_3d(k_s + s * kSubBytes, &map_k, &bars->in_full[st], 64 * s, kt * kTile, b * H + h);
          }
        }
        __syncwarp();
      }
      if (lane == 0 && *abort_flag) {  // winding down: let the copies in flight land (bounded)
        for (int j = max(0, v - C::kStages); j < v; ++j) {
          if (dbg_skip != 0 && j == 0) continue;
          mbar_wait(&bars->in_full[j % C::kStages], (uint32_t)(j / C::kStages) & 1u, max_polls);
        }
        if (bias_loads > 0) mbar_wait(&bars->bias_full, (uint32_t)(bias_loads - 1) & 1u, max_polls);
      }
    }
  } else if (warp == kIssuer) {
    // ------------------------------------------------------------ MMA issuer
    {
      const uint32_t idesc = idesc_bf16_f32(128, 128, false, false, f16 != 0);
      const uint32_t desc0 = smem_desc_lo(smem_u32(smem), 16);
      for (int v = 0; v < n_visits; ++v) {
        const int st = v % C::kStages;
        const uint32_t ph = (uint32_t)(v / C::kStages) & 1u;
        const int buf = v & 1;
        if (!wait(&bars->in_full[st], ph)) break;
        if (!wait(&bars->s_empty[buf], ((uint32_t)(v >> 1) & 1u) ^ 1u)) break;
        tc_fence_after_sync();
        if (elect_one()) {
          const uint32_t q_lo = desc0 + 2 * st * (C::kTileBytes >> 4), k_lo = q_lo + (C::kTileBytes >> 4);
          constexpr uint32_t kHi = smem_desc_hi_sw128(1024);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t step = (ks / 4) * (kSubBytes >> 4) + (ks % 4) * 2;
            mma_ss<kHi, kHi>(tmem + 128 * buf, q_lo + step, k_lo + step, idesc, ks > 0);
          }
          mma_commit(&bars->in_empty[st]);
          mma_commit(&bars->s_full[buf]);
        }
        __syncwarp();
      }
    }
  } else {
    // ------------------------------------------------------------ softmax (256 or 512 threads)
    const int wg = warp >> 2;
    const int r = (warp & 3) * 32 + lane;  // row of the tile == TMEM lane
    const int i = qt * kTile + r;
    const bool row_ok = i < Lq;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const int jend = causal ? min(Lk, i + 1 + off) : Lk;  // first key outside this row's domain
    const bool vec = (Lk & 3) == 0;
    const uint32_t s_addr = tmem + lane_addr + kCols * wg;          // + 128 * buf
    const uint32_t sum_addr = tmem + lane_addr + kSumCol + kCols * wg;
    const uint32_t stats = tmem + lane_addr + kStatsCol;            // + kCols * group + 2 * b
    const uint32_t my_stats = stats + kCols * wg;
    // this warp's 32 rows x 16 columns on their way to the accumulator, and the rows' place in it
    unsigned char *red_s = smem + C::kRedOffset + warp * kRedBytes;
    const int red_y = qt * kTile + (warp & 3) * 32;
    const int red_jend = causal ? min(Lk, red_y + 32 + off) : Lk;  // first key outside the domain of all 32 rows

    for (int b = 0; b < Bc; ++b) tmem_st2(my_stats + 2 * b, __float_as_uint(-CUDART_INF_F), 0u);

    float bias2[kCols];  // bias * log2(e) of this thread's columns of the current key tile
    bool ok = true;
    // the bias slice of key tile kt (tl: how many tiles were staged before it), once for all samples
    auto fetch_bias = [&](int kt, int tl) {
      const int j0 = kt * kTile + kCols * wg;
      if (bias_by_tma) {
        ok = wait(&bars->bias_full, (uint32_t)tl & 1u);
        if (!ok) return;
#pragma unroll
        for (int k = 0; k < kCols / 4; ++k) {  // 16-byte chunk k of a box's row sits at position k ^ (r % 8)
          const unsigned char *box = bias_s + (wg * (kCols / 32) + k / 8) * (kBiasBytes / 4) + r * 128;
          const float4 t = *reinterpret_cast<const float4 *>(box + (((k & 7) ^ (r & 7)) << 4));
          bias2[4 * k] = t.x * kLog2e; bias2[4 * k + 1] = t.y * kLog2e;
          bias2[4 * k + 2] = t.z * kLog2e; bias2[4 * k + 3] = t.w * kLog2e;
        }
        fence_proxy_async_smem();  // the reads are over before the next tile's copy may write
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->bias_empty);
      } else {
#pragma unroll
        for (int c = 0; c < kCols / 4; ++c) {
          float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
          const int j = j0 + 4 * c;
          if (bias && row_ok) {
            const float *brow = bias + ((size_t)h * Lq + i) * Lk;
            if (j < Lk) t.x = brow[j];
            if (j + 1 < Lk) t.y = brow[j + 1];
            if (j + 2 < Lk) t.z = brow[j + 2];
            if (j + 3 < Lk) t.w = brow[j + 3];
          }
          bias2[4 * c] = t.x * kLog2e; bias2[4 * c + 1] = t.y * kLog2e;
          bias2[4 * c + 2] = t.z * kLog2e; bias2[4 * c + 3] = t.w * kLog2e;
        }
      }
    };
    // S of visit v is ready: copy this thread's columns to registers and hand S back.  The MMA of
    // visit v + 2 may then overwrite the buffer while the arithmetic on the copy is still going on
    // (one arrival per warp: all threads arriving one by one would take longer than a visit's MMAs).
    auto take_s = [&](int v, uint32_t (&xs)[kCols]) {
      const int buf = v & 1;
      ok = wait(&bars->s_full[buf], (uint32_t)(v >> 1) & 1u);
      if (!ok) return;
      tc_fence_after_sync();
#pragma unroll
      for (int c = 0; c < kCols; c += 32) tmem_ld32(s_addr + 128 * buf + c, xs + c);
    };
    auto release_s = [&](int v) {
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->s_empty[v & 1]);
    };

    // ---- sweep 1: per sample and row, the maximum and the sum of exp2 over this thread's columns
    int v = 0;
    for (int kt = 0; kt < n_k && ok; ++kt) {
      fetch_bias(kt, kt);
      if (!ok) break;
      // columns of this slice inside the row's domain; whole warp inside => no masking
      const int n_valid = max(0, min(kCols, jend - (kt * kTile + kCols * wg)));
      const bool interior = __all_sync(0xffffffffu, n_valid == kCols);
      for (int b = 0; b < Bc; ++b, ++v) {
        uint32_t xs[kCols], sv[2];
        take_s(v, xs);
        if (!ok) break;
        tmem_wait_st();  // this sample's pair as the previous key tile left it
        tmem_ld2(my_stats + 2 * b, sv);
        tmem_wait_ld();
        release_s(v);
        float t[kCols];
#pragma unroll
        for (int e = 0; e < kCols; e += 2)
          ffma2(t[e], t[e + 1], __uint_as_float(xs[e]), __uint_as_float(xs[e + 1]), scale_log2, bias2[e], bias2[e + 1]);
        if (!interior) {
#pragma unroll
          for (int e = 0; e < kCols; ++e) t[e] = e < n_valid ? t[e] : -CUDART_INF_F;
        }
        const float m_old = __uint_as_float(sv[0]);
        // four independent chains each for the maximum and for the sum
        float m0 = m_old, m1 = -CUDART_INF_F, m2 = -CUDART_INF_F, m3 = -CUDART_INF_F;
#pragma unroll
        for (int e = 0; e < kCols; e += 8) {  // three-input maxima: half the instructions
          m0 = fmax3(m0, t[e], t[e + 4]);
          m1 = fmax3(m1, t[e + 1], t[e + 5]);
          m2 = fmax3(m2, t[e + 2], t[e + 6]);
          m3 = fmax3(m3, t[e + 3], t[e + 7]);
        }
        const float cm = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
        const float cm_safe = cm == -CUDART_INF_F ? 0.f : cm;
        float z0 = __uint_as_float(sv[1]) * ex2_approx(m_old - cm_safe), z1 = 0.f, z2 = 0.f, z3 = 0.f;
        const float neg_cm = -cm_safe;
#pragma unroll
        for (int e = 0; e < kCols; e += 4) {
          float a0, a1, a2, a3;
          fadd2(a0, a1, t[e], t[e + 1], neg_cm, neg_cm);
          fadd2(a2, a3, t[e + 2], t[e + 3], neg_cm, neg_cm);
          fadd2(z0, z1, z0, z1, ex2_approx(a0), ex2_approx(a1));
          fadd2(z2, z3, z2, z3, ex2_approx(a2), ex2_approx(a3));
        }
        tmem_st2(my_stats + 2 * b, __float_as_uint(cm), __float_as_uint((z0 + z1) + (z2 + z3)));
      }
    }
    if (ok) {
      // every statistic of sweep 1 is final once all groups of columns of every row are done
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->sweep1_done);
      ok = wait(&bars->sweep1_done, 0);
      tc_fence_after_sync();
    }
    if (ok) {
      // The groups' statistics of every sample combined, once for all visits of sweep 2: minus (max + log2(sum)), first to the
      // columns of the running sum, then, when all have read the pairs, over this group's pairs.  A row without any key
      // in its domain (possible when Lk < Lq) gets weight 0 everywhere.
      constexpr int kAhead = 16 / kGroups;  // samples at a time
#pragma unroll 1
      for (int b0 = 0; b0 < Bc; b0 += kAhead) {
        uint32_t st[kAhead][kGroups][2];
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
#pragma unroll
          for (int q = 0; q < kGroups; ++q) tmem_ld2(stats + kCols * q + 2 * (b0 + u), st[u][q]);  // (beyond the last: not used)
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
          float mm = __uint_as_float(st[u][0][0]);
#pragma unroll
          for (int q = 1; q < kGroups; ++q) mm = fmaxf(mm, __uint_as_float(st[u][q][0]));
          float z = 0.f;
#pragma unroll
          for (int q = 0; q < kGroups; ++q) z += __uint_as_float(st[u][q][1]) * ex2_approx(__uint_as_float(st[u][q][0]) - mm);
          tmem_st1(sum_addr + b0 + u, __float_as_uint(jend > 0 ? -(mm + lg2_approx(z)) : -CUDART_INF_F));
        }
      }
      tmem_wait_st();
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->stats_read);
      ok = wait(&bars->stats_read, 0);
      tc_fence_after_sync();
#pragma unroll
      for (int b0 = 0; b0 < kMaxB; b0 += 16) {
        uint32_t ref[16];
        tmem_ld16(sum_addr + b0, ref);
        tmem_wait_ld();
        tmem_st16(my_stats + b0, ref);
      }
      tmem_wait_st();
    }

    // ---- sweep 2: normalised weights, summed over b in TMEM, added to the accumulator per key tile
    for (int kt = 0; kt < n_k && ok; ++kt) {
      fetch_bias(kt, n_k + kt);
      if (!ok) break;
      const int j0 = kt * kTile + kCols * wg;  // first column of this thread's slice
      const int n_valid = max(0, min(kCols, jend - j0));
      const bool interior = __all_sync(0xffffffffu, n_valid == kCols);
      for (int b = 0; b < Bc; ++b, ++v) {
        uint32_t xs[kCols], ref;
        take_s(v, xs);
        if (!ok) break;
        tmem_ld1(my_stats + b, ref);
        tmem_wait_ld();
        release_s(v);
        const float neg_ref = __uint_as_float(ref);
#pragma unroll
        for (int c = 0; c < kCols / 16; ++c) {
          float p[16];
#pragma unroll
          for (int e = 0; e < 16; e += 2)
            ffma2(p[e], p[e + 1], __uint_as_float(xs[16 * c + e]), __uint_as_float(xs[16 * c + e + 1]), scale_log2,
                  bias2[16 * c + e], bias2[16 * c + e + 1]);
          if (!interior) {
#pragma unroll
            for (int e = 0; e < 16; ++e) p[e] = 16 * c + e < n_valid ? p[e] : -CUDART_INF_F;
          }
          uint32_t ps[16];
          if (b > 0) {
            tmem_ld16(sum_addr + 16 * c, ps);
            tmem_wait_ld();
          }
#pragma unroll
          for (int e = 0; e < 16; e += 2) {
            float a0, a1;
            fadd2(a0, a1, p[e], p[e + 1], neg_ref, neg_ref);
            float p0 = ex2_approx(a0), p1 = ex2_approx(a1);
            if (b > 0) fadd2(p0, p1, __uint_as_float(ps[e]), __uint_as_float(ps[e + 1]), p0, p1);
            ps[e] = __float_as_uint(p0);
            ps[e + 1] = __float_as_uint(p1);
          }
          if (b < Bc - 1) {
            tmem_st16(sum_addr + 16 * c, ps);
          } else {
            if (kChunked && c == 0) {
              // this key tile's entries have received the sums of all lower chunks once their
              // warps have counted themselves in (bounded wait)
              if (lane == 0) {
                const unsigned *flag = turn + ((size_t)h * n_qt + qt) * n_kt + kt;
                const unsigned want = (unsigned)chunk * kSoftmaxWarps;
                uint32_t polls = 0;
                while (ld_acquire_gpu(flag) < want && ok) {
                  if (*abort_flag || ++polls > max_polls) {
                    if (!*abort_flag) {
                      *abort_flag = 1;
                      atomicOr(err, kDevErrTimeout);
                    }
                    ok = false;
                  } else if (polls > 64) {
                    __nanosleep(128);
                  }
                }
              }
              ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
              if (!ok) break;
              __syncwarp();
            }
            if (acc_by_tma) {
              // last sample of this key tile: one addition per accumulator entry and launch, performed
              // in L2 by a TMA reduction of this warp's 32 x 16 block
              if (lane == 0) bulk_wait_group_read0();  // the block staged before has been read
              __syncwarp();
#pragma unroll
              for (int k = 0; k < 4; ++k)  // 16-byte chunk k of row `lane` goes to position k ^ (lane / 2 % 4)
                *reinterpret_cast<uint4 *>(red_s + lane * 64 + ((k ^ ((lane >> 1) & 3)) << 4)) =
                    make_uint4(ps[4 * k], ps[4 * k + 1], ps[4 * k + 2], ps[4 * k + 3]);
              fence_proxy_async_smem();
              __syncwarp();
              const int x = j0 + 16 * c;
              if (lane == 0 && red_y < Lq && x < red_jend) {
                tma_reduce_add_3d(&map_acc, red_s, x, red_y, h);
                bulk_commit_group();
              }
            } else if (row_ok) {
              // accumulator rows that are no 16-byte multiples: one red per entry (entries outside the
              // domain are not touched)
              float *arow = acc + ((size_t)h * Lq + i) * Lk + j0 + 16 * c;
              const int nv = n_valid - 16 * c;
#pragma unroll
              for (int g = 0; g < 4; ++g) {
                const int jj = 4 * g;
                if (jj >= nv) break;
                if (vec && jj + 4 <= nv) {
                  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(arow + jj),
                               "f"(__uint_as_float(ps[jj])), "f"(__uint_as_float(ps[jj + 1])),
                               "f"(__uint_as_float(ps[jj + 2])), "f"(__uint_as_float(ps[jj + 3]))
                               : "memory");
                } else {
#pragma unroll
                  for (int e = 0; e < 4; ++e)
                    if (jj + e < nv)
                      asm volatile("red.global.add.f32 [%0], %1;" ::"l"(arow + jj + e), "f"(__uint_as_float(ps[jj + e]))
                                   : "memory");
                }
              }
            }
            if (kChunked && c == kCols / 16 - 1) {
              // all blocks of this warp are in the accumulator: count this warp in for the next chunk
              if (acc_by_tma && lane == 0) bulk_wait_group0();
              __threadfence();
              __syncwarp();
              if (lane == 0) atomicAdd(turn + ((size_t)h * n_qt + qt) * n_kt + kt, 1u);
            }
          }
        }
        // the sums must be in TMEM before the next visit reads them
        if (b < Bc - 1) tmem_wait_st();
      }
    }
    if (lane == 0) bulk_wait_group0();  // shared memory stays valid until the reductions have read it
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == kIssuer) tmem_dealloc(tmem, kTmemCols);
}

// How a call's samples are spread over launches and CTAs.
//
// One CTA takes up to max_b samples of a (head, query tile) pair: 16 with sixteen softmax warps, 32 with eight, which are
// slower per visit (84 instead of 77 us at 16 x 16 heads x 512, causal) but save launches and additions.  Shapes with fewer
// pairs than SMs: several CTAs per pair, each with a chunk of the samples, taking turns at the accumulator, all in one wave
// (one CTA per SM).  Fewer visits per chunk keep more SMs busy, but the chunks' additions wait for one another; of all numbers
// of visits per chunk the one with the lowest estimate is taken.  Query tiles with more key tiles are cut into more chunks:
// with the same number for all, the longest CTA of 16 x 16 heads x 512 (causal) had 64 visits (77 us, now 48: 64 us).
// The estimates, in units of a visit (some 1.0 us with sixteen warps), are fitted to these measurements (us; chunks of as many
// samples): 300 x 2 heads x 128 60 x 5 210, 19 x 16 90; 20 x 2 heads x 333, rows added by entry, one CTA per pair 176, 10 x 2
// 176, 4 x 5 122; 7 x 4 heads x 250 x 231, by entry, one CTA 67, 2 x 4 73.
struct Shape {
  int B, H, n_qt, n_kt, memory, sms;  // memory: as for key_tiles
  bool by_tma;                        // accumulator rows have a tensor map
};
constexpr double kLaunch = 6.0;      // a launch
constexpr double kTurn = 3.3;        // an addition to a key tile that others wait for
constexpr double kTurnByEntry = 18.0, kAddByEntry = 13.0;  // by entry, with and without others waiting

// Estimate for n samples in one launch: chunks of about `visits` visits, or (0) one CTA per pair.
double estimate(const Shape &p, int n, int visits, int max_b) {
  const double visit = max_b == 16 ? 1.0 : 1.12, turn = !p.by_tma ? kTurnByEntry : kTurn;
  if (!visits) {  // whole rounds of CTAs; nobody waits, and the reductions of a tensor map run beside the next tile
    const int rounds = (p.H * p.n_qt + p.sms - 1) / p.sms;
    return kLaunch + rounds * p.n_kt * (2.0 * n * visit + (p.by_tma ? 0.0 : kAddByEntry));
  }
  double worst = 0.0;
  for (int qt = 0; qt < p.n_qt; ++qt) {
    const int n_k = key_tiles(qt, p.n_kt, p.memory), chunks = chunks_of(visits, n_k, n, max_b), per = (n + chunks - 1) / chunks;
    const double t = 2.0 * n_k * per * visit + chunks * turn + (n_k - 1) * (turn > per * visit ? turn - per * visit : 0.0);
    worst = t > worst ? t : worst;
  }
  return kLaunch + worst;
}

struct Launch {
  int samples, visits, grid;  // visits = 0: no chunks
  double time;
};

// The next launch of a call with `left` samples to go.
Launch plan_launch(const Shape &p, int left, int max_b, bool chunks) {
  const int n_units = p.H * p.n_qt;
  Launch best = {left < max_b ? left : max_b, 0, n_units, 0.0};
  best.time = estimate(p, best.samples, 0, max_b);
  if (!chunks) return best;
  const int most = max_b * (p.sms / n_units), n = left < most ? left : most;  // as many as one wave can take
  int total = 0;
  for (int qt = 0; qt < p.n_qt; ++qt) total += p.H * key_tiles(qt, p.n_kt, p.memory) * n;
  for (int visits = (total + p.sms - 1) / p.sms; visits <= max_b * p.n_kt; visits += 1 + visits / 16) {
    int grid = 0;
    for (int qt = 0; qt < p.n_qt; ++qt) grid += p.H * chunks_of(visits, key_tiles(qt, p.n_kt, p.memory), n, max_b);
    if (grid > p.sms || grid <= n_units) continue;
    const double time = estimate(p, n, visits, max_b);
    if (time * best.samples < best.time * n) best = {n, visits, grid, time};  // (per sample)
  }
  return best;
}

// Estimate for a whole call: launches of the first one's size, then what is left.
double plan_call(const Shape &p, int max_b, bool chunks) {
  const Launch first = plan_launch(p, p.B, max_b, chunks);
  const int full = p.B / first.samples, rest = p.B % first.samples;
  return full * first.time + (rest ? plan_launch(p, rest, max_b, chunks).time : 0.0);
}

template <int D, int kGroups>
cudaError_t launch(const CUtensorMap &mq, const CUtensorMap &mk, const CUtensorMap &mb, const CUtensorMap &ma,
                   int bias_by_tma, int acc_by_tma, float *acc, const float *bias, const Shape &p, unsigned *turn, int Lq,
                   int Lk, int causal, int f16, float scale, unsigned *err, cudaStream_t s) {
  using R = Roles<kGroups>;
  auto kern = accumulate_tc_kernel<D, false, kGroups>;
  auto kern_chunked = accumulate_tc_kernel<D, true, kGroups>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(kern_chunked, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<D>::kSmemBytes);
  if (e != cudaSuccess) return e;
  const DebugKnobs knobs = debug_knobs();
  // samples in ascending order; launches on one stream run in order
  for (int b0 = 0; b0 < p.B;) {
    const Launch l = plan_launch(p, p.B - b0, R::kMaxB, turn != nullptr);
    unsigned *t = l.visits ? turn : nullptr;
    if (t && (e = launch_clear(t, (size_t)p.H * p.n_qt * p.n_kt * sizeof(unsigned), s)) != cudaSuccess) return e;
    e = launch_early(t ? kern_chunked : kern, (unsigned)(knobs.skip_arrive ? 1 : l.grid), R::kThreads, Cfg<D>::kSmemBytes, s, mq,
                     mk, mb, ma, bias_by_tma, acc_by_tma, acc, bias, b0, l.samples, l.visits, t, p.H, Lq, Lk, p.n_qt, p.n_kt,
                     causal, f16, scale * kLog2e, err, knobs.max_polls, knobs.skip_arrive);
    if (e != cudaSuccess) return e;
    b0 += l.samples;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_accumulate_tc(float *acc, const void *Q, const void *K, const float *bias, int B, int H, int Lq,
                                 int Lk, int d, int causal, int f16, float scale, cudaStream_t s) {
  unsigned *err = device_error_word();
  if (!err) return cudaErrorUnknown;
  CUtensorMap mq, mk;
  if (!make_tile_map_bf16(&mq, Q, B * H, Lq, d) || !make_tile_map_bf16(&mk, K, B * H, Lk, d)) return cudaErrorUnknown;
  // the bias goes through TMA when its rows are 16-byte multiples; otherwise threads load it directly
  CUtensorMap mb = mq;
  const int bias_by_tma = (bias && (Lk & 3) == 0) ? 1 : 0;
  if (bias_by_tma && !make_tile_map_f32(&mb, bias, H, Lq, Lk)) return cudaErrorUnknown;
  // so does the accumulator's update (boxes of 32 rows x 16 columns, one softmax warp's half)
  CUtensorMap ma = mq;
  const int acc_by_tma = (Lk & 3) == 0 ? 1 : 0;
  if (acc_by_tma && !make_tile_map_f32(&ma, acc, H, Lq, Lk, 32, 16)) return cudaErrorUnknown;
  const Shape p = {B, H, ceil_div(Lq, kTile), ceil_div(Lk, kTile), causal ? Lk - Lq : -1, sm_count(), acc_by_tma != 0};
  if (p.sms <= 0) return cudaErrorUnknown;
  const int n_units = H * p.n_qt;
  unsigned *turn = nullptr;
  if (!debug_knobs().skip_arrive && n_units < p.sms && B >= 2 * kMinChunk && (size_t)n_units * p.n_kt <= kTurnWords)
    turn = turn_words();
  const bool eight = B > Roles<4>::kMaxB &&
                     plan_call(p, Roles<2>::kMaxB, turn != nullptr) < plan_call(p, Roles<4>::kMaxB, turn != nullptr);
  auto go = [&](auto fn) {
    return fn(mq, mk, mb, ma, bias_by_tma, acc_by_tma, acc, bias, p, turn, Lq, Lk, causal, f16, scale, err, s);
  };
  if (d == 64) return eight ? go(launch<64, 2>) : go(launch<64, 4>);
  return eight ? go(launch<128, 2>) : go(launch<128, 4>);
}

}  // namespace ap
