// Eq. 2 as an exact per-head top-k selection.
//
// Order of the entries of one head: forced (diagonal) first, then larger fp32
// value, then lower linear index i*Lk + j.  The k-th entry of that order is
// found with a most-significant-digit-first radix select over the pair (order-preserving
// 32-bit key of the value, complement of the index): digits of 11, 11 and 10 bits each.  The
// first three give the threshold; the last three, the index of the last kept entry equal to it,
// run only where some of those entries are kept and others are not.
//
// Inputs that fit into the shared memory of the SMs are read once and held there (held_kernel: select, mask and bitmaps in one).
// Larger ones of up to kDirectEntries in all, a few times less than L2 holds, select straight over the
// accumulator, one pass over it per digit.  Still larger ones take a shortcut that reads it once: a
// random sample of the selection brackets the threshold between two pivot keys, one
// pass counts the keys above the upper pivot and collects those between the
// pivots, and the select runs over the collected entries; it is exact whenever the bracket holds
// the threshold and the collected entries fit their buffer (checked with the exact counts), else
// the selection takes the passes over the accumulator.  All of the select is ONE cooperative kernel
// (select_kernel): the CTAs of a selection meet at a bounded barrier after each digit.  As a chain of
// kernels (a histogram per digit, a pick, a tie count, a scan, each launched whether or not it had
// work) the mask of one layer of 16 heads x 512 tokens took 18 launches and 132 us.
//
// The emit pass writes the element mask and per-tile bitmaps; ap_tiles.cu compacts them.  Integer work
// throughout: no floating-point arithmetic decides a bit.
//
// One threshold for the whole layer (Eq. 2 as stated) is the same selection run
// once over a virtual head of H*Lq rows: row i' = h*Lq + i has the domain of row
// i, and the linear index i'*Lk + j is the layer-wide tie order.
#include <cooperative_groups.h>

#include "ap_common.cuh"
#include "ap_grid.cuh"

namespace ap {

namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256;  // collect_kernel
constexpr int kWarps = kThreads / 32;
constexpr int kBins = 2048;
constexpr int kPasses = 3;     // digits of a key (and of an index)

__host__ __device__ constexpr int digit_shift(int pass) { return pass == 0 ? 21 : (pass == 1 ? 10 : 0); }
__host__ __device__ constexpr uint32_t digit_mask(int pass) { return pass == 2 ? 0x3ffu : 0x7ffu; }
// the bits above a digit
__host__ __device__ constexpr uint32_t above_digit(int pass) { return pass == 0 ? 0u : pass == 1 ? 0xffe00000u : 0xfffffc00u; }

// Larger float <=> larger key; -0 is mapped onto +0 first.
__device__ __forceinline__ uint32_t key_of(float f) {
  uint32_t b = __float_as_uint(f);
  if (b == 0x80000000u) b = 0u;
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// The float whose key is `key`.  Keys 0 and 0xffffffff (no pivot / no threshold) give NaNs, for
// which every ordered comparison is false.  For values and pivots that are not NaN,
// key_of(f) > key <=> f > float_of_key(key), and likewise for == and <.
__device__ __forceinline__ float float_of_key(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
}

struct alignas(64) SelectState {  // per selection; all zero before the first kernel of a call
  uint32_t thr;                  // threshold key; 0xffffffff: nothing but the forced entries is kept
  uint32_t tie_cut;              // entries equal to the threshold are kept up to this linear index
  // the shortcut's bracket and what the collecting pass found
  uint32_t lo, hi;               // pivot keys, lo <= hi; hi == 0xffffffff: no upper pivot
  unsigned long long above_hi;   // keys > hi
  uint32_t n_cand;               // keys in [lo, hi] (may exceed the buffer: then the shortcut fails)
  uint32_t use_shortcut;
  // the classifying pass and the select have written this selection's mask and tile bitmaps: the
  // emit pass has nothing left to do for it
  uint32_t emitted;
  uint32_t barrier;              // arrivals of the selection's CTAs so far
};

constexpr int kHistBuffers = 3;      // a digit's counts; zeroed again two digits later
constexpr int kMaxSharedSelections = 128;  // selections with more than one CTA (see select_kernel), at most

struct Scratch {
  SelectState *state;   // [H]
  uint32_t *hist;       // [min(H, kMaxSharedSelections)][kHistBuffers][kBins]
  uint2 *cand;          // [H][cand_cap] (key, linear index) of the entries collected by the shortcut
};

// The shortcut is tried for selections of at least this many entries, when all of them together have more
// than kDirectEntries: passes over an accumulator that L2 holds cost less than drawing the pivots and
// collecting (4 heads x 1024, causal, 2.1 M entries: 56 us without the shortcut, 82 with it).
constexpr long long kShortcutMinEntries = 1ll << 20;
constexpr long long kDirectEntries = 12ll << 20;
constexpr int kSamples = 16384;  // draws per selection; those of forced entries are dropped (with memory keys, those outside
                                 // the domain too)
constexpr int kSampleCtas = 8;   // CTAs (one cluster) that make them
__host__ __device__ inline long long cand_capacity(long long n_rest) {
  return n_rest >= kShortcutMinEntries ? n_rest / 16 : 0;
}

// 16 consecutive floats, from a 32-byte boundary (kVec = 8: two loads of a whole sector per lane) or a 16-byte one.
template <int kVec>
__device__ __forceinline__ void ldg_f16(const float *p, float v[16]) {
  static_assert(kVec == 8 || kVec == 4, "floats per load");
#pragma unroll
  for (int e = 0; e < 16; e += kVec) {
    if (kVec == 8) {
      asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=f"(v[e]), "=f"(v[e + 1]), "=f"(v[e + 2]), "=f"(v[e + 3]), "=f"(v[e + 4]), "=f"(v[e + 5]),
                     "=f"(v[e + 6]), "=f"(v[e + 7])
                   : "l"(p + e));
    } else {
      asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(v[e]), "=f"(v[e + 1]), "=f"(v[e + 2]), "=f"(v[e + 3])
                   : "l"(p + e));
    }
  }
}

__host__ __device__ inline size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// Loads 4 consecutive entries of a row starting at column j0 (j0 % 4 == 0).
// Entries at or beyond `jend` come back as 0 and are flagged invalid by the caller.
__device__ __forceinline__ void load4(const float *__restrict__ row, int j0, int jend, bool vec, float v[4]) {
  if (vec && j0 + 4 <= jend) {
    float4 t = *reinterpret_cast<const float4 *>(row + j0);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = (j0 + c < jend) ? row[j0 + c] : 0.f;
  }
}

// Here and below `rows` counts the rows of a selection and row i has the domain of row i % period
// of a head (period == rows unless heads are stacked).  Under the causal constraint row r of a head
// sees the keys j <= r + (Lk - period): Lk - period memory keys, then its own segment; its own
// position r + (Lk - period) is the forced entry when the diagonal is kept.

// ---- the one-pass shortcut ------------------------------------------------------------------

// A bijection of 32-bit words all of whose output bits depend on all input bits (the finaliser of MurmurHash3).
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x = (x ^ (x >> 16)) * 0x85ebca6bu;
  x = (x ^ (x >> 13)) * 0xc2b2ae35u;
  return x ^ (x >> 16);
}

// CTA-wide (1024 threads): the leading 22 bits of the key of rank `rank` (1 = largest) among keys[0..n) that are not 0,
// at least `rank` of them.  hist: kBins words of shared memory; xch: 2 words.
__device__ uint32_t block_select22(const uint32_t *keys, uint32_t n, uint32_t rank, uint32_t *hist, uint32_t *xch) {
  __shared__ uint32_t warp_sums[32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t prefix = 0u;
  for (int pass = 0; pass < 2; ++pass) {
    const int shift = digit_shift(pass);
    hist[t] = 0u;
    hist[t + 1024] = 0u;
    __syncthreads();
    for (uint32_t idx0 = t; idx0 < n; idx0 += 8 * 1024) {  // eight loads in flight per thread
      uint32_t kk[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) kk[u] = idx0 + u * 1024 < n ? keys[idx0 + u * 1024] : 0u;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (kk[u] != 0u && (kk[u] & above_digit(pass)) == prefix)
          atomicAdd(&hist[(kk[u] >> shift) & digit_mask(pass)], 1u);
    }
    __syncthreads();
    // thread t owns bins 2047 - 2t and 2046 - 2t (descending order of keys)
    const uint32_t c0 = hist[kBins - 1 - 2 * t], c1 = hist[kBins - 2 - 2 * t];
    const uint32_t mine = c0 + c1;
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    uint32_t before = incl - mine;
    for (int w = 0; w < warp; ++w) before += warp_sums[w];
    if (before < rank && before + mine >= rank) {  // exactly one thread
      const bool first = before + c0 >= rank;
      xch[0] = (uint32_t)(kBins - 1 - 2 * t - (first ? 0 : 1));
      xch[1] = rank - before - (first ? 0u : c0);
    }
    __syncthreads();
    prefix |= xch[0] << shift;
    rank = xch[1];
    __syncthreads();
  }
  return prefix;
}

// A cluster of CTAs per selection samples its entries and sets the bracket [lo, hi] around the expected threshold (rounded
// outwards to 22 bits: a third digit would not narrow it noticeably).  The draws of all CTAs go to the shared memory of the
// first two, which pick the upper and the lower pivot.
//
// What bounds it: the draws, each a sector of its own from somewhere in the selection, of which an SM has only so many under
// way, and then the histograms (most keys fall into a few bins).  A pair of CTAs that made all draws, in no order: 28 us for 16
// heads x 2048, 14 of them the draws; 16 x 4096 as a whole 265 us, 259 with a cluster.  32768 draws: 263.
__global__ void __cluster_dims__(kSampleCtas, 1, 1) __launch_bounds__(1024)
sample_pivots_kernel(const float *acc, int rows, int Lk, int period, int causal, int diag,
                     unsigned long long k_rest, unsigned long long n_rest, SelectState *state) {
  extern __shared__ uint32_t sm_dyn[];
  uint32_t *keys = sm_dyn;               // kSamples; 0 where a draw was dropped
  uint32_t *hist = sm_dyn + kSamples;    // kBins
  __shared__ uint32_t xch[2];
  __shared__ uint32_t n_valid_s;
  cg::cluster_group cluster = cg::this_cluster();
  after_previous();
  const int h = blockIdx.x / kSampleCtas, part = blockIdx.x % kSampleCtas, t = threadIdx.x, lane = t & 31;
  if (t == 0) n_valid_s = 0u;
  const int off = (causal || diag) ? Lk - period : 0;
  constexpr int kDraws = kSamples / (1024 * kSampleCtas);  // per thread, all loads in flight at once
  float drawn[kDraws];
  bool valid[kDraws];
#pragma unroll
  for (int u = 0; u < kDraws; ++u) {
    const int s = t + 1024 * (u + kDraws * part);
    // The rows are drawn in order (draw s from the s-th part of the selection's rows), which narrows the sample's spread if
    // anything and lets a warp's draws share a page; the column is a hash of the draw's number, scaled by multiplication.
    const uint32_t m = mix32((uint32_t)s + (uint32_t)h * (uint32_t)kSamples);
    constexpr uint32_t kSpan = (uint32_t)((1ull << 32) / kSamples);
    int i = (int)__umulhi((uint32_t)s * kSpan + (mix32(m ^ 0x9e3779b9u) & (kSpan - 1u)), (uint32_t)rows);
    int r = rows == period ? i : i % period;
    int j = (int)__umulhi(m, (uint32_t)Lk);
    if (causal && off == 0 && j > r) {
      // The part of the rectangle above the diagonal, turned by half a circle, covers the part below it once: no draw is
      // lost.  (The diagonal itself, which is usually forced anyway, is drawn half as often as the rest.)
      i += period - 1 - 2 * r;
      r = period - 1 - r;
      j = Lk - 1 - j;
    }
    const int own = r + off;
    valid[u] = !((causal && j > own) || (diag && j == own));
    drawn[u] = valid[u] ? acc[((size_t)h * rows + i) * Lk + j] : 0.f;
  }
  uint32_t mine = 0u;
#pragma unroll
  for (int u = 0; u < kDraws; ++u) mine += valid[u] ? 1u : 0u;
  mine = __reduce_add_sync(0xffffffffu, mine);
  cluster.sync();  // every CTA has started and cleared its count
#pragma unroll
  for (int to = 0; to < 2; ++to) {
    uint32_t *there = cluster.map_shared_rank(keys, to);
#pragma unroll
    for (int u = 0; u < kDraws; ++u) there[t + 1024 * (u + kDraws * part)] = valid[u] ? key_of(drawn[u]) : 0u;
    if (lane == 0) atomicAdd(cluster.map_shared_rank(&n_valid_s, to), mine);
  }
  cluster.sync();
  if (part >= 2) return;
  const uint32_t nv = n_valid_s;
  if (nv < 1024u) return;  // too few draws landed in the domain: no shortcut for this head
  // Expected rank of the threshold inside the sample and a bracket of 4.5 standard deviations: a selection that misses it
  // (one in a hundred thousand) takes the passes over the accumulator instead, and the collected entries, each of
  // which costs a push, three look-ups and a place in the buffer, are a quarter fewer than with six.  With the draws that
  // fall above the diagonal used as well (see below): 16 heads x 4096 (causal, 5 % kept) 333 -> 304 us.
  const double frac = (double)k_rest / (double)n_rest;
  const double r = frac * nv;
  const double dev = 4.5 * sqrt(fmax(r * (1.0 - frac), 1.0)) + 16.0;
  const long long r_hi = (long long)floor(r - dev), r_lo = (long long)ceil(r + dev);
  if (part == 0) {
    uint32_t hi = 0xffffffffu;
    if (r_hi >= 1) hi = block_select22(keys, (uint32_t)kSamples, (uint32_t)r_hi, hist, xch) | 0x3ffu;
    if (t == 0) state[h].hi = hi;
  } else {
    uint32_t lo = 0u;
    if (r_lo <= (long long)nv) lo = block_select22(keys, (uint32_t)kSamples, (uint32_t)r_lo, hist, xch);
    if (t == 0) state[h].lo = lo;
  }
  if (t == 0) state[h].use_shortcut = 1u;  // both CTAs take the same decision
}

// One pass over the selection's rows: counts the keys above the upper pivot and collects those
// inside the bracket.  grid = (row blocks, selections); a warp takes a row at a time.  Values are
// compared with the pivots as floats (the same order as their keys); the key is computed for the
// collected entries only.  Each warp stages its collected entries in shared memory and appends
// them to the selection's buffer, one reservation per flush, whenever the stage is half full at
// the end of a chunk of the row (an entry that finds the stage full goes straight to the buffer).
constexpr int kWarpStage = 512;
__global__ void __launch_bounds__(kThreads) collect_kernel(const float *__restrict__ acc, int Lq, int Lk, int period,
                                                           int causal, int diag, SelectState *state,
                                                           uint2 *__restrict__ cand, uint32_t cand_cap) {
  __shared__ uint2 stage_all[kWarps][kWarpStage];
  __shared__ uint32_t stage_n_all[kWarps];  // may run past the stage: those entries were not staged
  const int h = blockIdx.y;
  if (!state[h].use_shortcut) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint2 *stage = stage_all[warp];
  uint32_t *stage_n = &stage_n_all[warp];
  if (lane == 0) *stage_n = 0u;
  __syncwarp();
  const float lo_f = float_of_key(state[h].lo), hi_f = float_of_key(state[h].hi);
  uint2 *out = cand + (size_t)h * cand_cap;
  uint32_t *n_cand = &state[h].n_cand;
  auto push = [&](float f, uint32_t index) {  // a few per cent of the entries
    const uint2 entry = make_uint2(key_of(f), index);
    const uint32_t pos = atomicAdd(stage_n, 1u);
    if (pos < (uint32_t)kWarpStage) {
      stage[pos] = entry;
    } else {
      const uint32_t g = atomicAdd(n_cand, 1u);
      if (g < cand_cap) out[g] = entry;
    }
  };
  auto flush = [&](uint32_t at_least) {  // by the whole warp
    __syncwarp();
    const uint32_t n = min(*stage_n, (uint32_t)kWarpStage);
    if (n >= at_least && n > 0u) {
      uint32_t dst = 0u;
      if (lane == 0) dst = atomicAdd(n_cand, n);
      dst = __shfl_sync(0xffffffffu, dst, 0);
      for (uint32_t e = lane; e < n; e += 32)
        if (dst + e < cand_cap) out[dst + e] = stage[e];
      __syncwarp();
      if (lane == 0) *stage_n = 0u;
      __syncwarp();
    }
  };
  const bool vec = (Lk & 3) == 0;
  uint32_t above = 0u;  // per thread: fewer than 2^32 entries
  const int off = (causal || diag) ? Lk - period : 0;
  for (int i = blockIdx.x * kWarps + warp; i < Lq; i += gridDim.x * kWarps) {
    const float *row = acc + ((size_t)h * Lq + i) * Lk;
    const int own = i % period + off;  // the row's own position among the keys
    const int jend = causal ? min(Lk, own + 1) : Lk;
    const uint32_t row_index = (uint32_t)i * (uint32_t)Lk;
    for (int base = 0; base < jend; base += 512) {  // warp-uniform trip count
      float v[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j0 = base + 128 * u + 4 * lane;
        v[u][0] = v[u][1] = v[u][2] = v[u][3] = 0.f;
        if (j0 < jend) load4(row, j0, jend, vec, v[u]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j0 = base + 128 * u + 4 * lane;
        if (j0 + 4 <= jend && !(diag && own >= j0 && own < j0 + 4)) {
          // four entries of the domain: nothing to check per entry, and nothing to do at all where all
          // four lie below the bracket (most pieces of a row: the bracket sits near the top of the values)
          if (v[u][0] < lo_f && v[u][1] < lo_f && v[u][2] < lo_f && v[u][3] < lo_f) continue;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float f = v[u][c];
            const bool gt = f > hi_f;
            above += gt ? 1u : 0u;
            if (!(f < lo_f) && !gt) push(f, row_index + (uint32_t)(j0 + c));
          }
        } else if (j0 < jend) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int j = j0 + c;
            const float f = v[u][c];
            const bool in = j < jend && !(diag && j == own);
            const bool gt = in && f > hi_f;
            above += gt ? 1u : 0u;
            if (in && !(f < lo_f) && !gt) push(f, row_index + (uint32_t)j);
          }
        }
      }
      flush(kWarpStage / 2);
    }
  }
  flush(1u);
  unsigned long long above_warp = above;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) above_warp += __shfl_xor_sync(0xffffffffu, above_warp, o);
  if (lane == 0 && above_warp) atomicAdd(&state[h].above_hi, above_warp);
}

// ---- the select -----------------------------------------------------------------------------

constexpr int kSelThreads = 512;
constexpr int kSelCtasPerSm = 2;

// fn(value, linear index, whether the lane's entry is one of the selection's) for the selection's entries, spread over
// `n_warps` warps of which this is the `warp`-th: four 128-column pieces of rows at a time, a lane four consecutive
// entries of each (also where rows start anywhere: neighbours often fall into the same bin, and counting 32 of them at once,
// although the loads are contiguous then, is slower: 63 instead of 58 us at 16 heads x 375 x 759).  Called by whole warps, fn
// by all lanes together.
template <class F>
__device__ __forceinline__ void scan_domain(const float *__restrict__ base, int rows, int Lk, int period, int causal,
                                            int diag, uint32_t warp, uint32_t n_warps, int lane, F fn) {
  const int n_kt = (Lk + kTile - 1) / kTile, off = (causal || diag) ? Lk - period : 0;
  const uint32_t pieces = (uint32_t)rows * (uint32_t)n_kt;
  const bool vec = (Lk & 3) == 0;
  for (uint32_t p0 = 4u * warp; p0 < pieces; p0 += 4u * n_warps) {
    int i = (int)(p0 / (uint32_t)n_kt), kt = (int)(p0 - (uint32_t)i * (uint32_t)n_kt);
    float v[4][4];
    int row[4], col[4], jend[4], own[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      row[u] = i;
      col[u] = kt * kTile + 4 * lane;
      own[u] = i % period + off;
      jend[u] = i >= rows ? 0 : causal ? min(Lk, own[u] + 1) : Lk;
      v[u][0] = v[u][1] = v[u][2] = v[u][3] = 0.f;
      const float *from = base + (size_t)i * Lk + col[u];
      if (vec && col[u] + 4 <= jend[u]) {
        const float4 t = *reinterpret_cast<const float4 *>(from);
        v[u][0] = t.x, v[u][1] = t.y, v[u][2] = t.z, v[u][3] = t.w;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (col[u] + c < jend[u]) v[u][c] = from[c];
      }
      if (++kt == n_kt) {
        kt = 0;
        ++i;
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (!__any_sync(0xffffffffu, col[u] < jend[u])) continue;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int j = col[u] + c;
        fn(v[u][c], (uint32_t)row[u] * (uint32_t)Lk + (uint32_t)j, j < jend[u] && !(diag && j == own[u]));
      }
    }
  }
}

// The collected entries of a selection that the classifying pass left out and that are kept after all:
// above the threshold, or equal to it and within the ties that are kept.  By all threads of the selection's CTAs
// (warp-uniform trip count), four entries ahead each.  Entries that follow one another in the buffer were collected by one warp
// from one tile as a rule, so a warp's entries make one addition to that tile's count.  What bounds it: instructions.  (One
// entry at a time, and combining what falls into the same bitmap word: 25 us for 16 heads x 4096, 17 now.)
__device__ __forceinline__ void patch(const uint2 *__restrict__ cand, uint32_t n, uint32_t thr, uint32_t tie_cut, int h,
                                      uint32_t first, uint32_t step, int Lq, int Lk, int n_qt, int n_kt,
                                      uint8_t *__restrict__ mask, uint32_t *__restrict__ stage_bitmap,
                                      int32_t *__restrict__ stage_count, uint32_t *__restrict__ stage_groups) {
  constexpr int kAhead = 4;
  const int lane = threadIdx.x & 31;
  const uint32_t recip = 0xffffffffu / (uint32_t)Lk;
  for (uint32_t base = first - lane; base < n; base += kAhead * step) {
    uint2 c[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const uint32_t idx = base + u * step + lane;
      c[u] = make_uint2(0u, 0xffffffffu);
      if (idx < n) c[u] = cand[idx];
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const bool keep = base + u * step + lane < n && (c[u].x > thr || (c[u].x == thr && c[u].y <= tie_cut));
      uint32_t voters = __ballot_sync(0xffffffffu, keep);
      if (voters == 0u) continue;
      uint32_t i = __umulhi(c[u].y, recip), j = c[u].y - i * (uint32_t)Lk;  // (one too low at most)
      if (j >= (uint32_t)Lk) ++i, j -= (uint32_t)Lk;
      if (keep && mask) mask[((size_t)h * Lq + i) * Lk + j] = 1;
      if (!stage_bitmap) continue;
      const uint32_t tile = (uint32_t)((h * n_qt + (int)(i >> 7)) * n_kt + (int)(j >> 7));
      if (keep) atomicOr(stage_bitmap + (size_t)tile * kBitmapWords + 4u * (i & 127u) + ((j & 127u) >> 5), 1u << (j & 31u));
      const uint32_t group = keep ? 1u << ((j & 127u) >> 4) : 0u;
      while (voters) {
        const uint32_t lead = __shfl_sync(0xffffffffu, tile, __ffs((int)voters) - 1);
        const bool same = keep && tile == lead;
        const uint32_t group_bits = __reduce_or_sync(0xffffffffu, same ? group : 0u);
        const uint32_t sames = __ballot_sync(0xffffffffu, same);
        if (lane == 0) {
          atomicAdd(stage_count + lead, __popc(sames));
          atomicOr(stage_groups + lead, group_bits);
        }
        voters &= ~sames;
      }
    }
  }
}

// Cooperative.  Selection h belongs to per_sel CTAs (one CTA takes several selections in turn where there are more
// of them than CTAs): finds its threshold and the index of the last kept entry equal to it, and, where the
// classifying pass has written the mask and the bitmaps, adds the collected entries that are kept.
//
// What bounds it: three times (load latency + a few microseconds of shared-memory histogram + a barrier of about
// 1.5 us); the passes read from L2.  Two CTAs of 512 threads per SM, so that one's loads run under the other's counting.
// kCand: the launch has collected entries.  Without any, the scan alone: beside the rest it compiles to slower code (32 heads x
// 1407, causal: 337 us with it, 291 without).
template <bool kCand>
__global__ void __launch_bounds__(kSelThreads, kSelCtasPerSm)
select_kernel(const float *acc, int rows, int Lk, int period, int causal, int diag,
              unsigned long long k_rest, int n_sel, int per_sel, SelectState *state, uint32_t *hist,
              const uint2 *cand, uint32_t cand_cap, int keep_ties, int H, long long nnz_init,
              int64_t *__restrict__ nnz, int classified, int Lq, int n_qt, int n_kt, uint8_t *__restrict__ mask,
              uint32_t *__restrict__ stage_bitmap, int32_t *__restrict__ stage_count,
              uint32_t *__restrict__ stage_groups, unsigned *err) {
  __shared__ __align__(16) uint32_t sh[kBins];
  __shared__ uint32_t warp_sums[kSelThreads / 32];
  __shared__ uint32_t pick_bin, pick_count;
  __shared__ unsigned long long pick_rest;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  after_previous();
  if (nnz)
    for (int x = blockIdx.x * kSelThreads + threadIdx.x; x < H; x += gridDim.x * kSelThreads) nnz[x] = nnz_init;
  const int rank = (int)blockIdx.x % per_sel;
  for (int h = (int)blockIdx.x / per_sel; h < n_sel; h += (int)gridDim.x / per_sel) {
    SelectState &st = state[h];
    if (k_rest == 0ull) {  // nothing but the forced entries is kept
      if (rank == 0 && threadIdx.x == 0) st.thr = 0xffffffffu;
      continue;
    }
    // the bracket holds the threshold and every key of the bracket was collected
    const bool from_cand = kCand && st.use_shortcut && st.n_cand <= cand_cap && st.above_hi < k_rest &&
                           k_rest - st.above_hi <= st.n_cand;
    // offsets from the lower pivot, moved up so that the bracket's span begins with the leading digit: the last digits are
    // zero for all, and skipped, where the span is short (as a rule the last one: two digits instead of three)
    const uint32_t lo = from_cand ? st.lo : 0u, span = from_cand ? st.hi - st.lo : 0xffffffffu;
    const int up = span ? __clz((int)span) : 31;
    const uint32_t n_cand = st.n_cand;
    const uint2 *mine = cand + (size_t)h * cand_cap;
    const float *base = acc + (size_t)h * rows * Lk;
    unsigned long long rest = from_cand ? k_rest - st.above_hi : k_rest;
    uint32_t prefix = 0u, thr = 0u, arrived = 0u;
    uint32_t tie_cut = 0xffffffffu;
    int turn = 0;  // histogram buffers used so far
    for (int digit = 0; digit < 2 * kPasses; ++digit) {
      const int pass = digit % kPasses;
      const bool of_index = digit >= kPasses;
      if (digit == kPasses) {
        thr = (prefix >> up) + lo;
        prefix = 0u;
        if (keep_ties || rest == pick_count) break;  // every entry equal to the threshold is kept
      }
      if (!of_index && pass > 0 && digit_shift(pass - 1) <= up) continue;
      const int shift = digit_shift(pass);
      const uint32_t dmask = digit_mask(pass), hi_mask = above_digit(pass);
      for (int b = threadIdx.x; b < kBins; b += kSelThreads) sh[b] = 0u;
      __syncthreads();
      auto count = [&](uint32_t key, uint32_t index, bool there) {
        const uint32_t word = of_index ? ~index : (key - lo) << up;
        if (there && (word & hi_mask) == prefix && (!of_index || key == thr)) atomicAdd(&sh[(word >> shift) & dmask], 1u);
      };
      if (from_cand) {
        constexpr int kAhead = 8;  // loads in flight
        const uint32_t step = (uint32_t)per_sel * kSelThreads * kAhead;
        for (uint32_t x0 = (uint32_t)rank * (kAhead * kSelThreads) + threadIdx.x; x0 < n_cand + threadIdx.x; x0 += step) {
          uint2 c[kAhead];
#pragma unroll
          for (int u = 0; u < kAhead; ++u) {
            const uint32_t x = x0 + u * kSelThreads;
            c[u] = x < n_cand ? mine[x] : make_uint2(0u, 0u);
          }
#pragma unroll
          for (int u = 0; u < kAhead; ++u) count(c[u].x, c[u].y, x0 + u * kSelThreads < n_cand);
        }
      } else {
        scan_domain(base, rows, Lk, period, causal, diag, (uint32_t)(warp * per_sel + rank),
                    (uint32_t)(per_sel * (kSelThreads / 32)), lane,
                    [&](float f, uint32_t index, bool there) { count(key_of(f), index, there); });
      }
      __syncthreads();
      // thread t owns bins 2047 - 4t .. 2044 - 4t (descending); the owner of the wanted rank picks the digit
      uint4 own;
      if (per_sel > 1) {
        uint32_t *all = hist + ((size_t)h * kHistBuffers + turn % kHistBuffers) * kBins;
        for (int b = threadIdx.x; b < kBins; b += kSelThreads)
          if (sh[b]) atomicAdd(all + b, sh[b]);
        if (turn >= 2) {  // the buffer of two digits ago has been read by all: ready for the next digit but ...
          uint32_t *old = hist + ((size_t)h * kHistBuffers + (turn - 2) % kHistBuffers) * kBins;
          for (int b = rank * kSelThreads + threadIdx.x; b < kBins; b += per_sel * kSelThreads) old[b] = 0u;
        }
        arrived += (uint32_t)per_sel;
        if (!cta_barrier(&st.barrier, arrived, err)) return;
        own = __ldcg(reinterpret_cast<const uint4 *>(all) + (kBins / 4 - 1 - (int)threadIdx.x));
        ++turn;
      } else {
        own = reinterpret_cast<const uint4 *>(sh)[kBins / 4 - 1 - (int)threadIdx.x];
      }
      const uint32_t c[4] = {own.w, own.z, own.y, own.x}, sum = (own.x + own.y) + (own.z + own.w);
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) warp_sums[warp] = incl;
      __syncthreads();
      unsigned long long before = incl - sum;  // entries in bins above this thread's
      before += __reduce_add_sync(0xffffffffu, lane < warp ? warp_sums[lane] : 0u);  // (a selection has fewer than 2^32 entries)
      if (before < rest && before + sum >= rest) {  // exactly one thread
        int e = 0;
        for (; e < 3 && before + c[e] < rest; ++e) before += c[e];
        pick_bin = (uint32_t)(kBins - 1 - 4 * (int)threadIdx.x - e);
        pick_rest = rest - before;
        pick_count = e == 0 ? c[0] : e == 1 ? c[1] : e == 2 ? c[2] : c[3];
      }
      __syncthreads();
      prefix |= pick_bin << shift;
      rest = pick_rest;
      if (digit == 2 * kPasses - 1) tie_cut = ~prefix;
    }
    if (rank == 0 && threadIdx.x == 0) {
      st.thr = thr;
      st.tie_cut = tie_cut;
      st.emitted = classified && from_cand ? 1u : 0u;
    }
    if (classified && from_cand)
      patch(mine, n_cand, thr, tie_cut, h, (uint32_t)(rank * kSelThreads + threadIdx.x), (uint32_t)(per_sel * kSelThreads),
            Lq, Lk, n_qt, n_kt, mask, stage_bitmap, stage_count, stage_groups);
    __syncthreads();
  }
}

// A warp's way into a selection's buffer of collected entries: staged in shared memory and appended with one reservation
// per flush.  By the whole warp; the number staged is the same in all lanes.
struct Collector {
  uint2 *stage;      // this warp's kWarpStage entries of shared memory
  uint32_t staged;
  uint2 *out;        // the selection's buffer
  uint32_t *n_cand;  // entries reserved in it so far (may exceed the capacity: then the shortcut fails)
  uint32_t cap;
  // the lane's entries go to stage[at ...]; `total` <= kWarpStage is the warp's number of them
  __device__ __forceinline__ uint32_t reserve(uint32_t before_me, uint32_t total, int lane) {
    if (staged + total > (uint32_t)kWarpStage) flush(lane);
    const uint32_t at = staged + before_me;
    staged += total;
    return at;
  }
  __device__ __forceinline__ void flush(int lane) {
    if (staged == 0u) return;
    __syncwarp();
    uint32_t dst = 0u;
    if (lane == 0) dst = atomicAdd(n_cand, staged);
    dst = __shfl_sync(0xffffffffu, dst, 0);
    for (uint32_t e = lane; e < staged; e += 32)
      if (dst + e < cap) out[dst + e] = stage[e];
    __syncwarp();
    staged = 0u;
  }
};

// What the emit pass needs of a selection.
struct EmitSel {
  float thr_f;  // the threshold as a float (NaN when nothing but the forced entries is kept)
  float lo_f;   // classifying pass: thr_f is the bracket's upper pivot, lo_f its lower one
  uint32_t tie_cut;    // entries equal to the threshold are kept up to this index
  uint32_t first_row;  // of this head in the tie order
};

// The two ways over the rows of one tile, each by kCtaWarps warps.  Both write the mask and the bitmap and return what
// the lane has seen: `count` kept entries (to be added up over the lanes), `groups` of 16 columns with a kept entry (to be
// combined), `above` entries above the bracket (kClassify; to be added up).
// kClassify: the classifying pass of the one-pass shortcut instead of the emit pass proper.  Entries above the bracket are
// kept, entries inside it are collected (col) and left out for the select to decide, entries above the bracket are counted.
//
// What bounds them: instructions, not memory.  With four columns per lane (a test of each, three shuffles to a bitmap word
// and a four-byte mask store per row) the classifying pass issued 121 instructions per row of a tile and reached 2.6 TB/s at
// 16 heads x 2048 (causal).  Whole selections then and now: 16 x 4096 causal 304 -> 268 us; rows that start anywhere
// (16 x 2501) 240 -> 202 us, one threshold for the layer 260 -> 200 us.
struct TileSums {
  int count;
  uint32_t groups, above;
};

// Tiles all of whose rows and columns exist, lie in the domain and are not forced.  kVec = 8: in arrays whose rows
// start on 32-byte (scores) and 16-byte (mask) boundaries; 4: on 16-byte and 4-byte ones.  A lane takes 16
// consecutive columns of one row, i.e. one group of the tile: its bits are half a bitmap word, its mask bytes one
// 16-byte store, and where all 16 lie below the bracket (most of them do: it sits near the top of the values) one
// comparison of their maximum says so.  A warp has four rows under way and the next four loaded ahead.
template <bool kClassify, int kCtaWarps, int kVec>
__device__ __forceinline__ void emit_rows_by_group(const float *__restrict__ acc, int Lq, int Lk, int h, int qt, int kt,
                                                   int tile, const EmitSel &sel, uint8_t *__restrict__ mask,
                                                   uint32_t *__restrict__ stage_bitmap, Collector &col, TileSums &sums) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = kt * kTile + 16 * (lane & 7), r_lane = lane >> 3;
  const float thr_f = sel.thr_f;
  const float floor_f = kClassify ? sel.lo_f : thr_f;  // the lowest value that needs a closer look
  const int r_first = 4 * warp + r_lane;
  size_t at = ((size_t)h * Lq + qt * kTile + r_first) * Lk + j0;
  const size_t step = (size_t)(4 * kCtaWarps) * Lk;
  float v[16], ahead[16];
  ldg_f16<kVec>(acc + at, ahead);
  uint32_t first = (sel.first_row + (uint32_t)(qt * kTile + r_first)) * (uint32_t)Lk + (uint32_t)j0;
  size_t bits_at = (size_t)tile * (2 * kBitmapWords) + 8 * r_first + (lane & 7);  // in half-words
#pragma unroll 1
  for (int r0 = 4 * warp; r0 < kTile; r0 += 4 * kCtaWarps) {
#pragma unroll
    for (int c = 0; c < 16; ++c) v[c] = ahead[c];
    if (r0 + 4 * kCtaWarps < kTile) ldg_f16<kVec>(acc + at + step, ahead);
    uint32_t kept = 0u, ties = 0u;
    // (written so that a value that is not a number gets the closer look as well)
    bool below = true;
#pragma unroll
    for (int c = 0; c < 16; ++c) below = below && v[c] < floor_f;
    if (!below) {
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const bool gt = v[c] > thr_f;
        kept |= (gt ? 1u : 0u) << c;
        ties |= ((kClassify ? !(v[c] < floor_f) && !gt : v[c] == thr_f) ? 1u : 0u) << c;
      }
      if (kClassify) {
        sums.above += (uint32_t)__popc(kept);
      } else if (ties && first <= sel.tie_cut) {  // entries equal to the threshold, up to the last kept one
        const uint32_t last = sel.tie_cut - first;
        kept |= last >= 15u ? ties : ties & ((2u << last) - 1u);
      }
    }
    if (kClassify && __any_sync(0xffffffffu, ties != 0u)) {
      const uint32_t mine = (uint32_t)__popc(ties);
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      uint32_t pos = col.reserve(incl - mine, __shfl_sync(0xffffffffu, incl, 31), lane);
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if ((ties >> c) & 1u) col.stage[pos++] = make_uint2(key_of(v[c]), first + c);
    }
    if (mask) {
      uint4 bytes;  // four bits to four bytes: the products of the shifted copies do not meet
      bytes.x = ((kept & 15u) * 0x00204081u) & 0x01010101u;
      bytes.y = (((kept >> 4) & 15u) * 0x00204081u) & 0x01010101u;
      bytes.z = (((kept >> 8) & 15u) * 0x00204081u) & 0x01010101u;
      bytes.w = ((kept >> 12) * 0x00204081u) & 0x01010101u;
      if (kVec == 8) {
        *reinterpret_cast<uint4 *>(mask + at) = bytes;
      } else {
        uint32_t *words = reinterpret_cast<uint32_t *>(mask + at);
        words[0] = bytes.x, words[1] = bytes.y, words[2] = bytes.z, words[3] = bytes.w;
      }
    }
    if (stage_bitmap) reinterpret_cast<uint16_t *>(stage_bitmap)[bits_at] = (uint16_t)kept;
    sums.count += __popc(kept);
    sums.groups |= kept ? 1u << (lane & 7) : 0u;
    at += step;
    first += (uint32_t)(4 * kCtaWarps) * (uint32_t)Lk;
    bits_at += 8 * 4 * kCtaWarps;
  }
}

// Every other tile: a lane takes the columns lane, lane + 32, ... of a row, so that loads and mask stores of a warp are
// contiguous wherever the row starts, and a vote of the warp is a bitmap word.  Four rows loaded ahead.
// kInterior: as for emit_rows_by_group (rows that start anywhere), nothing is checked per entry and a row all of whose
// entries lie below the bracket takes one vote.
template <bool kClassify, int kCtaWarps, bool kInterior>
__device__ __forceinline__ void emit_rows_by_column(const float *__restrict__ acc, int Lq, int Lk, int h, int qt, int kt,
                                                    int tile, int causal, int diag, const EmitSel &sel,
                                                    uint8_t *__restrict__ mask, uint32_t *__restrict__ stage_bitmap,
                                                    Collector &col, TileSums &sums) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float thr_f = sel.thr_f;
  const float floor_f = kClassify ? sel.lo_f : thr_f;
  const int off = (causal || diag) ? Lk - Lq : 0;  // row i's own position is key i + off
  const int j_lane = kt * kTile + lane;
  const int rows = kInterior ? kTile : min(kTile, Lq - qt * kTile);
  int count = 0;  // the same in all lanes
  uint32_t any[4] = {0u, 0u, 0u, 0u};
#pragma unroll 1
  for (int r0 = warp; r0 < rows; r0 += 4 * kCtaWarps) {
    float v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = qt * kTile + r0 + kCtaWarps * u;
      const int jend = i >= Lq ? 0 : causal ? min(Lk, i + 1 + off) : Lk;
      const float *row = acc + ((size_t)h * Lq + i) * Lk + j_lane;
#pragma unroll
      for (int q = 0; q < 4; ++q) v[u][q] = kInterior || j_lane + 32 * q < jend ? row[32 * q] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + kCtaWarps * u, i = qt * kTile + r;
      if (r >= rows) break;
      uint32_t w[4] = {0u, 0u, 0u, 0u};
      if (!kInterior ||
          __any_sync(0xffffffffu, !(v[u][0] < floor_f && v[u][1] < floor_f && v[u][2] < floor_f && v[u][3] < floor_f))) {
        const int jend = causal ? min(Lk, i + 1 + off) : Lk;
        const int own = diag ? i + off : -1;
        const uint32_t first = (sel.first_row + (uint32_t)i) * (uint32_t)Lk + (uint32_t)j_lane;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int j = j_lane + 32 * q;
          const bool forced = !kInterior && j == own;
          const bool in = kInterior || (j < jend && !forced);
          const bool gt = in && v[u][q] > thr_f;
          bool keep = gt || forced;
          if (kClassify) {
            const bool tie = in && !gt && !(v[u][q] < floor_f);
            sums.above += gt ? 1u : 0u;
            const uint32_t inside = __ballot_sync(0xffffffffu, tie);
            if (inside) {
              const uint32_t pos = col.reserve(__popc(inside & ((1u << lane) - 1u)), (uint32_t)__popc(inside), lane);
              if (tie) col.stage[pos] = make_uint2(key_of(v[u][q]), first + 32u * q);
            }
          } else {
            keep = keep || (in && v[u][q] == thr_f && first + 32u * q <= sel.tie_cut);
          }
          w[q] = __ballot_sync(0xffffffffu, keep);
          count += __popc(w[q]);
          any[q] |= w[q];
        }
      }
      if (mask) {
        uint8_t *mrow = mask + ((size_t)h * Lq + i) * Lk + j_lane;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (kInterior || j_lane + 32 * q < Lk) mrow[32 * q] = (w[q] >> lane) & 1u;
      }
      if (stage_bitmap && lane == 0)
        *reinterpret_cast<uint4 *>(stage_bitmap + (size_t)tile * kBitmapWords + 4 * r) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  if (!kInterior && stage_bitmap)  // rows beyond the last query keep nothing
    for (int x = rows + (int)threadIdx.x; x < kTile; x += 32 * kCtaWarps)
      *reinterpret_cast<uint4 *>(stage_bitmap + (size_t)tile * kBitmapWords + 4 * x) = make_uint4(0u, 0u, 0u, 0u);
  if (lane == 0) {
    sums.count += count;
#pragma unroll
    for (int q = 0; q < 4; ++q) sums.groups |= ((any[q] & 0xffffu ? 1u : 0u) | (any[q] >> 16 ? 2u : 0u)) << (2 * q);
  }
}

// A CTA per tile of the (h, qt, kt) grid (a CTA takes several in turn where the grid is smaller).
// Writes the element mask, the tile's bitmap, popcount and group summary into the staging area.
// Values are compared with the threshold as floats (the same order as their keys).  per_layer:
// all heads share selection 0, ties are ordered by (h*Lq + i)*Lk + j, and the
// tiles' popcounts are added up into nnz[h].  keep_ties: every entry equal to the threshold is
// kept, and the popcounts are added up as well (the count is not known beforehand).
// kClassify: the shortcut's one pass over the accumulator, which does the collecting pass's work
// (entries above the upper pivot counted, entries inside the bracket appended to the selection's
// buffer) and most of the emit pass's at once: everything above the bracket is kept, everything else
// left out, and the select adds the collected entries that turn out to be kept.  Only for exact
// per-head selections (the kept count is known beforehand, nothing is counted here).
template <bool kClassify, int kCtaWarps>
__global__ void __launch_bounds__(32 * kCtaWarps, kCtaWarps == 4 ? 8 : 2) emit_kernel(const float *acc, int Lq, int Lk, int n_qt,
                                                              int n_kt, int n_tiles, int causal, int diag, int per_layer,
                                                              int keep_ties, SelectState *state,
                                                              uint8_t *__restrict__ mask,
                                                              uint32_t *__restrict__ stage_bitmap,
                                                              int32_t *__restrict__ stage_count,
                                                              uint32_t *__restrict__ stage_groups,
                                                              int64_t *__restrict__ nnz, uint2 *__restrict__ cand,
                                                              uint32_t cand_cap) {
  __shared__ int warp_count[kCtaWarps];
  __shared__ uint32_t warp_groups[kCtaWarps];
  __shared__ uint2 stage_all[kClassify ? kCtaWarps : 1][kClassify ? kWarpStage : 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  after_previous();
  // rows of the scores start on 32-byte boundaries and rows of the mask on 16-byte ones
  const bool aligned4 = (Lk & 3) == 0 && ((reinterpret_cast<uintptr_t>(acc) & 15) | (reinterpret_cast<uintptr_t>(mask) & 3)) == 0;
  const bool aligned = (Lk & 15) == 0 && ((reinterpret_cast<uintptr_t>(acc) & 31) | (reinterpret_cast<uintptr_t>(mask) & 15)) == 0;
  if (!kClassify && !per_layer) {  // as a rule a classified selection has its mask by now: one look at all of them
    bool pending = false;
    const int H = n_tiles / (n_qt * n_kt);
    for (int x = lane; x < H; x += 32) pending |= state[x].emitted == 0u;
    if (!__any_sync(0xffffffffu, pending)) return;
  }
  for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int kt = tile % n_kt;
    const int qt = (tile / n_kt) % n_qt;
    const int h = tile / (n_kt * n_qt);
    SelectState &st = state[per_layer ? 0 : h];
    if (kClassify ? !st.use_shortcut : st.emitted != 0u) continue;  // not this pass's selection
    // own positions of the tile's rows among the keys: columns own_lo .. own_hi
    const int own_lo = qt * kTile + ((causal || diag) ? Lk - Lq : 0), own_hi = own_lo + kTile - 1;
    if (causal && kt * kTile > own_hi) {
      // the whole tile lies above the diagonal: nothing is kept, nothing needs to be read
      if (mask && aligned) {
        const int j0 = kt * kTile + 16 * (lane & 7);
        for (int r = 4 * warp + (lane >> 3); r < kTile; r += 4 * kCtaWarps) {
          const int i = qt * kTile + r;
          if (i < Lq && j0 < Lk) *reinterpret_cast<uint4 *>(mask + ((size_t)h * Lq + i) * Lk + j0) = make_uint4(0u, 0u, 0u, 0u);
        }
      } else if (mask) {
        for (int r = warp; r < kTile; r += kCtaWarps) {
          const int i = qt * kTile + r;
          if (i >= Lq) break;
          for (int j = kt * kTile + lane; j < min(Lk, (kt + 1) * kTile); j += 32) mask[((size_t)h * Lq + i) * Lk + j] = 0;
        }
      }
      // (the bitmap of an empty tile is not read)
      if (stage_count && threadIdx.x == 0) {
        stage_count[tile] = 0;
        stage_groups[tile] = 0u;
      }
      continue;
    }
    EmitSel sel;
    sel.thr_f = float_of_key(kClassify ? st.hi : st.thr);
    sel.lo_f = float_of_key(st.lo);
    sel.tie_cut = st.tie_cut;
    sel.first_row = per_layer ? (uint32_t)h * (uint32_t)Lq : 0u;
    Collector col;
    col.stage = stage_all[kClassify ? warp : 0];
    col.staged = 0u;
    col.out = cand + (size_t)(per_layer ? 0 : h) * cand_cap;
    col.n_cand = &st.n_cand;
    col.cap = cand_cap;
    TileSums sums = {0, 0u, 0u};
    const bool below = !causal || kt * kTile + kTile - 1 <= own_lo;  // every column in every row's domain
    const bool has_diag = diag && own_lo <= kt * kTile + kTile - 1 && own_hi >= kt * kTile;
    if ((qt + 1) * kTile <= Lq && (kt + 1) * kTile <= Lk && below && !has_diag) {
      if (aligned)
        emit_rows_by_group<kClassify, kCtaWarps, 8>(acc, Lq, Lk, h, qt, kt, tile, sel, mask, stage_bitmap, col, sums);
      else if (aligned4)
        emit_rows_by_group<kClassify, kCtaWarps, 4>(acc, Lq, Lk, h, qt, kt, tile, sel, mask, stage_bitmap, col, sums);
      else
        emit_rows_by_column<kClassify, kCtaWarps, true>(acc, Lq, Lk, h, qt, kt, tile, causal, diag, sel, mask, stage_bitmap,
                                                        col, sums);
    } else {
      emit_rows_by_column<kClassify, kCtaWarps, false>(acc, Lq, Lk, h, qt, kt, tile, causal, diag, sel, mask, stage_bitmap,
                                                       col, sums);
    }
    if (kClassify) {
      col.flush(lane);
      const uint32_t above = __reduce_add_sync(0xffffffffu, sums.above);
      if (lane == 0 && above) atomicAdd(&st.above_hi, (unsigned long long)above);
    }
    if (!stage_bitmap && !(nnz && !kClassify && (per_layer || keep_ties))) continue;
    const int count = __reduce_add_sync(0xffffffffu, sums.count);
    const uint32_t groups = __reduce_or_sync(0xffffffffu, sums.groups);
    if (lane == 0) {
      warp_count[warp] = count;
      warp_groups[warp] = groups;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      int total = 0;
      uint32_t all = 0u;
#pragma unroll
      for (int w = 0; w < kCtaWarps; ++w) {
        total += warp_count[w];
        all |= warp_groups[w];
      }
      if (stage_count) {
        stage_count[tile] = total;
        stage_groups[tile] = all;
      }
      if (!kClassify && (per_layer || keep_ties) && nnz && total)
        atomicAdd(reinterpret_cast<unsigned long long *>(nnz + h), (unsigned long long)total);
    }
    __syncthreads();  // warp_count is read
  }
}

// ---- inputs that fit into shared memory --------------------------------------------------------

constexpr int kHeldThreads = 1024;
constexpr int kUnitRows = 32, kUnitWords = kUnitRows * kTile;  // a quarter of a 128 x 128 tile: a row per warp
constexpr int kHeldUnits = 12;                                 // per CTA at most, one CTA per SM
constexpr int kHeldSels = kHeldUnits / 4 + 1;                  // selections that these belong to at most (four units each or more)

// The units of the domain's tiles, selection by selection, dealt out evenly to the CTAs of the grid.
struct Held {
  int H, Lq, Lk, n_qt, n_kt, causal, per_layer;
  int per_head;  // units of a head's domain
  __host__ __device__ int total() const { return H * per_head; }
  __device__ int first_of(int cta, int ctas) const { return (int)((long long)cta * total() / ctas); }
  __device__ int owner_of(int u, int ctas) const { return (int)(((long long)(u + 1) * ctas - 1) / total()); }
  __device__ int sel_of(int u) const { return per_layer ? 0 : u / per_head; }
  // the CTAs that hold a unit of the selection: `first` and how many
  __device__ int2 ctas_of(int sel, int ctas) const {
    const int n = per_layer ? total() : per_head, first = owner_of(sel * n, ctas);
    return make_int2(first, owner_of((sel + 1) * n - 1, ctas) - first + 1);
  }
};

// Cooperative.  The whole of a call but the compaction in one kernel: every CTA copies its units into shared memory as keys,
// takes part in the select of the selections they belong to, and writes their mask and bitmaps.
//
// What bounds it: latency, three times a histogram, its merging into global memory, a barrier of the selection's CTAs and the
// pick of a digit.  The accumulator is read once; with a scan of it per digit and an emit pass of its own one layer of
// 16 heads x 512 took 60 us, 39 with this kernel, some 20 of them its own (59 with whole tiles instead of quarters, of which a
// few CTAs then have two; 31 with the list's and the launches' part shortened as well).  The first histogram's counts fall into
// few bins (a digit is little more than the exponent), so a warp takes entries of different rows and columns: neighbours,
// which are alike, would queue for the same bin.  The price of the shared memory: the CTAs have an SM each to themselves, all of
// them at once, so beside another stream's kernel that fills the SMs the call begins when that one has left them.
__global__ void __launch_bounds__(kHeldThreads, 1)
held_kernel(const float *acc, const Held p, int diag, unsigned long long k_rest, SelectState *state,
            uint32_t *hist, int keep_ties, long long nnz_init, int64_t *__restrict__ nnz, uint8_t *__restrict__ mask,
            uint32_t *__restrict__ stage_bitmap, int32_t *__restrict__ stage_count, uint32_t *__restrict__ stage_groups,
            unsigned *err) {
  extern __shared__ __align__(16) uint32_t held_smem[];
  uint32_t *counts_s = held_smem;                     // [kHeldSels][kBins]: a histogram per selection of the CTA
  uint32_t *keys_s = held_smem + kHeldSels * kBins;   // [units][32][128]; 0: not one of the selection's
  struct Unit {
    int h, row0, kt, tile;
  };
  struct Sel {  // the select's progress
    unsigned long long rest;
    uint32_t prefix, thr, tie_cut, count;
    int going, sharers, rank;
  };
  __shared__ Unit units[kHeldUnits];
  __shared__ Sel sels[kHeldSels];
  __shared__ uint32_t warp_sums[kHeldThreads / 32], unit_votes[kHeldUnits];
  __shared__ int unit_count[kHeldUnits], ok_s;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, ctas = (int)gridDim.x, cta = (int)blockIdx.x;
  const int Lq = p.Lq, Lk = p.Lk, off = (p.causal || diag) ? Lk - Lq : 0;
  const int u0 = p.first_of(cta, ctas), n_units = p.first_of(cta + 1, ctas) - u0;
  const int sel0 = p.sel_of(u0), n_sel = p.sel_of(u0 + n_units - 1) - sel0 + 1;
  after_previous();
  if (t < n_units) {
    const int h = (u0 + t) / p.per_head, in_head = (u0 + t) - h * p.per_head;
    int qt = 0;
    while (qt + 1 < p.n_qt && (int)dense_row_start(qt + 1, p.n_kt, Lq, Lk, p.causal) <= in_head / 4) ++qt;
    const int kt = in_head / 4 - (int)dense_row_start(qt, p.n_kt, Lq, Lk, p.causal), tile = (h * p.n_qt + qt) * p.n_kt + kt;
    units[t] = Unit{h, qt * kTile + kUnitRows * (in_head & 3), kt, tile};
    unit_votes[t] = 0u;
    unit_count[t] = 0;
    // (added to by the CTAs of the selection, behind a barrier of theirs)
    if (stage_count && (in_head & 3) == 0) {
      stage_count[tile] = 0;
      stage_groups[tile] = 0u;
    }
    if (nnz && in_head == 0) nnz[h] = nnz_init;
  }
  if (t < n_sel) {
    const int2 c = p.ctas_of(sel0 + t, ctas);
    sels[t] = Sel{k_rest, 0u, 0u, 0xffffffffu, 0u, 1, c.y, cta - c.x};
  }
  __syncthreads();
  // ---- keys of this CTA's units
  const bool vec = (Lk & 3) == 0 && (reinterpret_cast<uintptr_t>(acc) & 15) == 0;
#pragma unroll 1
  for (int x0 = 0; x0 < n_units; x0 += 4) {
    float v[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      v[u][0] = v[u][1] = v[u][2] = v[u][3] = 0.f;
      if (x0 + u < n_units) {
        const Unit un = units[x0 + u];
        const int i = un.row0 + warp;
        if (i < Lq) load4(acc + ((size_t)un.h * Lq + i) * Lk, un.kt * kTile + 4 * lane, Lk, vec, v[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (x0 + u < n_units) {
        const Unit un = units[x0 + u];
        const int i = un.row0 + warp, own = i + off, j = un.kt * kTile + 4 * lane;
        const int jend = i >= Lq ? 0 : p.causal ? min(Lk, own + 1) : Lk;
        uint32_t k[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) k[c] = j + c < jend && !(diag && j + c == own) ? key_of(v[u][c]) : 0u;
        reinterpret_cast<uint4 *>(keys_s + (x0 + u) * kUnitWords)[t] = make_uint4(k[0], k[1], k[2], k[3]);
      }
  }
  // Tiles outside the domain: nothing is kept (their bitmaps are not read).  Written while the first digit's counts come in.
  const bool mask4 = (Lk & 3) == 0 && (reinterpret_cast<uintptr_t>(mask) & 3) == 0;
  auto clear_outside = [&]() {
    const int n_rows = p.H * p.n_qt;
    for (int x = cta; x < n_rows; x += ctas) {
      const int h = x / p.n_qt, qt = x % p.n_qt, kt0 = dense_row_tiles(qt, p.n_kt, Lq, Lk, 1);
      if (mask) {
        const int j0 = kt0 * kTile;
        for (int i = qt * kTile + warp; i < min(Lq, (qt + 1) * kTile); i += kHeldThreads / 32) {
          uint8_t *m = mask + ((size_t)h * Lq + i) * Lk;
          if (mask4) {
            for (int j = j0 + 4 * lane; j < Lk; j += kTile) *reinterpret_cast<uint32_t *>(m + j) = 0u;
          } else {
            for (int j = j0 + lane; j < Lk; j += 32) m[j] = 0;
          }
        }
      }
      if (stage_count && t < p.n_kt - kt0) {
        stage_count[x * p.n_kt + kt0 + t] = 0;
        stage_groups[x * p.n_kt + kt0 + t] = 0u;
      }
    }
  };
  // ---- select
  const uint32_t *my_keys = keys_s + ((warp + 11 * lane) & 31) * kTile + lane;  // + 32 e: this thread's four entries of a unit
#pragma unroll 1
  for (int digit = 0; digit < 2 * kPasses; ++digit) {
    const int pass = digit % kPasses, shift = digit_shift(pass);
    const bool of_index = digit >= kPasses;
    const uint32_t dmask = digit_mask(pass), hi_mask = above_digit(pass);
    for (int b = t; b < n_sel * kBins; b += kHeldThreads) counts_s[b] = 0u;
    __syncthreads();  // (the keys are there, the last digit has been picked)
    bool any = false;
#pragma unroll 1
    for (int q = 0; q < n_sel; ++q) {
      if (!sels[q].going) continue;
      any = true;
      const uint32_t pre = sels[q].prefix, thr = sels[q].thr;
      uint32_t *mine = counts_s + q * kBins;
      const int n = p.per_layer ? p.total() : p.per_head;  // units of a selection
      const int x0 = max((sel0 + q) * n - u0, 0), x1 = min((sel0 + q + 1) * n - u0, n_units);
      if (!of_index) {
#pragma unroll 2
        for (int x = x0; x < x1; ++x) {
          uint32_t k[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) k[e] = my_keys[x * kUnitWords + 32 * e];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (k[e] != 0u && (k[e] & hi_mask) == pre) atomicAdd(&mine[(k[e] >> shift) & dmask], 1u);
        }
      } else {
        for (int x = x0; x < x1; ++x) {
          const Unit un = units[x];
          const uint32_t row = (p.per_layer ? (uint32_t)un.h * (uint32_t)Lq : 0u) + (uint32_t)(un.row0 + ((warp + 11 * lane) & 31));
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t word = ~(row * (uint32_t)Lk + (uint32_t)(un.kt * kTile + lane + 32 * e));
            if (my_keys[x * kUnitWords + 32 * e] == thr && (word & hi_mask) == pre)
              atomicAdd(&mine[(word >> shift) & dmask], 1u);
          }
        }
      }
    }
    if (!any) break;
    __syncthreads();
    // the histograms of selections that several CTAs share meet in global memory
    for (int q = 0; q < n_sel; ++q) {
      const int sharers = sels[q].sharers;
      if (!sels[q].going || sharers == 1) continue;
      uint32_t *all = hist + ((size_t)(sel0 + q) * kHistBuffers + digit % kHistBuffers) * kBins;
      for (int b = t; b < kBins; b += kHeldThreads)
        if (counts_s[q * kBins + b]) atomicAdd(all + b, counts_s[q * kBins + b]);
      if (digit >= 2) {  // the buffer of two digits ago has been read by all: ready for the next digit but ...
        uint32_t *old = hist + ((size_t)(sel0 + q) * kHistBuffers + (digit - 2) % kHistBuffers) * kBins;
        for (int b = sels[q].rank * kHeldThreads + t; b < kBins; b += sharers * kHeldThreads) old[b] = 0u;
      }
    }
    __syncthreads();
    if (t == 0) {
      __threadfence();
      for (int q = 0; q < n_sel; ++q)
        if (sels[q].going && sels[q].sharers > 1) atomicAdd(&state[sel0 + q].barrier, 1u);
    }
    if (digit == 0 && p.causal) clear_outside();
    if (t == 0) {
      bool ok = true;
      for (int q = 0; q < n_sel; ++q)
        if (sels[q].going && sels[q].sharers > 1)
          ok = ok && reached(&state[sel0 + q].barrier, (uint32_t)sels[q].sharers * (uint32_t)(digit + 1));
      __threadfence();
      ok_s = ok;
      if (!ok) atomicOr(err, kDevErrTimeout);
    }
    __syncthreads();
    if (!ok_s) return;
    for (int q = 0; q < n_sel; ++q) {
      if (!sels[q].going) continue;
      const unsigned long long rest = sels[q].rest;
      // thread t owns bins 2047 - 2t and 2046 - 2t (descending); the owner of the wanted rank picks the digit
      uint2 c;
      if (sels[q].sharers > 1) {
        const uint32_t *all = hist + ((size_t)(sel0 + q) * kHistBuffers + digit % kHistBuffers) * kBins;
        c = __ldcg(reinterpret_cast<const uint2 *>(all) + (kBins / 2 - 1 - t));
      } else {
        c = reinterpret_cast<const uint2 *>(counts_s + q * kBins)[kBins / 2 - 1 - t];
      }
      const uint32_t sum = c.x + c.y;
      uint32_t incl = sum;  // (fewer than 2^32 entries: at most kHeldUnits units per SM)
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) warp_sums[warp] = incl;
      __syncthreads();
      const unsigned long long before = incl - sum + __reduce_add_sync(0xffffffffu, lane < warp ? warp_sums[lane] : 0u);
      if (before < rest && before + sum >= rest) {  // exactly one thread
        Sel &st = sels[q];
        const bool first = before + c.y >= rest;
        const uint32_t bin = (uint32_t)(kBins - 1 - 2 * t - (first ? 0 : 1)), count = first ? c.y : c.x;
        const uint32_t prefix = st.prefix | bin << shift;
        st.rest = rest - before - (first ? 0u : c.y);
        st.prefix = digit == kPasses - 1 ? 0u : prefix;
        if (digit == kPasses - 1) {
          st.thr = prefix;
          if (keep_ties || st.rest == count) st.going = 0;  // every entry equal to the threshold is kept
        } else if (digit == 2 * kPasses - 1) {
          st.tie_cut = ~prefix;
        }
      }
      __syncthreads();
    }
  }
  // ---- mask and bitmaps
#pragma unroll 2
  for (int x = 0; x < n_units; ++x) {
    const Unit un = units[x];
    const int q = p.sel_of(u0 + x) - sel0;
    const uint32_t thr = sels[q].thr;
    const int i = un.row0 + warp, j = un.kt * kTile + 4 * lane;
    const uint4 k = reinterpret_cast<const uint4 *>(keys_s + x * kUnitWords)[t];
    uint32_t kept = (k.x >= thr ? 1u : 0u) | (k.y >= thr ? 2u : 0u) | (k.z >= thr ? 4u : 0u) | (k.w >= thr ? 8u : 0u);
    if (sels[q].tie_cut != 0xffffffffu) {  // entries equal to the threshold are kept up to the last kept one only
      const uint32_t cut = sels[q].tie_cut;
      const uint32_t ties = (k.x == thr ? 1u : 0u) | (k.y == thr ? 2u : 0u) | (k.z == thr ? 4u : 0u) | (k.w == thr ? 8u : 0u);
      const uint32_t first = ((p.per_layer ? (uint32_t)un.h * (uint32_t)Lq : 0u) + (uint32_t)i) * (uint32_t)Lk + (uint32_t)j;
      if (first > cut)
        kept &= ~ties;
      else if (cut - first < 3u)
        kept &= ~(ties & ~((2u << (cut - first)) - 1u));
    }
    if (diag && i < Lq && (unsigned)(i + off - j) < 4u) kept |= 1u << (i + off - j);
    if (mask && i < Lq) {
      uint8_t *m = mask + ((size_t)un.h * Lq + i) * Lk + j;
      if (mask4) {  // four bits to four bytes: the products of the shifted copies do not meet
        if (j < Lk) *reinterpret_cast<uint32_t *>(m) = (kept * 0x00204081u) & 0x01010101u;
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (j + c < Lk) m[c] = (kept >> c) & 1u;
      }
    }
    const int count = __reduce_add_sync(0xffffffffu, __popc(kept));
    if (stage_bitmap) {  // eight lanes make a word
      uint32_t w = kept << (4 * (lane & 7));
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, o);
      const int r = un.row0 % kTile + warp;
      if ((lane & 7) == 0) stage_bitmap[(size_t)un.tile * kBitmapWords + 4 * r + (lane >> 3)] = w;
      const uint32_t vote = __ballot_sync(0xffffffffu, kept != 0u);
      if (lane == 0 && vote) atomicOr(&unit_votes[x], vote);
    }
    if (lane == 0 && count) atomicAdd(&unit_count[x], count);
  }
  __syncthreads();
  if (t < n_units && unit_count[t]) {
    const Unit un = units[t];
    if (stage_count) {
      atomicAdd(stage_count + un.tile, unit_count[t]);
      uint32_t groups = 0u;  // a group is four lanes
#pragma unroll
      for (int g = 0; g < 8; ++g) groups |= ((unit_votes[t] >> (4 * g)) & 15u ? 1u : 0u) << g;
      atomicOr(stage_groups + un.tile, groups);
    }
    if (nnz && (p.per_layer || keep_ties))
      atomicAdd(reinterpret_cast<unsigned long long *>(nnz + un.h), (unsigned long long)unit_count[t]);
  }
}

// Where the arrays of the select scratch lie.  The header and the states (and the histograms, where the select shares
// them between CTAs) are zeroed before the first kernel of a call.
struct Header {
  uint32_t compact_barrier;
  uint32_t pad[15];
};

Scratch carve(void *scratch, int H, Header **header) {
  char *p = static_cast<char *>(scratch);
  Scratch s;
  *header = reinterpret_cast<Header *>(p);
  p += sizeof(Header);
  s.state = reinterpret_cast<SelectState *>(p);
  p += (size_t)H * sizeof(SelectState);
  p = reinterpret_cast<char *>(align256(reinterpret_cast<size_t>(p)));
  s.hist = reinterpret_cast<uint32_t *>(p);
  p += (size_t)min(H, kMaxSharedSelections) * kHistBuffers * kBins * sizeof(uint32_t);
  s.cand = reinterpret_cast<uint2 *>(p);
  return s;
}

}  // namespace

size_t select_scratch_bytes(int H, int Lq, int Lk) {
  // the candidate buffer is sized for the larger of the causal and the full domain, and for one
  // selection over all heads (never smaller than H selections of one head each)
  return align256(sizeof(Header) + (size_t)H * sizeof(SelectState)) + 256 +
         (size_t)min(H, kMaxSharedSelections) * kHistBuffers * kBins * sizeof(uint32_t) +
         align256((size_t)cand_capacity((long long)H * Lq * Lk) * sizeof(uint2));
}

cudaError_t launch_build_mask(const BuildMaskArgs &a, cudaStream_t s) {
  const int n_qt = ceil_div(a.Lq, kTile), n_kt = ceil_div(a.Lk, kTile), n_tiles = a.H * n_qt * n_kt;
  const int diag = (a.keep_diag && (a.Lq == a.Lk || a.causal)) ? 1 : 0;
  const int sms = sm_count();
  unsigned *err = device_error_word();
  if (sms <= 0 || !err) return cudaErrorUnknown;
  Header *header;
  Scratch sc = carve(a.scratch, a.H, &header);
  // the selections: one per head over Lq rows, or one over the H*Lq rows of the layer
  const int n_sel = a.per_layer ? 1 : a.H;
  // per head nnz = k; per layer, or with all ties kept, it is counted
  const bool count_nnz = a.per_layer || a.keep_ties;
  // What fits into the shared memory of the SMs is read once and held there.
  Held held = {a.H, a.Lq, a.Lk, n_qt, n_kt, a.causal, a.per_layer, 4 * (int)dense_row_start(n_qt, n_kt, a.Lq, a.Lk, a.causal)};
  if ((long long)a.H * held.per_head <= (long long)kHeldUnits * sms && n_sel <= kMaxSharedSelections && a.k_rest > 0) {
    cudaError_t e = launch_clear(header, (reinterpret_cast<char *>(sc.hist) - reinterpret_cast<char *>(header)) +
                                                   (size_t)n_sel * kHistBuffers * kBins * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    const int grid = held.total() < sms ? held.total() : sms;
    int diag_arg = diag, keep_ties = a.keep_ties;
    auto smem_of = [](int units) { return (kHeldSels * kBins + units * kUnitWords) * sizeof(uint32_t); };
    e = cudaFuncSetAttribute(held_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(kHeldUnits));
    if (e != cudaSuccess) return e;
    const size_t smem = smem_of(ceil_div(held.total(), grid));
    unsigned long long k_rest = (unsigned long long)a.k_rest;
    long long nnz_init = count_nnz ? 0ll : (long long)a.k;
    const float *acc = a.acc;
    int64_t *nnz = a.nnz;
    uint8_t *mask = a.mask;
    uint32_t *stage_bitmap = a.stage_bitmap, *stage_groups = a.stage_groups;
    int32_t *stage_count = a.stage_count;
    void *args[] = {&acc, &held, &diag_arg, &k_rest, &sc.state, &sc.hist, &keep_ties, &nnz_init, &nnz, &mask, &stage_bitmap,
                    &stage_count, &stage_groups, &err};
    e = launch_early_cooperative(reinterpret_cast<const void *>(held_kernel), grid, kHeldThreads, args, smem, s);
    if (e != cudaSuccess) return e;
    if (!a.tiles) return cudaSuccess;
    return launch_compact_staged(a.stage_bitmap, a.stage_count, a.stage_groups, *a.tiles, reinterpret_cast<int2 *>(sc.hist),
                                 (size_t)kHistBuffers * kBins * sizeof(uint32_t) / sizeof(int2), &header->compact_barrier, s);
  }
  const int rows = a.per_layer ? a.H * a.Lq : a.Lq;
  const int period = a.Lq;
  // CTAs per selection: all that fit, as far as there is a row for each of their warps
  const int max_ctas = kSelCtasPerSm * sms;
  int per_sel = max_ctas / n_sel;
  const long long pieces = (long long)rows * n_kt;
  if ((long long)per_sel * (kSelThreads / 32) > pieces) per_sel = (int)((pieces + kSelThreads / 32 - 1) / (kSelThreads / 32));
  if (per_sel < 1 || n_sel > kMaxSharedSelections) per_sel = 1;
  const size_t hist_bytes = per_sel > 1 ? (size_t)n_sel * kHistBuffers * kBins * sizeof(uint32_t) : 0;
  cudaError_t e = launch_clear(header, (reinterpret_cast<char *>(sc.hist) - reinterpret_cast<char *>(header)) + hist_bytes, s);
  if (e != cudaSuccess) return e;
  const long long n_valid = domain_size(a.Lq, a.Lk, a.causal);
  const long long n_rest = (n_valid - (diag ? a.Lq : 0)) * (a.per_layer ? a.H : 1);
  const long long cap = cand_capacity(n_rest);
  const bool shortcut = a.k_rest > 0 && cap > 0 && n_valid * a.H > kDirectEntries;
  // Exact per-head selections: the one pass over the accumulator also writes what is certain of the
  // mask and the tile bitmaps (the select adds the collected entries that are kept), so
  // the emit pass at the end has nothing to read for the selections the shortcut resolves.  Other
  // selections count what they keep in the emit pass, which therefore has to see every entry.
  const bool classify = shortcut && !a.per_layer && !a.keep_ties;
  if (shortcut) {
    const size_t smem = (kSamples + kBins) * sizeof(uint32_t);
    e = cudaFuncSetAttribute(sample_pivots_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    e = launch_early(sample_pivots_kernel, (unsigned)(n_sel * kSampleCtas), 1024, smem, s, a.acc, rows, a.Lk, period, a.causal,
                     diag, (unsigned long long)a.k_rest, (unsigned long long)n_rest, sc.state);
    if (e != cudaSuccess) return e;
    if (classify) {
      e = launch_early(emit_kernel<true, 4>, (unsigned)n_tiles, 128, 0, s, a.acc, a.Lq, a.Lk, n_qt, n_kt, n_tiles, a.causal, diag,
                       0, 0, sc.state, a.mask, a.stage_bitmap, a.stage_count, a.stage_groups, a.nnz, sc.cand, (uint32_t)cap);
    } else {
      // one wave of CTAs (five fit an SM), so that no SM idles while a second, partial wave runs
      int collect_blocks = ceil_div(rows, kWarps);
      if (collect_blocks > sms * 5 / n_sel) collect_blocks = max(sms * 5 / n_sel, 1);
      collect_kernel<<<dim3(collect_blocks, n_sel), kThreads, 0, s>>>(a.acc, rows, a.Lk, period, a.causal, diag, sc.state,
                                                                     sc.cand, (uint32_t)cap);
      e = launched(cudaGetLastError());
    }
    if (e != cudaSuccess) return e;
  }
  {
    const int grid = per_sel > 1 ? n_sel * per_sel : n_sel < max_ctas ? n_sel : max_ctas;
    unsigned long long k_rest = (unsigned long long)a.k_rest;
    long long nnz_init = count_nnz ? 0ll : (long long)a.k;
    int classified = classify ? 1 : 0, n_sel_arg = n_sel, rows_arg = rows, period_arg = period, per_sel_arg = per_sel;
    int diag_arg = diag, n_qt_arg = n_qt, n_kt_arg = n_kt, Lk = a.Lk, Lq = a.Lq, H = a.H, causal = a.causal;
    int keep_ties = a.keep_ties;
    uint32_t cap_arg = shortcut ? (uint32_t)cap : 0u;
    const float *acc = a.acc;
    const uint2 *cand = sc.cand;
    int64_t *nnz = a.nnz;
    uint8_t *mask = a.mask;
    uint32_t *stage_bitmap = a.stage_bitmap, *stage_groups = a.stage_groups;
    int32_t *stage_count = a.stage_count;
    void *args[] = {&acc, &rows_arg, &Lk, &period_arg, &causal, &diag_arg, &k_rest, &n_sel_arg, &per_sel_arg, &sc.state,
                    &sc.hist, &cand, &cap_arg, &keep_ties, &H, &nnz_init, &nnz, &classified, &Lq, &n_qt_arg, &n_kt_arg,
                    &mask, &stage_bitmap, &stage_count, &stage_groups, &err};
    e = launch_early_cooperative(reinterpret_cast<const void *>(shortcut ? select_kernel<true> : select_kernel<false>), grid,
                                 kSelThreads, args, 0, s);
    if (e != cudaSuccess) return e;
  }
  // Few tiles: sixteen warps each, so that a tile's rows are all in flight at once.  With the mask written by then (the
  // usual end of a classified selection) the launch only has to look.
  if (n_tiles <= 4 * sms) {
    e = launch_early(emit_kernel<false, 16>, (unsigned)n_tiles, 512, 0, s, a.acc, a.Lq, a.Lk, n_qt, n_kt, n_tiles, a.causal, diag,
                     a.per_layer, a.keep_ties, sc.state, a.mask, a.stage_bitmap, a.stage_count, a.stage_groups, a.nnz, nullptr, 0u);
  } else {
    const int most = (classify ? 2 : 16) * sms;
    e = launch_early(emit_kernel<false, 4>, (unsigned)(n_tiles < most ? n_tiles : most), 128, 0, s, a.acc, a.Lq, a.Lk, n_qt, n_kt,
                     n_tiles, a.causal, diag, a.per_layer, a.keep_ties, sc.state, a.mask, a.stage_bitmap, a.stage_count,
                     a.stage_groups, a.nnz, nullptr, 0u);
  }
  if (e != cudaSuccess || !a.tiles) return e;
  // the histograms are free by now: the compaction keeps its CTAs' totals there
  return launch_compact_staged(a.stage_bitmap, a.stage_count, a.stage_groups, *a.tiles, reinterpret_cast<int2 *>(sc.hist),
                               (size_t)kHistBuffers * kBins * sizeof(uint32_t) / sizeof(int2), &header->compact_barrier, s);
}

}  // namespace ap
