// Masked attention of Section 3.2 on CUDA cores (fp32 FMA), for fp32 tensors.
//
// fwd_simt_kernel: one CTA takes R query rows of one (b, h) through the keys that any of them keeps.  Planning: the R rows'
// words of the next two tiles' bitmaps, transposed by shuffles, give every key the rows that keep it; keys kept by none
// are left out, the others are appended to a list in shared memory.  Work: a batch of 64 or 128 listed keys at a time, whatever
// tiles they come from.  S = Q K^T with a register tile per thread, S to shared memory, a warp's share of the rows for maxima,
// weights and sums, O += P V with a register tile per thread and the batch's keys split over groups of threads (summed
// once, at the end).  K and V rows arrive by asynchronous 16-byte copies; the next batch's K is copied during the
// softmax and P V, this one's V during its S, and the next batch is planned meanwhile.  Pruned entries get weight exactly 0;
// rows that never see a kept entry output zeros.
//
// What bounds it: at small shapes the chain plan -> copy -> S -> softmax -> P V of one batch (a few microseconds), so R
// goes down to 8 until the SMs are covered; at large ones the products, at half of the FMA rate, and the reductions of
// the softmax.  Without the list, every key of a stored tile copied and multiplied: 32 x 16 heads x 512 x 64 causal 600 us at
// 5 % kept, 729 at 50 %, 737 unpruned (170, 452, 642 now); with two threads per query row that walked the kept keys one by
// one: 227, 792, 1069.
#include <math_constants.h>

#include <type_traits>

#include "ap_common.cuh"

namespace ap {

namespace {

constexpr int kEntmaxThreads = 256;

template <typename T>
__device__ __forceinline__ float4 load4(const T *p);
template <>
__device__ __forceinline__ float4 load4<float>(const float *p) {
  return *reinterpret_cast<const float4 *>(p);
}

template <typename T>
__device__ __forceinline__ void store4(T *p, float4 v);
template <>
__device__ __forceinline__ void store4<float>(float *p, float4 v) {
  *reinterpret_cast<float4 *>(p) = v;
}

// 16 bytes global -> shared memory, asynchronously; zeros where `valid` is false (nothing is read then).
__device__ __forceinline__ void copy16(float *dst, const float *src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Rows of D floats in shared memory, 16-byte chunk c of row r at chunk c ^ (r mod 8): the eight lanes of
// a 16-byte access phase read the same chunk of eight consecutive rows without a bank conflict.
template <int D>
__device__ __forceinline__ float4 *chunk_at(float *base, int r, int c) {
  return reinterpret_cast<float4 *>(base + r * D) + (c ^ (r & 7));
}

// N values per lane, each combined over the 32 lanes by op: every lane gets the result of value lane / (32 / N).  (One by one they
// would take 5 N exchanges, this way N - 1 + log2(32 / N).)
template <int N, class Op>
__device__ __forceinline__ float reduce_rows(float (&v)[N], int lane, Op op) {
#pragma unroll
  for (int n = N, o = 16; o > 0; o >>= 1) {
    if (n > 1) {
      n >>= 1;
#pragma unroll
      for (int x = 0; x < N / 2; ++x)
        if (x < n) {
          const bool upper = (lane & o) != 0;
          const float there = __shfl_xor_sync(0xffffffffu, upper ? v[x] : v[x + n], o);
          v[x] = op(upper ? v[x + n] : v[x], there);
        }
    } else {
      v[0] = op(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
    }
  }
  return v[0];
}

template <class T, int N>
struct alignas(sizeof(T) * N) Run {
  T v[N];
};

template <int D, int R>
struct SimtCfg {
  // Four CTAs of four warps with 64 keys at a time fill an SM better than two of eight with 128, but d = 128 has no registers
  // for that and eight rows (a grid that does not fill the GPU) are done sooner by eight warps: 8 x 12 heads x 512 x 64, 5 and
  // 50 % kept, 63 and 257 us with eight warps and 128 keys, 47 and 263 with 64 keys, 45 and 250 with four warps (before the
  // reductions over rows were combined: 41 and 224 now).
  static constexpr int kThreads = D == 64 && R > 8 ? 128 : 256, kWarps = kThreads / 32;
  static constexpr int kBatch = D == 64 && R == 8 ? 128 : 64;  // keys worked on at a time
  static constexpr int kCtas = D == 64 && R > 8 ? 4 : 2;       // per SM
  // S: a warp computes (4 RT) x (8 KT) of the R x kBatch scores, lane = 4 row lanes x 8 key lanes
  static constexpr int RT = R == 32 ? 4 : 2;
  static constexpr int KT = (R / (4 * RT)) * (kBatch / 8) / kWarps;
  static_assert((R / (4 * RT)) * (kBatch / (8 * KT)) == kWarps, "the warps cover S");
  static constexpr int kMyKeys = kBatch / 32;  // softmax: consecutive keys of a lane
  // P V: a thread owns PR rows x 4 columns; D/4 column lanes, R/PR row groups, the rest splits the keys
  static constexpr int PR = R == 32 ? 4 : 2;
  static constexpr int kSplit = kThreads / ((D / 4) * (R / PR));
  static_assert(kSplit >= 1 && kBatch % (4 * kSplit) == 0, "keys split evenly");
  static constexpr int kPitch = kBatch + 4;  // floats per row of S
  // a planning step adds up to 256 keys to at most 2 kBatch - 1
  static constexpr int kList = 512;
  static_assert(2 * kBatch - 1 + 256 <= kList && kList % kBatch == 0, "the list holds what is planned ahead");
  static constexpr int kKOff = R * D, kVOff = kKOff + kBatch * D, kSOff = kVOff + kBatch * D,
                       kAlphaOff = kSOff + R * kPitch, kListOff = kAlphaOff + 2 * R, kFloats = kListOff + 2 * kList;
  static_assert(kSplit * R * D <= 2 * kBatch * D, "the partial outputs fit over K and V");
};

template <int D, int R>
__global__ void __launch_bounds__((SimtCfg<D, R>::kThreads), (SimtCfg<D, R>::kCtas))
fwd_simt_kernel(const float *Q, const float *K, const float *V,
                const int32_t *row_ptr, const int32_t *col_idx,
                const uint8_t *flags, const uint32_t *bitmap, float *__restrict__ O, int H,
                int Lq, int Lk, int n_qt, int n_rt, float scale) {
  using C = SimtCfg<D, R>;
  constexpr int kThreads = C::kThreads;
  constexpr int CH = D / 4;  // 16-byte chunks per row
  extern __shared__ __align__(16) float smem[];
  __shared__ int counts[2][8];
  float *q_s = smem, *k_s = smem + C::kKOff, *v_s = smem + C::kVOff, *s_s = smem + C::kSOff,
        *alpha_s = smem + C::kAlphaOff, *l_s = alpha_s + R;
  // the kept keys of these rows in list order: the key, and a bit for each row that keeps it
  uint32_t *list_key = reinterpret_cast<uint32_t *>(smem + C::kListOff), *list_rows = list_key + C::kList;
  const int rt = blockIdx.x % n_rt;
  const size_t bh = blockIdx.x / n_rt;
  const int i0 = rt * R, qt = i0 / kTile, h = (int)(bh % H);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  after_previous();
  const int t_begin = row_ptr[h * n_qt + qt], t_end = row_ptr[h * n_qt + qt + 1];

  for (int e = threadIdx.x; e < R * CH; e += kThreads) {
    const int r = e / CH, c = e % CH, i = i0 + r;
    const bool valid = i < Lq;
    copy16(reinterpret_cast<float *>(chunk_at<D>(q_s, r, c)), Q + (bh * Lq + (valid ? i : 0)) * D + 4 * c, valid);
  }
  // scores: this thread's rows sr + 4 x and keys sk + 8 y
  constexpr int kKeyWarps = C::kBatch / (8 * C::KT);
  const int s_key0 = (warp % kKeyWarps) * 8 * C::KT;  // first key of the warp
  const int sr = (warp / kKeyWarps) * 4 * C::RT + (lane >> 3), sk = s_key0 + (lane & 7);
  constexpr int kMyRows = R / C::kWarps, kRowLanes = 32 / kMyRows;  // softmax: rows of a warp
  // P V: column chunk pc, rows pr .. pr + PR - 1, keys of split part ps
  const int pc = threadIdx.x % CH, pr = (threadIdx.x / CH) % (R / C::PR) * C::PR, ps = threadIdx.x / (CH * (R / C::PR));

  // A pruned entry's weight is -0 (a kept one's that underflows is +0).  Where V holds infinities or NaNs, its product is
  // not zero: a CTA that finds a NaN among its outputs works them out once more with `careful`, which leaves the products
  // of pruned entries out.
  bool careful = false;
#pragma unroll 1
  while (true) {
    // Planning: two tiles a step, a warp a 32-column word of one of them (or of both), lane = row; transposed, lane = column.
    constexpr int kWords = 256 / kThreads;  // per warp
    int t_plan = t_begin, tail = 0, step = 0, ahead_kt[kWords];
    uint32_t ahead_word[kWords];
    auto look_ahead = [&]() {  // (raw loads, used a step later)
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        const int t = t_plan + (warp >> 2) + u;
        ahead_word[u] = 0u;
        ahead_kt[u] = 0;
        if (t < t_end) {
          ahead_kt[u] = col_idx[t];
          const bool full = flags[t] & 1;
          if (lane < R)
            ahead_word[u] = full ? 0xffffffffu : bitmap[(size_t)t * kBitmapWords + 4 * ((i0 & (kTile - 1)) + lane) + (warp & 3)];
        }
      }
    };
    auto plan = [&]() {
      uint32_t key[kWords], rows[kWords], vote[kWords];
      int *n = counts[step++ & 1];
#pragma unroll
      for (int u = 0; u < kWords; ++u) {
        rows[u] = transpose32(ahead_word[u], lane);
        key[u] = (uint32_t)(ahead_kt[u] * kTile + 32 * (warp & 3) + lane);
        vote[u] = __ballot_sync(0xffffffffu, rows[u] != 0u);
        if (lane == 0) n[warp + 4 * u] = __popc(vote[u]);
      }
      t_plan += 2;
      look_ahead();
      __syncthreads();
      int before[kWords] = {}, all = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) {
#pragma unroll
        for (int u = 0; u < kWords; ++u) before[u] += w < warp + 4 * u ? n[w] : 0;
        all += n[w];
      }
#pragma unroll
      for (int u = 0; u < kWords; ++u)
        if (rows[u] != 0u) {
          const int at = (tail + before[u] + __popc(vote[u] & ((1u << lane) - 1u))) & (C::kList - 1);
          list_key[at] = key[u];
          list_rows[at] = rows[u];
        }
      tail += all;
    };
    look_ahead();
    // Rows of `src` that belong to the n keys from list position `first` on; rows [n, n_zero) become zeros.
    auto copy_rows = [&](float *dst, const float *src, int first, int n, int n_zero) {
      const int c = threadIdx.x % CH, j0 = threadIdx.x / CH;
      const float *from = src + bh * Lk * D + 4 * c;
      constexpr int kStep = kThreads / CH;
      if (n == C::kBatch) {
        const uint32_t *keys = list_key + (first & (C::kList - 1)) + j0;
#pragma unroll
        for (int x = 0; x < C::kBatch / kStep; ++x)
          copy16(reinterpret_cast<float *>(chunk_at<D>(dst, j0 + x * kStep, c)), from + (size_t)keys[x * kStep] * D, true);
      } else {
        for (int jj = j0; jj < n_zero; jj += kStep) {
          const bool valid = jj < n;
          const size_t j = valid ? list_key[(first + jj) & (C::kList - 1)] : 0u;
          copy16(reinterpret_cast<float *>(chunk_at<D>(dst, jj, c)), from + j * D, valid);
        }
      }
    };
    while (tail < C::kBatch && t_plan < t_end) plan();
    __syncthreads();
    int head = 0, nb = min(C::kBatch, tail);
    copy_rows(k_s, K, 0, nb, nb);
    copy_commit();

    float m = -CUDART_INF_F, l = 0.f;  // of row lane / kRowLanes of the warp's
    float4 o[C::PR];
#pragma unroll
    for (int x = 0; x < C::PR; ++x) o[x] = make_float4(0.f, 0.f, 0.f, 0.f);

#pragma unroll 1
    while (nb > 0) {
      const int part = (nb + 4 * C::kSplit - 1) / (4 * C::kSplit) * 4;  // keys of a split part of P V
      copy_rows(v_s, V, head, nb, part * C::kSplit);  // (every thread is past the last P V, see the barrier at the loop's end)
      copy_commit();
      while (tail - head - nb < C::kBatch && t_plan < t_end) plan();  // the next batch
      copy_wait<1>();  // K of this batch (and Q)
      __syncthreads();
      if (s_key0 < nb) {
        float s[C::RT][C::KT];
#pragma unroll
        for (int x = 0; x < C::RT; ++x)
#pragma unroll
          for (int y = 0; y < C::KT; ++y) s[x][y] = 0.f;
#pragma unroll 4
        for (int c = 0; c < CH; ++c) {
          float4 qv[C::RT], kv[C::KT];
#pragma unroll
          for (int x = 0; x < C::RT; ++x) qv[x] = *chunk_at<D>(q_s, sr + 4 * x, c);
#pragma unroll
          for (int y = 0; y < C::KT; ++y) kv[y] = *chunk_at<D>(k_s, sk + 8 * y, c);
#pragma unroll
          for (int x = 0; x < C::RT; ++x)
#pragma unroll
            for (int y = 0; y < C::KT; ++y) {
              s[x][y] = fmaf(qv[x].x, kv[y].x, s[x][y]);
              s[x][y] = fmaf(qv[x].y, kv[y].y, s[x][y]);
              s[x][y] = fmaf(qv[x].z, kv[y].z, s[x][y]);
              s[x][y] = fmaf(qv[x].w, kv[y].w, s[x][y]);
            }
        }
#pragma unroll
        for (int x = 0; x < C::RT; ++x)
#pragma unroll
          for (int y = 0; y < C::KT; ++y) s_s[(sr + 4 * x) * C::kPitch + sk + 8 * y] = s[x][y] * scale;
      }
      __syncthreads();
      const int n_next = min(C::kBatch, tail - head - nb);
      copy_rows(k_s, K, head + nb, n_next, n_next);
      copy_commit();
      using Rows = Run<uint32_t, C::kMyKeys>;
      using Keys = Run<float, C::kMyKeys>;
      const int my_key = C::kMyKeys * lane;  // (batches start at multiples of their size)
      Rows rows = *reinterpret_cast<const Rows *>(list_rows + (head & (C::kList - 1)) + my_key);
#pragma unroll
      for (int y = 0; y < C::kMyKeys; ++y) rows.v[y] = my_key + y < nb ? rows.v[y] : 0u;
      float *my_s = s_s + warp * kMyRows * C::kPitch + my_key;
      Keys w[kMyRows];
      float top[kMyRows], sum[kMyRows];
#pragma unroll
      for (int x = 0; x < kMyRows; ++x) {
        w[x] = *reinterpret_cast<const Keys *>(my_s + x * C::kPitch);
        top[x] = -CUDART_INF_F;
#pragma unroll
        for (int y = 0; y < C::kMyKeys; ++y) {
          w[x].v[y] = (rows.v[y] >> (warp * kMyRows + x)) & 1u ? w[x].v[y] : -CUDART_INF_F;
          top[x] = fmaxf(top[x], w[x].v[y]);
        }
      }
      const float m_new = fmaxf(m, reduce_rows<kMyRows>(top, lane, [](float a, float b) { return fmaxf(a, b); }));
      const float ref = m_new == -CUDART_INF_F ? 0.f : m_new;
      const float alpha = expf(m - ref);  // exp(-inf) = 0 before the row's first kept entry
      m = m_new;
#pragma unroll
      for (int x = 0; x < kMyRows; ++x) {
        const float ref_x = __shfl_sync(0xffffffffu, ref, x * kRowLanes);
        sum[x] = 0.f;
#pragma unroll
        for (int y = 0; y < C::kMyKeys; ++y) {
          w[x].v[y] = (rows.v[y] >> (warp * kMyRows + x)) & 1u ? expf(w[x].v[y] - ref_x) : -0.f;
          sum[x] += w[x].v[y];
        }
        *reinterpret_cast<Keys *>(my_s + x * C::kPitch) = w[x];
      }
      l = l * alpha + reduce_rows<kMyRows>(sum, lane, [](float a, float b) { return a + b; });
      if (lane % kRowLanes == 0) alpha_s[warp * kMyRows + lane / kRowLanes] = alpha;
      copy_wait<1>();  // V of this batch
      __syncthreads();
#pragma unroll
      for (int x = 0; x < C::PR; ++x) {
        const float alpha = alpha_s[pr + x];
        o[x].x *= alpha, o[x].y *= alpha, o[x].z *= alpha, o[x].w *= alpha;
      }
      auto add = [&](auto with_care, int from, int n) {
#pragma unroll 2
        for (int j = from; j < from + n; j += 4) {
          float4 p[C::PR];
#pragma unroll
          for (int x = 0; x < C::PR; ++x) p[x] = *reinterpret_cast<const float4 *>(s_s + (pr + x) * C::kPitch + j);
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            const float4 v = *chunk_at<D>(v_s, j + y, pc);
#pragma unroll
            for (int x = 0; x < C::PR; ++x) {
              const float w = y == 0 ? p[x].x : y == 1 ? p[x].y : y == 2 ? p[x].z : p[x].w;
              if (decltype(with_care)::value && signbit(w)) continue;
              o[x].x = fmaf(w, v.x, o[x].x), o[x].y = fmaf(w, v.y, o[x].y);
              o[x].z = fmaf(w, v.z, o[x].z), o[x].w = fmaf(w, v.w, o[x].w);
            }
          }
        }
      };
      constexpr int kPart = C::kBatch / C::kSplit;
      if (careful)
        add(std::true_type{}, ps * part, part);
      else if (nb == C::kBatch)
        add(std::false_type{}, ps * kPart, kPart);
      else
        add(std::false_type{}, ps * part, part);
      __syncthreads();  // S, alpha, V and this batch's place in the list are read
      head += nb;
      nb = n_next;
    }
    // sums of the key parts (over K and V), then the division by l
    copy_wait<0>();
    float *part = k_s;
#pragma unroll
    for (int x = 0; x < C::PR; ++x)
      *reinterpret_cast<float4 *>(part + ((ps * R) + pr + x) * D + 4 * pc) = o[x];
    if (lane % kRowLanes == 0) l_s[warp * kMyRows + lane / kRowLanes] = l;
    __syncthreads();
    bool nan = false;
    for (int e = threadIdx.x; e < R * CH; e += kThreads) {
      const int r = e / CH, c = e % CH;
      if (i0 + r >= Lq) continue;
      float4 sum = *reinterpret_cast<const float4 *>(part + r * D + 4 * c);
#pragma unroll
      for (int y = 1; y < C::kSplit; ++y) {
        const float4 v = *reinterpret_cast<const float4 *>(part + (y * R + r) * D + 4 * c);
        sum.x += v.x, sum.y += v.y, sum.z += v.z, sum.w += v.w;
      }
      const float lr = l_s[r];
      float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
      if (lr > 0.f) out = make_float4(sum.x / lr, sum.y / lr, sum.z / lr, sum.w / lr);
      nan = nan || out.x != out.x || out.y != out.y || out.z != out.z || out.w != out.w;
      *reinterpret_cast<float4 *>(O + (bh * Lq + i0 + r) * D + 4 * c) = out;
    }
    if (careful || !__syncthreads_or(nan ? 1 : 0)) break;
    careful = true;
  }
}

// The same attention with 1.5-entmax as the normaliser (the section on sparse normalisation):
// p_j = max(s_j / 2 - tau, 0)^2 over the kept keys, tau such that the row sums to 1.  tau depends
// on all kept scores of a row, so the CTA walks its tiles once per sweep: row maxima first
// (tau = max/2 - 0.625; the root lies in [max/2 - 1, max/2)), then sweeps that collect the size n of the support of the
// trial threshold and its sums S1, S2 of (s_j/2 - tau) and of its square and move tau to the smaller
// root of the support's parabola, tau + (S2 - 1) / (S1 + sqrt(S1^2 - n (S2 - 1))) (Newton's step
// (S2 - 1) / (2 S1) where it has none), until no row of the CTA moves by more than
// 5e-7 max(1, |tau|) (at most 30 sweeps), then the sweep that forms the weights and adds p V.
// Both threads of a row see the same scores and keep the same statistics.
template <typename T, int D>
__global__ void __launch_bounds__(kEntmaxThreads) fwd_entmax_simt_kernel(const T *Q, const T *K,
                                                                   const T *V,
                                                                   const int32_t *row_ptr,
                                                                   const int32_t *col_idx,
                                                                   const uint8_t *flags,
                                                                   const uint32_t *bitmap,
                                                                   T *__restrict__ O, int H, int Lq, int Lk, int n_qt,
                                                                   float half_scale) {
  constexpr int G = D / 8;
  extern __shared__ __align__(16) float smem[];
  float *k_s = smem;               // [128][D]
  float *v_s = smem + kTile * D;   // [128][D]
  const int qt = blockIdx.x % n_qt;
  const int h = (blockIdx.x / n_qt) % H;
  const int b = blockIdx.x / (n_qt * H);
  const int r = threadIdx.x >> 1, half = threadIdx.x & 1;
  const int i = qt * kTile + r;
  const size_t bh = (size_t)b * H + h;

  after_previous();
  float4 q[G], o[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    o[g] = make_float4(0.f, 0.f, 0.f, 0.f);
    q[g] = i < Lq ? load4<T>(Q + (bh * Lq + i) * D + 4 * (2 * g + half)) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float m = -CUDART_INF_F, tau = 0.f, l = 0.f;
  const int t_begin = row_ptr[h * n_qt + qt], t_end = row_ptr[h * n_qt + qt + 1];
  int kind = 0;  // 0 maxima, 1 sums over the support, 2 weights
  for (int sw = 0;; ++sw) {
    float n = 0.f, S1 = 0.f, S2 = 0.f;
    for (int t = t_begin; t < t_end; ++t) {
      const int kt = col_idx[t];
      __syncthreads();  // previous tile fully consumed
      for (int e = threadIdx.x; e < kTile * D / 4; e += kEntmaxThreads) {
        const int jj = e / (D / 4), c = e % (D / 4);
        const int j = kt * kTile + jj;
        float4 kv = make_float4(0.f, 0.f, 0.f, 0.f), vv = kv;
        if (j < Lk) {
          kv = load4<T>(K + (bh * Lk + j) * D + 4 * c);
          if (kind == 2) vv = load4<T>(V + (bh * Lk + j) * D + 4 * c);
        }
        reinterpret_cast<float4 *>(k_s)[e] = kv;
        if (kind == 2) reinterpret_cast<float4 *>(v_s)[e] = vv;
      }
      const bool full = flags[t] & 1;
      const uint4 bw = reinterpret_cast<const uint4 *>(bitmap + (size_t)t * kBitmapWords)[r];
      const uint32_t words[4] = {bw.x, bw.y, bw.z, bw.w};
      __syncthreads();
#pragma unroll 1
      for (int w = 0; w < 4; ++w) {
        const uint32_t bits = full ? 0xffffffffu : words[w];
        if (!__any_sync(0xffffffffu, bits != 0u)) continue;
#pragma unroll 1
        for (int c = 0; c < 32; ++c) {
          const bool keep = (bits >> c) & 1u;
          if (!__any_sync(0xffffffffu, keep)) continue;
          const int jj = 32 * w + c;
          const float4 *krow = reinterpret_cast<const float4 *>(k_s + jj * D);
          float dot = 0.f;
#pragma unroll
          for (int g = 0; g < G; ++g) {
            const float4 kv = krow[2 * g + half];
            dot = fmaf(q[g].x, kv.x, dot); dot = fmaf(q[g].y, kv.y, dot);
            dot = fmaf(q[g].z, kv.z, dot); dot = fmaf(q[g].w, kv.w, dot);
          }
          dot += __shfl_xor_sync(0xffffffffu, dot, 1);
          if (!keep) continue;
          const float x = dot * half_scale;
          if (kind == 0) {
            m = fmaxf(m, x);
          } else {
            const float u = x - tau;
            if (u > 0.f) {
              if (kind == 1) {
                n += 1.f;
                S1 += u;
                S2 = fmaf(u, u, S2);
              } else {
                const float p = u * u;
                l += p;
                const float4 *vrow = reinterpret_cast<const float4 *>(v_s + jj * D);
#pragma unroll
                for (int g = 0; g < G; ++g) {
                  const float4 vv = vrow[2 * g + half];
                  o[g].x = fmaf(p, vv.x, o[g].x); o[g].y = fmaf(p, vv.y, o[g].y);
                  o[g].z = fmaf(p, vv.z, o[g].z); o[g].w = fmaf(p, vv.w, o[g].w);
                }
              }
            }
          }
        }
      }
    }
    if (kind == 2) break;
    bool moved = false;
    if (kind == 0) {
      // no kept key: every weight is 0 whatever the threshold
      tau = m == -CUDART_INF_F ? CUDART_INF_F : m - 0.625f;
    } else {
      const float disc = S1 * S1 - n * (S2 - 1.f);
      const float step = S1 > 0.f ? (S2 - 1.f) / (S1 + (disc >= 0.f ? sqrtf(disc) : S1)) : 0.f;
      tau += step;
      moved = i < Lq && fabsf(step) > 5e-7f * fmaxf(1.f, fabsf(tau));
    }
    const int more = __syncthreads_or(moved ? 1 : 0);
    kind = kind == 0 ? 1 : ((more && sw < 30) ? 1 : 2);
  }
  if (i < Lq) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
      if (l > 0.f) out = make_float4(o[g].x / l, o[g].y / l, o[g].z / l, o[g].w / l);
      store4<T>(O + (bh * Lq + i) * D + 4 * (2 * g + half), out);
    }
  }
}

template <typename T, int D>
cudaError_t launch_entmax(const void *Q, const void *K, const void *V, const ap_tiles &t, void *O, int B, int H, int Lq,
                          int Lk, float scale, cudaStream_t s) {
  const size_t smem = 2 * (size_t)kTile * D * sizeof(float);
  auto kern = fwd_entmax_simt_kernel<T, D>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = launch_early(kern, (unsigned)(B * H * t.n_qt), kEntmaxThreads, smem, s, static_cast<const T *>(Q), static_cast<const T *>(K),
                   static_cast<const T *>(V), t.row_ptr, t.col_idx, t.flags, t.bitmap, static_cast<T *>(O), H, Lq, Lk, t.n_qt,
                   0.5f * scale);
  return e;
}

template <int D, int R>
cudaError_t launch_rows(const void *Q, const void *K, const void *V, const ap_tiles &t, void *O, int B, int H, int Lq,
                        int Lk, float scale, cudaStream_t s) {
  constexpr size_t smem = SimtCfg<D, R>::kFloats * sizeof(float);
  auto kern = fwd_simt_kernel<D, R>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int n_rt = ceil_div(Lq, R);
  e = launch_early(kern, (unsigned)((int64_t)B * H * n_rt), SimtCfg<D, R>::kThreads, smem, s, static_cast<const float *>(Q),
                   static_cast<const float *>(K), static_cast<const float *>(V), t.row_ptr, t.col_idx, t.flags, t.bitmap,
                   static_cast<float *>(O), H, Lq, Lk, t.n_qt, n_rt, scale);
  return e;
}

// Query rows per CTA: the most (they share the K and V copies and the register tile grows) that still
// give every SM two CTAs.
template <int D>
cudaError_t launch(const void *Q, const void *K, const void *V, const ap_tiles &t, void *O, int B, int H, int Lq,
                   int Lk, float scale, cudaStream_t s) {
  const int64_t bh = (int64_t)B * H, want = 2 * (int64_t)sm_count();
  if (bh * ceil_div(Lq, 32) >= want) return launch_rows<D, 32>(Q, K, V, t, O, B, H, Lq, Lk, scale, s);
  if (bh * ceil_div(Lq, 16) >= want) return launch_rows<D, 16>(Q, K, V, t, O, B, H, Lq, Lk, scale, s);
  return launch_rows<D, 8>(Q, K, V, t, O, B, H, Lq, Lk, scale, s);
}

}  // namespace

cudaError_t launch_fwd_simt(const void *Q, const void *K, const void *V, const ap_tiles &t, void *O, int B, int H,
                            int Lq, int Lk, int d, float scale, cudaStream_t s) {
  return d == 64 ? launch<64>(Q, K, V, t, O, B, H, Lq, Lk, scale, s)
                 : launch<128>(Q, K, V, t, O, B, H, Lq, Lk, scale, s);
}

cudaError_t launch_fwd_entmax_simt(const void *Q, const void *K, const void *V, const ap_tiles &t, void *O, int B,
                                   int H, int Lq, int Lk, int d, float scale, cudaStream_t s) {
  return d == 64 ? launch_entmax<float, 64>(Q, K, V, t, O, B, H, Lq, Lk, scale, s)
                 : launch_entmax<float, 128>(Q, K, V, t, O, B, H, Lq, Lk, scale, s);
}

}  // namespace ap
