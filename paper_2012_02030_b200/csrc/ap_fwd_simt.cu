// Masked attention of Section 3.2 on CUDA cores (fp32 FMA), for fp32 tensors.
//
// fwd_simt_kernel: one CTA takes R query rows of one (b, h) through the stored tiles of their list row.
// Per tile: S = Q K^T with a register tile per thread, S (pruned entries -inf) to shared memory, a warp
// per row for maximum, weights and sum, O += P V with a register tile per thread and the tile's keys
// split over groups of threads (summed once, at the end).  K and V rows arrive by asynchronous 16-byte
// copies; the next tile's K is copied during the softmax and P V, its V during the next S.  Pruned entries
// get weight exactly 0; rows that never see a kept entry output zeros.
//
// What bounds it: at small shapes the chain copy -> S -> softmax -> P V of one tile (a few
// microseconds), so R goes down to 8 until the SMs are covered; at large ones shared-memory bandwidth
// (S: KT + RT 16-byte reads per 4 KT RT FMAs).  The version with two threads per query row that walked the
// kept keys one by one took 24 us where a toy model's 4 (head, sequence) pairs of 128 x 128 gave it 4
// CTAs of 128 dependent steps each; see kRowsRule for what R measured.
#include <math_constants.h>

#include "ap_common.cuh"

namespace ap {

namespace {

constexpr int kThreads = 256;

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

template <int D, int R>
struct SimtCfg {
  // S: a warp computes (4 RT) x (8 KT) of the R x 128 scores, lane = 4 row lanes x 8 key lanes
  static constexpr int RT = R == 32 ? 4 : 2;
  static constexpr int KT = R == 8 ? 2 : 4;
  static_assert((R / (4 * RT)) * (kTile / (8 * KT)) == kThreads / 32, "eight warps cover S");
  // P V: a thread owns PR rows x 4 columns; D/4 column lanes, R/PR row groups, the rest splits the keys
  static constexpr int PR = R == 32 ? 4 : 2;
  static constexpr int kSplit = kThreads / ((D / 4) * (R / PR));
  static_assert(kSplit >= 1 && kTile % (4 * kSplit) == 0, "keys split evenly");
  static constexpr int kPitch = kTile + 4;  // floats per row of S
  static constexpr int kKOff = R * D, kVOff = kKOff + kTile * D, kSOff = kVOff + kTile * D,
                       kAlphaOff = kSOff + R * kPitch, kFloats = kAlphaOff + 2 * R;
  static_assert(kSplit * R * D <= 2 * kTile * D, "the partial outputs fit over K and V");
};

template <int D, int R>
__global__ void __launch_bounds__(kThreads) fwd_simt_kernel(const float *__restrict__ Q, const float *__restrict__ K,
                                                            const float *__restrict__ V,
                                                            const int32_t *__restrict__ row_ptr,
                                                            const int32_t *__restrict__ col_idx,
                                                            const uint8_t *__restrict__ flags,
                                                            const uint32_t *__restrict__ bitmap,
                                                            float *__restrict__ O, int H, int Lq, int Lk, int n_qt,
                                                            int n_rt, float scale) {
  using C = SimtCfg<D, R>;
  constexpr int CH = D / 4;  // 16-byte chunks per row
  extern __shared__ __align__(16) float smem[];
  float *q_s = smem, *k_s = smem + C::kKOff, *v_s = smem + C::kVOff, *s_s = smem + C::kSOff,
        *alpha_s = smem + C::kAlphaOff, *l_s = alpha_s + R;
  const int rt = blockIdx.x % n_rt;
  const size_t bh = blockIdx.x / n_rt;
  const int i0 = rt * R, qt = i0 / kTile, h = (int)(bh % H);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t_begin = row_ptr[h * n_qt + qt], t_end = row_ptr[h * n_qt + qt + 1];

  auto copy_tile = [&](float *dst, const float *src, int kt) {
    for (int e = threadIdx.x; e < kTile * CH; e += kThreads) {
      const int jj = e / CH, c = e % CH, j = kt * kTile + jj;
      const bool valid = j < Lk;
      copy16(reinterpret_cast<float *>(chunk_at<D>(dst, jj, c)), src + (bh * Lk + (valid ? j : 0)) * D + 4 * c, valid);
    }
  };
  int kt_next = t_begin < t_end ? col_idx[t_begin] : 0;
  for (int e = threadIdx.x; e < R * CH; e += kThreads) {
    const int r = e / CH, c = e % CH, i = i0 + r;
    const bool valid = i < Lq;
    copy16(reinterpret_cast<float *>(chunk_at<D>(q_s, r, c)), Q + (bh * Lq + (valid ? i : 0)) * D + 4 * c, valid);
  }
  if (t_begin < t_end) copy_tile(k_s, K, kt_next);
  copy_commit();

  // scores: this thread's rows sr + 4 x and keys sk + 8 y
  constexpr int kKeyWarps = kTile / (8 * C::KT);
  const int sr = (warp / kKeyWarps) * 4 * C::RT + (lane >> 3), sk = (warp % kKeyWarps) * 8 * C::KT + (lane & 7);
  // softmax: this warp's rows, R / 8 of them; a lane owns four consecutive keys
  constexpr int kMyRows = R / 8;
  float m[kMyRows], l[kMyRows];
#pragma unroll
  for (int x = 0; x < kMyRows; ++x) m[x] = -CUDART_INF_F, l[x] = 0.f;
  // P V: column chunk pc, rows pr .. pr + PR - 1, keys of split part ps
  const int pc = threadIdx.x % CH, pr = (threadIdx.x / CH) % (R / C::PR) * C::PR, ps = threadIdx.x / (CH * (R / C::PR));
  float4 o[C::PR];
#pragma unroll
  for (int x = 0; x < C::PR; ++x) o[x] = make_float4(0.f, 0.f, 0.f, 0.f);

  for (int t = t_begin; t < t_end; ++t) {
    const int kt = kt_next;
    copy_tile(v_s, V, kt);  // (every thread is past the last P V, see the barrier at the loop's end)
    copy_commit();
    if (t + 1 < t_end) kt_next = col_idx[t + 1];
    const bool full = flags[t] & 1;
    uint32_t keep[kMyRows];
#pragma unroll
    for (int x = 0; x < kMyRows; ++x) {
      const int r = (i0 & (kTile - 1)) + warp * kMyRows + x;
      const uint32_t w = full ? 0xffffffffu : bitmap[(size_t)t * kBitmapWords + 4 * r + (lane >> 3)];
      keep[x] = w >> (4 * (lane & 7)) & 15u;
    }
    copy_wait<1>();  // K of this tile (and Q)
    __syncthreads();
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
    __syncthreads();
    if (t + 1 < t_end) copy_tile(k_s, K, kt_next);
    copy_commit();
#pragma unroll
    for (int x = 0; x < kMyRows; ++x) {
      const int r = warp * kMyRows + x;
      float4 *cell = reinterpret_cast<float4 *>(s_s + r * C::kPitch + 4 * lane);
      float4 v = *cell;
      v.x = keep[x] & 1u ? v.x : -CUDART_INF_F;
      v.y = keep[x] & 2u ? v.y : -CUDART_INF_F;
      v.z = keep[x] & 4u ? v.z : -CUDART_INF_F;
      v.w = keep[x] & 8u ? v.w : -CUDART_INF_F;
      float top = fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w));
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, d));
      const float m_new = fmaxf(m[x], top);
      const float ref = m_new == -CUDART_INF_F ? 0.f : m_new;
      const float alpha = expf(m[x] - ref);  // exp(-inf) = 0 before the row's first kept entry
      m[x] = m_new;
      v.x = expf(v.x - ref), v.y = expf(v.y - ref), v.z = expf(v.z - ref), v.w = expf(v.w - ref);
      *cell = v;
      float sum = (v.x + v.y) + (v.z + v.w);
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
      l[x] = l[x] * alpha + sum;
      if (lane == 0) alpha_s[r] = alpha;
    }
    copy_wait<1>();  // V of this tile
    __syncthreads();
#pragma unroll
    for (int x = 0; x < C::PR; ++x) {
      const float alpha = alpha_s[pr + x];
      o[x].x *= alpha, o[x].y *= alpha, o[x].z *= alpha, o[x].w *= alpha;
    }
    constexpr int kPart = kTile / C::kSplit;
#pragma unroll 2
    for (int j = ps * kPart; j < (ps + 1) * kPart; j += 4) {
      float4 p[C::PR];
#pragma unroll
      for (int x = 0; x < C::PR; ++x) p[x] = *reinterpret_cast<const float4 *>(s_s + (pr + x) * C::kPitch + j);
#pragma unroll
      for (int y = 0; y < 4; ++y) {
        const float4 v = *chunk_at<D>(v_s, j + y, pc);
#pragma unroll
        for (int x = 0; x < C::PR; ++x) {
          const float w = y == 0 ? p[x].x : y == 1 ? p[x].y : y == 2 ? p[x].z : p[x].w;
          o[x].x = fmaf(w, v.x, o[x].x), o[x].y = fmaf(w, v.y, o[x].y);
          o[x].z = fmaf(w, v.z, o[x].z), o[x].w = fmaf(w, v.w, o[x].w);
        }
      }
    }
    __syncthreads();  // S, alpha and V of this tile are read
  }
  // sums of the key parts (over K and V), then the division by l
  copy_wait<0>();
  float *part = k_s;
#pragma unroll
  for (int x = 0; x < C::PR; ++x)
    *reinterpret_cast<float4 *>(part + ((ps * R) + pr + x) * D + 4 * pc) = o[x];
#pragma unroll
  for (int x = 0; x < kMyRows; ++x)
    if (lane == 0) l_s[warp * kMyRows + x] = l[x];
  __syncthreads();
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
    *reinterpret_cast<float4 *>(O + (bh * Lq + i0 + r) * D + 4 * c) = out;
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
__global__ void __launch_bounds__(kThreads) fwd_entmax_simt_kernel(const T *__restrict__ Q, const T *__restrict__ K,
                                                                   const T *__restrict__ V,
                                                                   const int32_t *__restrict__ row_ptr,
                                                                   const int32_t *__restrict__ col_idx,
                                                                   const uint8_t *__restrict__ flags,
                                                                   const uint32_t *__restrict__ bitmap,
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
      for (int e = threadIdx.x; e < kTile * D / 4; e += kThreads) {
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
  kern<<<B * H * t.n_qt, kThreads, smem, s>>>(static_cast<const T *>(Q), static_cast<const T *>(K),
                                              static_cast<const T *>(V), t.row_ptr, t.col_idx, t.flags, t.bitmap,
                                              static_cast<T *>(O), H, Lq, Lk, t.n_qt, 0.5f * scale);
  count_launches(1);
  return cudaGetLastError();
}

template <int D, int R>
cudaError_t launch_rows(const void *Q, const void *K, const void *V, const ap_tiles &t, void *O, int B, int H, int Lq,
                        int Lk, float scale, cudaStream_t s) {
  constexpr size_t smem = SimtCfg<D, R>::kFloats * sizeof(float);
  auto kern = fwd_simt_kernel<D, R>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int n_rt = ceil_div(Lq, R);
  kern<<<(unsigned)((int64_t)B * H * n_rt), kThreads, smem, s>>>(
      static_cast<const float *>(Q), static_cast<const float *>(K), static_cast<const float *>(V), t.row_ptr, t.col_idx,
      t.flags, t.bitmap, static_cast<float *>(O), H, Lq, Lk, t.n_qt, n_rt, scale);
  count_launches(1);
  return cudaGetLastError();
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
