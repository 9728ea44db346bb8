// Eq. 1 as a running sum, CUDA-core (fp32 FMA) version.
//
// One CTA owns up to 8 query rows of one head and loops over the B samples in
// ascending order, so every accumulator entry is updated by exactly one thread
// in a fixed order (no floating-point atomics; results are reproducible).  Per
// sample: scores of the rows against all keys of the row domain go to shared
// memory, then one warp per row takes the row maximum, the sum of exponentials
// and adds the normalised row to the accumulator with coalesced read-modify-
// writes.  Used for fp32 inputs, where tensor-core precision would not do.
//
// What bounds it: the key rows' loads (a lane per row: as many lines per load as lanes) and the latency of a sample's
// phases.  With 16-byte loads four at a time, the exponentials computed twice and one load of the accumulator under way:
// 168 us at 16 x 8 heads x 256 x 64, 122 now; 34 -> 26 us at 3 x 16 heads x 194 x 64 (causal).
//
// kEntmax: the same sum with 1.5-entmax as the normaliser (the section on sparse normalisation),
// p_j = max(s_j / 2 - tau, 0)^2 with tau such that the row sums to 1.  The row's scores are in
// shared memory, so the warp iterates on tau there: from max/2 - 0.625 (the root lies in [max/2 - 1, max/2)) to the
// smaller root of the parabola of the current support, tau + (S2 - 1) / (S1 + sqrt(S1^2 - n (S2 - 1)))
// with n, S1, S2 the support's size and its sums of (s_j/2 - tau) and of its square (Newton's
// step (S2 - 1) / (2 S1) where the parabola has no root), until the step falls under
// 5e-7 max(1, |tau|) (at most 30 steps).
#include <math_constants.h>

#include "ap_common.cuh"

namespace ap {

namespace {

constexpr int kRows = 8;
constexpr int kThreads = 256;
constexpr int kPiece = 64;  // elements of a key row loaded at once

// kPiece elements of a key row, from a 32-byte boundary (wide) or a 16-byte one.  A thread reads a row of its own, so that
// a load touches as many lines as the warp has lanes whatever its size: twice the size, half the lines' cycles.  (Volatile: all
// loads are under way before the first product.)
__device__ __forceinline__ void load_piece(const float *p, float v[kPiece], bool wide) {
  if (wide) {
#pragma unroll
    for (int t = 0; t < kPiece; t += 8)
      asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=f"(v[t]), "=f"(v[t + 1]), "=f"(v[t + 2]), "=f"(v[t + 3]), "=f"(v[t + 4]), "=f"(v[t + 5]),
                     "=f"(v[t + 6]), "=f"(v[t + 7])
                   : "l"(p + t));
  } else {
#pragma unroll
    for (int t = 0; t < kPiece; t += 4)
      asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                   : "=f"(v[t]), "=f"(v[t + 1]), "=f"(v[t + 2]), "=f"(v[t + 3])
                   : "l"(p + t));
  }
}

template <int D, bool kEntmax>
__global__ void __launch_bounds__(kThreads) accumulate_simt_kernel(float *__restrict__ acc, const float *Q,
                                                                   const float *K,
                                                                   const float *bias, int B, int H,
                                                                   int Lq, int Lk, int rows, int causal,
                                                                   float scale) {
  extern __shared__ __align__(16) float smem[];
  float *q_s = smem;                 // [rows][D]
  float *s_s = smem + kRows * D;     // [rows][Lk]
  const int h = blockIdx.y;
  const int i0 = blockIdx.x * rows;
  const int n_rows = min(rows, Lq - i0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // keys any row of this block may look at
  const int off = causal ? Lk - Lq : 0;  // causal: row i looks at keys j <= i + (Lk - Lq)
  const int jmax = causal ? min(Lk, i0 + n_rows + off) : Lk;

  // Nothing is allowed to the kernel behind before the blocks end: several blocks share an SM, and the next call's would gather on
  // the SMs that are left first instead of spreading over all of them (8 x 8 heads x 256, causal, calls in a row: 72 us with it,
  // 58 without, 60 as an ordinary launch; 2 x 8 x 500, d = 128: 77, 72, 74).
  wait_previous();
  const bool wide = (reinterpret_cast<uintptr_t>(K) & 31) == 0;
  for (int b = 0; b < B; ++b) {
    const float *Qb = Q + (((size_t)b * H + h) * Lq + i0) * D;
    const float *Kb = K + ((size_t)b * H + h) * (size_t)Lk * D;
    for (int e = threadIdx.x; e < kRows * D; e += kThreads) {
      const int r = e / D;
      q_s[e] = r < n_rows ? Qb[e] : 0.f;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < jmax; j += kThreads) {
      float dot[kRows];
#pragma unroll
      for (int r = 0; r < kRows; ++r) dot[r] = 0.f;
      const float *krow = Kb + (size_t)j * D;
#pragma unroll 1
      for (int t0 = 0; t0 < D; t0 += kPiece) {
        float kv[kPiece];
        load_piece(krow + t0, kv, wide);
#pragma unroll
        for (int t = 0; t < kPiece; t += 4)
#pragma unroll
          for (int r = 0; r < kRows; ++r) {
            const float4 q = *reinterpret_cast<const float4 *>(q_s + r * D + t0 + t);
            dot[r] = fmaf(q.x, kv[t], dot[r]); dot[r] = fmaf(q.y, kv[t + 1], dot[r]);
            dot[r] = fmaf(q.z, kv[t + 2], dot[r]); dot[r] = fmaf(q.w, kv[t + 3], dot[r]);
          }
      }
#pragma unroll
      for (int r = 0; r < kRows; ++r) {
        if (r < n_rows) {
          float s = dot[r] * scale;
          if (bias) s += bias[((size_t)h * Lq + i0 + r) * Lk + j];
          s_s[(size_t)r * Lk + j] = s;
        }
      }
    }
    __syncthreads();
    // warp r normalises row r and adds it to the accumulator
    for (int r = warp; r < n_rows; r += kThreads / 32) {
      const int i = i0 + r;
      const int jend = causal ? min(Lk, i + 1 + off) : Lk;
      float *srow = s_s + (size_t)r * Lk;
      float m = -CUDART_INF_F;
      for (int j = lane; j < jend; j += 32) m = fmaxf(m, srow[j]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      float *arow = acc + ((size_t)h * Lq + i) * Lk;
      if (kEntmax) {
        float tau = 0.5f * m - 0.625f;  // the root lies in [max/2 - 1, max/2)
        for (int it = 0; it < 30; ++it) {
          float n = 0.f, S1 = 0.f, S2 = 0.f;
          for (int j = lane; j < jend; j += 32) {
            const float u = fmaf(0.5f, srow[j], -tau);
            if (u > 0.f) {
              n += 1.f;
              S1 += u;
              S2 = fmaf(u, u, S2);
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {  // every lane ends with the same bits
            n += __shfl_xor_sync(0xffffffffu, n, o);
            S1 += __shfl_xor_sync(0xffffffffu, S1, o);
            S2 += __shfl_xor_sync(0xffffffffu, S2, o);
          }
          const float disc = S1 * S1 - n * (S2 - 1.f);
          const float step = S1 > 0.f ? (S2 - 1.f) / (S1 + (disc >= 0.f ? sqrtf(disc) : S1)) : 0.f;
          tau += step;
          if (fabsf(step) <= 5e-7f * fmaxf(1.f, fabsf(tau))) break;
        }
        for (int j = lane; j < jend; j += 32) {
          const float u = fmaf(0.5f, srow[j], -tau);
          if (u > 0.f) arow[j] += u * u;
        }
        continue;
      }
      float z = 0.f;
      for (int j = lane; j < jend; j += 32) {
        const float e = expf(srow[j] - m);
        srow[j] = e;
        z += e;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
      for (int j0 = lane; j0 < jend; j0 += 128) {  // four of the accumulator's loads under way
        float a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = j0 + 32 * u < jend ? arow[j0 + 32 * u] : 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (j0 + 32 * u < jend) arow[j0 + 32 * u] = a[u] + srow[j0 + 32 * u] / z;
      }
    }
    __syncthreads();
  }
}

template <int D, bool kEntmax>
cudaError_t launch(float *acc, const void *Q, const void *K, const float *bias, int B, int H, int Lq, int Lk,
                   int causal, float scale, cudaStream_t s) {
  // as many rows per CTA (up to 8) as the score rows allow in shared memory
  int rows = kRows;
  const size_t budget = 200 * 1024;
  while (rows > 1 && (size_t)(kRows * D + (size_t)rows * Lk) * sizeof(float) > budget) rows >>= 1;
  const size_t smem = (size_t)(kRows * D + (size_t)rows * Lk) * sizeof(float);
  if (smem > budget) return cudaErrorInvalidValue;
  auto kern = accumulate_simt_kernel<D, kEntmax>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  dim3 grid(ceil_div(Lq, rows), H);
  e = launch_early(kern, grid, kThreads, smem, s, acc, static_cast<const float *>(Q), static_cast<const float *>(K), bias, B, H,
                   Lq, Lk, rows, causal, scale);
  return e;
}

}  // namespace

cudaError_t launch_accumulate_simt(float *acc, const void *Q, const void *K, const float *bias, int B, int H,
                                   int Lq, int Lk, int d, int causal, float scale,
                                   cudaStream_t s, int entmax) {
  if (entmax)
    return d == 64 ? launch<64, true>(acc, Q, K, bias, B, H, Lq, Lk, causal, scale, s)
                   : launch<128, true>(acc, Q, K, bias, B, H, Lq, Lk, causal, scale, s);
  return d == 64 ? launch<64, false>(acc, Q, K, bias, B, H, Lq, Lk, causal, scale, s)
                 : launch<128, false>(acc, Q, K, bias, B, H, Lq, Lk, causal, scale, s);
}

}  // namespace ap
