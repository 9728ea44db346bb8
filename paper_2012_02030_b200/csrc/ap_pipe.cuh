// What the warp-specialised kernels share: the 16-bit packing of the tensors' types, copies of runs of key rows, and the coalesced store of accumulator rows.
#pragma once

#include "ap_common.cuh"
#include "ap_sm100.cuh"

namespace ap {
namespace pipe {

using namespace sm100;

constexpr int kSubBytes = 128 * 128;  // one slab of a staged tile: 128 rows x 64 elements of 2 bytes
constexpr float kLog2e = 1.4426950408889634f;

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

template <bool kF16>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  if constexpr (kF16) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
}
template <bool kF16>
__device__ __forceinline__ float2 unpack2(uint32_t pk) {
  if constexpr (kF16) {
    return __half22float2(*reinterpret_cast<const __half2 *>(&pk));
  } else {
    return make_float2(__uint_as_float(pk << 16), __uint_as_float(pk & 0xffff0000u));
  }
}

// Layout of a staged tile of D columns.  kSplit = false: [slab][row][128 B], one box per 64-column slab;
// kSplit = true (d = 128, whole groups of eight rows): [row / 8][slab][8 rows][128 B], one box for both.
template <int D, bool kSplit>
struct TileLayout {
  static_assert(!kSplit || D == 128, "the split layout is for d = 128");
  static constexpr int kSub = D / 64;
  static constexpr int kBytes = kSub * kSubBytes;
  static constexpr int kSlabStride = kSplit ? 1024 : kSubBytes;  // slab 0 -> slab 1 of the same rows
  static constexpr int kSbo = kSplit ? 2048 : 1024;              // one group of eight rows -> the next
  static constexpr int kSlotStride = 2 * kSbo;                   // 16 rows -> the next 16
};

// (16 << lg) consecutive rows from `row` on, to slot q (16 rows each) of a staged tile.
template <int D, bool kSplit>
__device__ __forceinline__ void load_piece(unsigned char *tile, const CUtensorMap *m, uint64_t *bar, int q, int row,
                                           int bh) {
  using L = TileLayout<D, kSplit>;
  if constexpr (kSplit) {
    tma_load_5d(tile + q * L::kSlotStride, m, bar, 0, 0, 0, row >> 3, bh);
  } else {
#pragma unroll
    for (int s = 0; s < L::kSub; ++s)
      tma_load_3d(tile + s * kSubBytes + q * L::kSlotStride, m, bar, 64 * s, row, bh);
  }
}

// A run of `run` slots whose rows follow one another, starting with slot q at row `row`: pieces of 8, 4, 2 or 1
// slots (m4: maps of 16-, 32-, 64- and 128-row boxes).
template <int D, bool kSplit>
__device__ __forceinline__ void load_run(unsigned char *tile, const CUtensorMap *m4, uint64_t *bar, int q, int row,
                                         int run, int bh) {
  while (run > 0) {
    const int lg = run >= 8 ? 3 : run >= 4 ? 2 : run >= 2 ? 1 : 0;
    load_piece<D, kSplit>(tile, m4 + lg, bar, q, row, bh);
    q += 1 << lg;
    row += 16 << lg;
    run -= 1 << lg;
  }
}

// Lanes 0 .. ng-1 hold the first row of their slot (16 rows each).  A run starts at every slot that does not
// continue the one before; returns the run's length in slots for its first lane, 0 for every other lane.
__device__ __forceinline__ int run_of_slots(int lane, int ng, int row) {
  const int before = __shfl_up_sync(0xffffffffu, row, 1);
  const bool head = lane < ng && (lane == 0 || row != before + 16);
  const uint32_t heads = __ballot_sync(0xffffffffu, head);
  const uint32_t later = lane < 31 ? heads >> (lane + 1) : 0u;
  return head ? (later ? __ffs((int)later) : ng - lane) : 0;
}

// A warp's 32 accumulator rows, 32 columns of them packed to 16 bits in pk (lane = row), to global memory in whole 64-byte
// pieces: through 2 KB of shared memory, swizzled so that neither side has bank conflicts.  row_out(r): address of those columns
// of row r of the warp, or null.
template <class F>
__device__ __forceinline__ void store_rows(unsigned char *stage, int lane, const uint32_t *pk, F row_out) {
  auto place = [](int r, int p) { return r * 4 + (p ^ ((r >> 1) & 3)); };
  uint4 *s = reinterpret_cast<uint4 *>(stage);
#pragma unroll
  for (int p = 0; p < 4; ++p) s[place(lane, p)] = make_uint4(pk[4 * p], pk[4 * p + 1], pk[4 * p + 2], pk[4 * p + 3]);
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = 8 * k + lane / 4, p = lane % 4;
    uint16_t *out = row_out(r);
    if (out) *reinterpret_cast<uint4 *>(out + 8 * p) = s[place(r, p)];
  }
  __syncwarp();
}

}  // namespace pipe
}  // namespace ap
