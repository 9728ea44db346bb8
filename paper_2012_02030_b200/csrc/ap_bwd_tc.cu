// Derivative of the masked attention of Section 3.2 (what retraining under the mask, step 4 of
// the procedure, needs) for bf16 / fp16 tensors, on the tcgen05 tensor cores.
//
// With S = scale Q K^T, P = softmax of S over the kept entries of a row, O = P V and an incoming dO:
//   dV = P^T dO,   dP = dO V^T,   dS = P o (dP - D),  D_i = dO_i . O_i,
//   dQ = scale dS K,   dK = scale dS^T Q.
// Four kernels: a plan of the key side (here, two small ones), the rows kernel (dQ and the row statistics
// L = log2 sum 2^(c S), c = scale log2 e, and D; ap_bwd_rows_tc.cu) and the columns kernel (dK, dV;
// ap_bwd_cols_tc.cu).
//
// THE PLAN.  The rows kernel follows the tile list's rounds, which gather the key columns a query tile keeps.
// The columns kernel needs the same thing from the key side: blocks of 128 keys and, per block, the query
// tiles that keep an entry of it.  Masks of the method have a few heavy columns (attention sinks, strided
// positions) that nearly every query keeps, among bands that a few neighbouring query tiles keep; a block of
// 128 consecutive keys with one heavy column in it is visited by nearly every query tile.  So the keys of a
// head are put in an order of 16-key groups: first, in their natural order, the groups that are kept by about
// as many query tiles as their neighbours in the key tile, then the heavy ones (kept by more than twice the
// key tile's lower median + 2), and a block is eight groups at consecutive positions.  On 16 heads of 4096
// tokens, 5 % kept, a head is left with some 150 (block, query tile) visits of 333 stored tiles.  A mask
// without heavy groups keeps the natural order and is visited exactly at its stored tiles.
#include "ap_bwd_tc.cuh"

namespace ap {
namespace bwd {

namespace {

constexpr int kOrderThreads = 1024;
constexpr int kMaxOrdered = 8192;  // groups of a head that the order is worked out for (131 072 keys); beyond: natural order
constexpr int kVisitThreads = 256;

// One CTA per head: the (query tile, key tile) -> list position table and the key order.
__global__ void __launch_bounds__(kOrderThreads) order_kernel(const int32_t *__restrict__ row_ptr,
                                                              const int32_t *__restrict__ col_idx,
                                                              const uint8_t *__restrict__ flags,
                                                              const uint8_t *__restrict__ groups, int n_qt, int n_kt,
                                                              int32_t *__restrict__ tile_id,
                                                              int32_t *__restrict__ order, int32_t *__restrict__ next) {
  __shared__ int count[kMaxOrdered];
  __shared__ int warp_heavy[kOrderThreads / 32];
  const int h = blockIdx.x, n_groups = 8 * n_kt, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool ordered = n_groups <= kMaxOrdered;
  int32_t *ids = tile_id + (size_t)h * n_qt * n_kt;
  if (h == 0 && threadIdx.x < 2) next[threadIdx.x] = 0;
  for (int x = threadIdx.x; x < n_qt * n_kt; x += kOrderThreads) ids[x] = -1;
  if (ordered)
    for (int x = threadIdx.x; x < n_groups; x += kOrderThreads) count[x] = 0;
  __syncthreads();
  for (int qt = warp; qt < n_qt; qt += kOrderThreads / 32) {
    const int t1 = row_ptr[h * n_qt + qt + 1];
    for (int t = row_ptr[h * n_qt + qt] + lane; t < t1; t += 32) {
      const int kt = col_idx[t];
      ids[(size_t)qt * n_kt + kt] = t;
      const uint32_t gm = (flags[t] & 1u) ? 0xffu : groups[t];
      if (ordered)
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if ((gm >> q) & 1u) atomicAdd(&count[8 * kt + q], 1);
    }
  }
  __syncthreads();
  int32_t *out = order + (size_t)h * n_groups;
  if (!ordered) {
    for (int x = threadIdx.x; x < n_groups; x += kOrderThreads) out[x] = x;
    return;
  }
  // heavy: more than 2 * (lower median of the key tile's eight groups) + 2
  auto heavy = [&](int x) {
    const int mine = count[x];
    if (mine <= 2) return false;
    int below = 0;  // groups of the tile with a count under (mine - 2) / 2: at least four of them <=> mine > 2 * median + 2
    for (int q = 0; q < 8; ++q) below += 2 * count[(x & ~7) + q] + 2 < mine;
    return below >= 4;
  };
  int n_heavy_all = 0;
  for (int x0 = 0; x0 < n_groups; x0 += kOrderThreads)
    n_heavy_all += __syncthreads_count(x0 + (int)threadIdx.x < n_groups && heavy(x0 + (int)threadIdx.x));
  int heavy_before = 0;  // among the groups below x0
  for (int x0 = 0; x0 < n_groups; x0 += kOrderThreads) {
    const int x = x0 + (int)threadIdx.x;
    const bool is = x < n_groups && heavy(x);
    const uint32_t vote = __ballot_sync(0xffffffffu, is);
    __syncthreads();  // (warp_heavy of the previous step is read)
    if (lane == 0) warp_heavy[warp] = __popc(vote);
    __syncthreads();
    int before = heavy_before + __popc(vote & ((1u << lane) - 1u));
    for (int w = 0; w < kOrderThreads / 32; ++w) {
      const int c = warp_heavy[w];
      if (w < warp) before += c;
      heavy_before += c;
    }
    if (x < n_groups) out[is ? n_groups - n_heavy_all + before : x - before] = x;
  }
}

// 32 x 32 bit transpose across a warp: lane i's bit j becomes lane j's bit i.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane) {
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) {
    const uint32_t low = s == 16 ? 0x0000ffffu : s == 8 ? 0x00ff00ffu : s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u
                                                                                                  : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
    x = (lane & s) ? ((y >> s) & low) | (x & ~low) : (x & low) | ((y & low) << s);
  }
  return x;
}

// One CTA per (head, key block): its query tiles in ascending order and the transposed bitmap of each visit (a warp
// per visit).
__global__ void __launch_bounds__(kVisitThreads) visits_kernel(const int32_t *__restrict__ tile_id,
                                                               const int32_t *__restrict__ order,
                                                               const uint8_t *__restrict__ flags,
                                                               const uint8_t *__restrict__ groups,
                                                               const uint32_t *__restrict__ bitmap, int n_qt, int n_kt,
                                                               int32_t *__restrict__ n_visits,
                                                               uint32_t *__restrict__ visit,
                                                               uint32_t *__restrict__ bits) {
  __shared__ int list[kVisitThreads];
  __shared__ int warp_count[kVisitThreads / 32];
  const int h = blockIdx.x / n_kt, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t *ids = tile_id + (size_t)h * n_qt * n_kt;
  int group[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) group[q] = order[(size_t)blockIdx.x * 8 + q];
  // list position of the tile that holds group q's keys in query tile qt, -1 if the group keeps nothing there
  auto position = [&](int qt, int grp) {
    const int t = ids[(size_t)qt * n_kt + (grp >> 3)];
    if (t < 0) return -1;
    const uint32_t gm = (flags[t] & 1u) ? 0xffu : groups[t];
    return ((gm >> (grp & 7)) & 1u) ? t : -1;
  };
  int total = 0;
  for (int q0 = 0; q0 < n_qt; q0 += kVisitThreads) {
    const int qt = q0 + (int)threadIdx.x;
    bool any = false;
    if (qt < n_qt) {
#pragma unroll
      for (int q = 0; q < 8; ++q) any = any || position(qt, group[q]) >= 0;
    }
    const uint32_t vote = __ballot_sync(0xffffffffu, any);
    if (lane == 0) warp_count[warp] = __popc(vote);
    __syncthreads();
    int at = __popc(vote & ((1u << lane) - 1u)), found = 0;
    for (int w = 0; w < kVisitThreads / 32; ++w) {
      if (w < warp) at += warp_count[w];
      found += warp_count[w];
    }
    if (any) list[at] = qt;
    __syncthreads();
    for (int v = warp; v < found; v += kVisitThreads / 32) {
      const int tile = list[v];
      int pos[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) pos[q] = position(tile, group[q]);
      const size_t slot = (size_t)blockIdx.x * n_qt + total + v;
      uint32_t out[4][4];  // [word of 32 keys][block of 32 query rows]: lane = key
      uint32_t kept = 0u;  // 16-row query groups with a kept entry
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        uint32_t any_bits = 0u;
        const int row = 32 * b + lane;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          uint32_t x = 0u;
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int q = 2 * w + u;
            if (pos[q] >= 0)
              x |= (uint32_t)reinterpret_cast<const uint16_t *>(bitmap)[((size_t)pos[q] * kTile + row) * 8 + (group[q] & 7)]
                   << (16 * u);
          }
          any_bits |= x;
          out[w][b] = transpose32(x, lane);
        }
        const uint32_t rows = __ballot_sync(0xffffffffu, any_bits != 0u);
        kept |= ((rows & 0xffffu) ? 1u : 0u) << (2 * b) | ((rows >> 16) ? 2u : 0u) << (2 * b);
      }
      uint4 *dst = reinterpret_cast<uint4 *>(bits + slot * kBitmapWords);
#pragma unroll
      for (int w = 0; w < 4; ++w) dst[32 * w + lane] = make_uint4(out[w][0], out[w][1], out[w][2], out[w][3]);
      if (lane == 0) visit[slot] = (uint32_t)tile | (kept << 24);
    }
    total += found;
    __syncthreads();  // list and warp_count are read
  }
  if (threadIdx.x == 0) n_visits[blockIdx.x] = total;
}

size_t align256(size_t n) { return (n + 255) / 256 * 256; }

}  // namespace

Plan plan_at(void *workspace, int B, int H, int Lq, int Lk) {
  const size_t n_qt = ceil_div(Lq, kTile), n_kt = ceil_div(Lk, kTile), rows = (size_t)B * H * n_qt * kTile;
  char *p = static_cast<char *>(workspace);
  auto take = [&](size_t bytes) {
    char *at = p;
    p += align256(bytes);
    return at;
  };
  Plan plan;
  plan.neg_l = reinterpret_cast<float *>(take(rows * 4));
  plan.dsum = reinterpret_cast<float *>(take(rows * 4));
  plan.next = reinterpret_cast<int32_t *>(take(8));
  plan.tile_id = reinterpret_cast<int32_t *>(take(H * n_qt * n_kt * 4));
  plan.order = reinterpret_cast<int32_t *>(take(H * n_kt * 8 * 4));
  plan.n_visits = reinterpret_cast<int32_t *>(take(H * n_kt * 4));
  plan.visit = reinterpret_cast<uint32_t *>(take(H * n_qt * n_kt * 4));
  plan.bits = reinterpret_cast<uint32_t *>(take(H * n_qt * n_kt * kBitmapWords * 4));
  return plan;
}

size_t plan_bytes(int B, int H, int Lq, int Lk) {
  const size_t n_qt = ceil_div(Lq, kTile), n_kt = ceil_div(Lk, kTile), rows = (size_t)B * H * n_qt * kTile;
  return 2 * align256(rows * 4) + 256 + 2 * align256(H * n_qt * n_kt * 4) + align256(H * n_kt * 8 * 4) +
         align256(H * n_kt * 4) + align256(H * n_qt * n_kt * kBitmapWords * 4);
}

cudaError_t launch_plan(const Args &a) {
  const ap_tiles &t = *a.t;
  order_kernel<<<a.H, kOrderThreads, 0, a.s>>>(t.row_ptr, t.col_idx, t.flags, t.groups, t.n_qt, t.n_kt, a.plan.tile_id,
                                               a.plan.order, a.plan.next);
  visits_kernel<<<a.H * t.n_kt, kVisitThreads, 0, a.s>>>(a.plan.tile_id, a.plan.order, t.flags, t.groups, t.bitmap, t.n_qt,
                                                         t.n_kt, a.plan.n_visits, a.plan.visit, a.plan.bits);
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace bwd

size_t bwd_workspace_bytes(int B, int H, int Lq, int Lk) { return bwd::plan_bytes(B, H, Lq, Lk); }

cudaError_t launch_bwd_tc(const void *Q, const void *K, const void *V, const void *O, const void *dO,
                          const ap_tiles &t, void *dQ, void *dK, void *dV, void *workspace, int B, int H, int Lq,
                          int Lk, int d, int f16, float scale, cudaStream_t s) {
  unsigned *err = device_error_word();
  if (!err) return cudaErrorUnknown;
  const bool split = d == 128 && Lk % 8 == 0;
  bwd::RowsMaps rows;
  bwd::ColsMaps cols;
  bool ok = make_tile_map_bf16(&rows.q, Q, B * H, Lq, d) && make_tile_map_bf16(&rows.d_o, dO, B * H, Lq, d);
  cols.q = rows.q;
  cols.d_o = rows.d_o;
  for (int i = 0; i < 4 && ok; ++i) {
    const int n = 16 << i;
    ok = make_tile_map_bf16(&cols.k[i], K, B * H, Lk, d, n) && make_tile_map_bf16(&cols.v[i], V, B * H, Lk, d, n);
    if (!ok) break;
    if (split) {
      ok = make_split_map_bf16_d128(&rows.k[i], K, B * H, Lk, n) && make_split_map_bf16_d128(&rows.v[i], V, B * H, Lk, n);
    } else {
      rows.k[i] = cols.k[i];
      rows.v[i] = cols.v[i];
    }
  }
  if (!ok) return cudaErrorUnknown;
  bwd::Args a;
  a.t = &t;
  a.O = O, a.dO = dO, a.dQ = dQ, a.dK = dK, a.dV = dV;
  a.plan = bwd::plan_at(workspace, B, H, Lq, Lk);
  a.B = B, a.H = H, a.Lq = Lq, a.Lk = Lk, a.d = d, a.f16 = f16, a.split = split ? 1 : 0;
  a.scale = scale;
  a.err = err;
  a.s = s;
  cudaError_t e = bwd::launch_plan(a);
  if (e == cudaSuccess) e = bwd::launch_rows(rows, a);
  if (e == cudaSuccess) e = bwd::launch_cols(cols, a);
  return e;
}

}  // namespace ap
