// Derivative of the masked attention of Section 3.2 (what retraining under the mask, step 4 of
// the procedure, needs) for bf16 / fp16 tensors, on the tcgen05 tensor cores.
//
// With S = scale Q K^T, P = softmax of S over the kept entries of a row, O = P V and an incoming dO:
//   dV = P^T dO,   dP = dO V^T,   dS = P o (dP - D),  D_i = dO_i . O_i,
//   dQ = scale dS K,   dK = scale dS^T Q.
// Two kernels: the rows kernel (dQ, the row statistics L = log2 sum 2^(c S), c = scale log2 e, and D, and the (query tile,
// key tile) table; ap_bwd_rows_tc.cu) and the columns kernel (dK, dV; ap_bwd_cols_tc.cu).
#include "ap_bwd_tc.cuh"

namespace ap {
namespace bwd {

namespace {

size_t stats_bytes(int B, int H, int Lq) { return (2 * sizeof(float) * (size_t)B * H * Lq + 255) / 256 * 256; }

}  // namespace
}  // namespace bwd

// row statistics (L and D, one float each per query row) and the (query tile, key tile) table
size_t bwd_workspace_bytes(int B, int H, int Lq, int Lk) {
  return bwd::stats_bytes(B, H, Lq) + sizeof(uint32_t) * (size_t)H * ceil_div(Lq, kTile) * ceil_div(Lk, kTile);
}

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
  a.plan.neg_l = static_cast<float *>(workspace);
  a.plan.dsum = a.plan.neg_l + (size_t)B * H * Lq;
  a.plan.table = reinterpret_cast<uint32_t *>(static_cast<char *>(workspace) + bwd::stats_bytes(B, H, Lq));
  a.B = B, a.H = H, a.Lq = Lq, a.Lk = Lk, a.d = d, a.f16 = f16, a.split = split ? 1 : 0;
  a.scale = scale;
  a.err = err;
  a.s = s;
  cudaError_t e = bwd::launch_rows(rows, a);
  if (e == cudaSuccess) e = bwd::launch_cols(cols, a);
  return e;
}

}  // namespace ap
