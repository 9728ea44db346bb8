// Shared between the backward's launcher, its rows kernel and its columns kernel.
#pragma once

#include "ap_pipe.cuh"

namespace ap {
namespace bwd {

// Everything the two kernels read that is not a tensor: carved out of the caller's workspace.
struct Plan {
  float *neg_l;       // [B*H][n_qt*128]  -log2 of the row's sum of 2^(c S); -inf: no kept entry
  float *dsum;        // [B*H][n_qt*128]  D_i = dO_i . O_i
  int32_t *next;      // [2]              next item to hand out (rows kernel, columns kernel)
  int32_t *tile_id;   // [H][n_qt][n_kt]  list position of a tile, -1 if it is not stored
  int32_t *order;     // [H][8*n_kt]      16-key group at each position of the head's key order
  int32_t *n_visits;  // [H][n_kt]        query tiles a key block of eight groups is visited by
  uint32_t *visit;    // [H][n_kt][n_qt]  bits 0..23: query tile; bits 24..31: its 16-row groups that keep an entry
  uint32_t *bits;     // [H][n_kt][n_qt][128 keys][4]  transposed bitmap of a visit: bit q of key row k
};

struct RowsMaps {
  CUtensorMap q, d_o;      // boxes of 128 rows
  CUtensorMap k[4], v[4];  // boxes of 16, 32, 64, 128 rows
};
struct ColsMaps {
  CUtensorMap q, d_o;
  CUtensorMap k[4], v[4];
};

struct Args {
  const ap_tiles *t;
  const void *O, *dO;
  void *dQ, *dK, *dV;
  Plan plan;
  int B, H, Lq, Lk, d, f16, split;
  float scale;
  unsigned *err;
  cudaStream_t s;
};

size_t plan_bytes(int B, int H, int Lq, int Lk);
Plan plan_at(void *workspace, int B, int H, int Lq, int Lk);
cudaError_t launch_plan(const Args &a);
cudaError_t launch_rows(const RowsMaps &maps, const Args &a);
cudaError_t launch_cols(const ColsMaps &maps, const Args &a);

}  // namespace bwd
}  // namespace ap
