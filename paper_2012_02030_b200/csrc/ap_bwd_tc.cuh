// Shared between the backward's launcher, its rows kernel and its columns kernel.
#pragma once

#include "ap_pipe.cuh"

namespace ap {
namespace bwd {

// What the two kernels hand on to one another.
struct Plan {
  float *neg_l;     // [B*H][Lq]        -log2 of the row's sum of 2^(c S); -inf: no kept entry
  float *dsum;      // [B*H][Lq]        D_i = dO_i . O_i
  uint32_t *table;  // [H][n_qt][n_kt]  bits 0..23: list position of a tile; 24..31: its groups that keep an entry (0: not stored)
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

cudaError_t launch_rows(const RowsMaps &maps, const Args &a);
cudaError_t launch_cols(const ColsMaps &maps, const Args &a);

}  // namespace bwd
}  // namespace ap
