// Host-side interface of the GEMM for few activation rows (weights as the rows of the product, split K inside clusters).
#pragma once
#include "gemm.cuh"

namespace dpara {

constexpr int kManyRows = 128;   // above this many activation rows only launches whose tiles all run at once

struct SkinnyShape {
  double cost;      // model, ns beside ~3500 of a launch; < 0: the shape is not taken
  int T, rows, halves, tiles, split, clusters, one_round;
  int chunk, stages, slabs, ring_bytes, bar_offset, smem, tmem_cols;
};
SkinnyShape skinny_shape(const GemmArgs &g);
dpara_status launch_gemm_skinny(const GemmArgs &g, const SkinnyShape &sh, int32_t *status, cudaStream_t st);

}  // namespace dpara
