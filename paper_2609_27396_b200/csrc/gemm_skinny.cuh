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

struct PairPlan {
  int t_tiles, nt;   // tiles of activation rows of one product, rows of each
  double us;         // model
};

// The kernel and the tiles of a launch, from its sizes (no pointer is looked at).
struct GemmRoute {
  int few;               // the kernel for few rows, with `skinny`; else CTA pairs, with `pair`
  SkinnyShape skinny;
  PairPlan pair;
  int n_tiles, n_all, most;   // CTA pairs: weight tiles of one product, of all products and parts of K; pairs of the device
  int nt_tail, main_units;    // activation rows of the units that the tiles of a nearly empty last round are cut into, whole tiles ahead of them; 0: none are cut
};
dpara_status gemm_route(const GemmArgs &g, GemmRoute &r);
dpara_status launch_gemm_skinny(const GemmArgs &g, const SkinnyShape &sh, int32_t *status, cudaStream_t st);

}  // namespace dpara
