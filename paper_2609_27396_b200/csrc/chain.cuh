// Host-side interface of the few-row chain: what lies between two attentions of a stack of blocks, in one launch.
#pragma once
#include "common.cuh"

namespace dpara {

constexpr int kChainRows = 128;       // activation rows at most
constexpr int kChainHidden = 5120;    // widest row that the row steps hold in registers
constexpr int kChainCounters = 8;     // of a launch, a 128-byte line each
constexpr int kChainCounterWords = kChainCounters * 32;

// Tiles of one product: `rows` weight rows each (gated: as many gate and up rows), its K range in `split` parts.
struct ChainTiles {
  int rows, tiles, split;
};
struct ChainShape {
  int ok;                 // 0: not a shape for this kernel
  int T;                  // activation rows, rounded up to 16
  ChainTiles o, gate_up, down, qkv;
  int op_bytes, w_stages, a_slots, smem;
  int on_way;             // stages of weights on their way at most
};
ChainShape chain_shape(int M, int hidden, int intermediate, int q_dim, int kv_dim, int head_dim);
// Room for the partial sums of a chain of up to M rows: what any tiles of it can need, and as much above kChainRows as at them, so that the scratch of a larger
// batch serves a smaller one.
size_t chain_plane_bytes(long M, int hidden, int q_dim, int kv_dim);

struct ChainArgs {
  int M, hidden, intermediate, n_q_heads, n_kv_heads, head_dim;
  // behind the attention: x + a W_o -> h1 -> norm -> gate/up -> down -> y
  int tail;
  const void *a, *w_o, *x, *rms2_w, *w_gate_up, *w_down;
  float eps2;
  float *h1;
  void *hn, *act;
  float *y_f32;           // may be null (between blocks)
  void *y_bf16;           // may be null (last block)
  // ahead of the next attention: (norm of y ->) QKV -> norm, rotation -> q, k, v
  int head;
  const void *rms1_w, *w_qkv, *qnorm_w, *knorm_w;
  float eps1;
  int use_norm;
  const float *angles;    // [row][cos of D / 2 angles | sin]; null: no rotation
  void *xn, *qkv, *q, *k, *v;
  float *planes;
  uint32_t *counters;     // kChainCounterWords of them, zero
};
// DPARA_ERR_UNSUPPORTED: nothing was launched, because this device (or the part of it the stream may use) cannot hold the grid at once.
dpara_status launch_chain(const ChainShape &sh, const ChainArgs &a, int32_t *status, cudaStream_t st);

}  // namespace dpara
