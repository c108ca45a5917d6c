// One backbone block around the all-boundary attention (Sec. 3.1 lists a block's parts, no
// equations; the block equations are stated with dpara_draft_all_boundaries in the header):
//   rmsnorm -> QKV GEMM -> per-head RMS norm + rotary embedding -> all-boundary attention ->
//   O GEMM (+x) -> rmsnorm -> gate/up GEMM with fused SiLU*up -> down GEMM (+h1).
// The GEMMs and the attention are the tensor-core kernels; the three small kernels here are row-wise
// and HBM-bound (M rows of a few KB each).  Few rows: everything between two attentions is one launch (chain.cu).
#include <math.h>

#include <algorithm>

#include "attention_tc.cuh"
#include "chain.cuh"
#include "gemm.cuh"
#include "layer.cuh"

namespace dpara {

void fill_attn_params(AttnParams &P, const dpara_shape *s, const dpara_attn_io *io, int32_t *status_word);

// ------------------------------------------------------------------------------------------------ rmsnorm
// out[row] = bf16( x[row] / sqrt(mean(x^2) + eps) * gain ),  x bf16 or fp32, one 128-thread CTA per row.  A row is a few KB: what the
// kernel takes is round trips to memory, so a thread has up to kHeld of its 8-element pieces and their gains in flight together and
// keeps them for the second pass (longer rows: the rest is read twice).  With the angles of the next kernel ahead of its wait: five blocks
// of 72 rows 655 -> 638 us.
template <bool kF32In>
__device__ __forceinline__ void rms_load(const void *x, size_t at, float (&v)[8]) {
  if (kF32In) {
    const float4 *p = reinterpret_cast<const float4 *>(static_cast<const float *>(x) + at);
    const float4 a = p[0], b = p[1];
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
    const uint4 w = *reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(x) + at);
    v[0] = bf16lo(w.x); v[1] = bf16hi(w.x); v[2] = bf16lo(w.y); v[3] = bf16hi(w.y);
    v[4] = bf16lo(w.z); v[5] = bf16hi(w.z); v[6] = bf16lo(w.w); v[7] = bf16hi(w.w);
  }
}

__device__ __forceinline__ void rms_store(uint16_t *out, const float (&v)[8], float rs, uint4 g) {
  uint4 o;
  o.x = pack_bf16(v[0] * rs * bf16lo(g.x), v[1] * rs * bf16hi(g.x));
  o.y = pack_bf16(v[2] * rs * bf16lo(g.y), v[3] * rs * bf16hi(g.y));
  o.z = pack_bf16(v[4] * rs * bf16lo(g.z), v[5] * rs * bf16hi(g.z));
  o.w = pack_bf16(v[6] * rs * bf16lo(g.w), v[7] * rs * bf16hi(g.w));
  *reinterpret_cast<uint4 *>(out) = o;
}

// Rotary angles of a call's rows, in double precision.  Slot i of boundary j of request n sits at position L_n + j + 2 + i (the unknown bonus of
// boundary j at L_n + j + 1), spine row s at L_n + s.
struct AngleJob {
  float *table = nullptr;                     // [row][cos of D / 2 angles | sin of D / 2]; null: no table
  const int64_t *ctx_offsets = nullptr, *ctx_lens = nullptr;   // lengths: ctx_lens, or the offsets' differences
  int rows = 0, per_request = 1, slot_rows = 0, block = 1;     // a request's first slot_rows rows are slots of boundaries of `block`, the others spine rows
  int half = 0;                               // D / 2
  double inv_freq[64] = {};                   // theta^(-2 d / D), d < D / 2, worked out on the host in double precision
  uint32_t *clear = nullptr;                  // the counters of a call's chains, n_clear of them, to zero
  int n_clear = 0;
  const int64_t *copy = nullptr;              // lengths to be kept as they were, n_copy of them
  int64_t *copy_to = nullptr;
  int n_copy = 0;
};
__device__ __forceinline__ void row_angle(const AngleJob &A, int row, int d, float &c, float &s) {
  const int n = row / A.per_request, rr = row - n * A.per_request;
  const int rel = rr < A.slot_rows ? rr / A.block + 2 + rr % A.block : rr - A.slot_rows;
  const double pos = (double)(A.ctx_lens ? A.ctx_lens[n] : A.ctx_offsets[n + 1] - A.ctx_offsets[n]) + rel;
  double sn, cs;
  sincos(pos * A.inv_freq[d], &sn, &cs);
  c = (float)cs;
  s = (float)sn;
}
constexpr int kAnglesPerBlock = 256;
__device__ __noinline__ void angle_block(const AngleJob &A, int first) {
  for (int k = first + threadIdx.x; k < min(first + kAnglesPerBlock, A.rows * A.half); k += 128) {
    const int row = k / A.half, d = k - row * A.half;
    float *t = A.table + (size_t)row * 2 * A.half + d;
    row_angle(A, row, d, t[0], t[A.half]);
  }
}

template <bool kF32In, bool kAngles>
__global__ void __launch_bounds__(128) rmsnorm_kernel(const void *__restrict__ x, const uint16_t *__restrict__ gain,
                                                      uint16_t *__restrict__ out, int M, int H, float eps, const __grid_constant__ AngleJob angles) {
  constexpr int kHeld = 5;   // rows of 5120 elements
  const int row = blockIdx.x, tid = threadIdx.x;
  if (kAngles && row >= M) {
    pdl_wait();
    pdl_launch_dependents();
    if (row == M) {
      for (int k = tid; k < angles.n_clear; k += 128) angles.clear[k] = 0u;
      for (int k = tid; k < angles.n_copy; k += 128) angles.copy_to[k] = angles.copy[k];
    }
    if (angles.table) angle_block(angles, (row - M) * kAnglesPerBlock);
    return;
  }
  const size_t base = (size_t)row * H;
  // (no gain: bf16 ones)
  auto gain_at = [&](int c) { return gain ? *reinterpret_cast<const uint4 *>(gain + c) : make_uint4(0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u); };
  pdl_wait();
  pdl_launch_dependents();
  float v[kHeld][8];
  uint4 g[kHeld];
#pragma unroll
  for (int i = 0; i < kHeld; ++i) {
    const int c = tid * 8 + i * 1024;
    if (c < H) rms_load<kF32In>(x, base + c, v[i]);
  }
#pragma unroll
  for (int i = 0; i < kHeld; ++i) {
    const int c = tid * 8 + i * 1024;
    if (c < H) g[i] = gain_at(c);
  }
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < kHeld; ++i)
    if (tid * 8 + i * 1024 < H) {
#pragma unroll
      for (int e = 0; e < 8; ++e) ss = fmaf(v[i][e], v[i][e], ss);
    }
  for (int c = tid * 8 + kHeld * 1024; c < H; c += 1024) {
    float t[8];
    rms_load<kF32In>(x, base + c, t);
#pragma unroll
    for (int e = 0; e < 8; ++e) ss = fmaf(t[e], t[e], ss);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  __shared__ float s_part[4];
  if ((tid & 31) == 0) s_part[tid >> 5] = ss;
  __syncthreads();
  const float tot = s_part[0] + s_part[1] + s_part[2] + s_part[3];
  const float rs = rsqrtf(tot / (float)H + eps);
#pragma unroll
  for (int i = 0; i < kHeld; ++i) {
    const int c = tid * 8 + i * 1024;
    if (c < H) rms_store(out + base + c, v[i], rs, g[i]);
  }
  for (int c = tid * 8 + kHeld * 1024; c < H; c += 1024) {
    float t[8];
    rms_load<kF32In>(x, base + c, t);
    rms_store(out + base + c, t, rs, gain_at(c));
  }
}

// ------------------------------------------------------------------------------------------------ q/k norm + rope, v copy
// gridDim.y CTAs of four warps per token row (few rows: enough that a warp has one or two heads, the kernel is then one round trip to memory; one CTA
// per row took 7 us behind the product at 72 rows of 40 heads).  qkv row = [Hq*D | Hkv*D | Hkv*D].  q and k heads: optional RMS norm over D
// (rounded to bf16), then rotate-half rotary embedding by the row's angles (rounded to bf16).
// With spine query rows a request has J * Bq + S rows: the mask-slot rows, then the spine rows.
struct QkParams {
  const uint16_t *qkv;
  const uint16_t *qnorm_w, *knorm_w;
  uint16_t *q, *k, *v;
  int Hq, Hkv, D;
  int use_rope, use_norm;
  float eps;
  AngleJob angles;
};

template <bool kSplit>
__global__ void __launch_bounds__(128) qk_norm_rope_kernel(const QkParams P) {
  extern __shared__ float s_cs[];  // cos[D/2], sin[D/2]
  const int row = blockIdx.x, tid = threadIdx.x;
  const int half = P.D / 2;
  // The angles before the wait: the kernel in front is the QKV product, which writes neither lengths nor offsets and lets this one go only when
  // everything before it has ended, the norm that made a table among it.
  if (P.use_rope) {
    if (kSplit) {
      for (int d = tid; d < P.D; d += 128) s_cs[d] = P.angles.table[(size_t)row * P.D + d];
    } else {
      for (int d = tid; d < half; d += 128) row_angle(P.angles, row, d, s_cs[d], s_cs[half + d]);
    }
  }
  pdl_wait();
  pdl_launch_dependents();
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  const size_t qkv_row = (size_t)row * (P.Hq + 2 * P.Hkv) * P.D;
  // A lane owns the element pairs (2 lane, 2 lane + 1) of both halves of a head (one 4-byte load each); a warp takes heads
  // warp, warp + 4 gridDim.y, ... and fetches kChunk of them before it works on the first, so that a row costs a few global round
  // trips instead of one per head.
  constexpr int kChunk = 6;
  const bool active = 2 * lane < half;
  const int n_heads = P.Hq + P.Hkv;
  const int part = kSplit ? (int)blockIdx.y : 0, stride = kSplit ? 4 * (int)gridDim.y : 4;
  for (int hd0 = part * 4 + warp; hd0 < n_heads; hd0 += stride * kChunk) {
    uint32_t lo[kChunk], hi[kChunk];
#pragma unroll
    for (int c = 0; c < kChunk; ++c) {
      const int hd = hd0 + stride * c;
      lo[c] = hi[c] = 0u;
      if (hd < n_heads && active) {
        const uint16_t *src = P.qkv + qkv_row + (size_t)hd * P.D;
        lo[c] = *reinterpret_cast<const uint32_t *>(src + 2 * lane);
        hi[c] = *reinterpret_cast<const uint32_t *>(src + half + 2 * lane);
      }
    }
#pragma unroll
    for (int c = 0; c < kChunk; ++c) {
      const int hd = hd0 + stride * c;
      if (hd >= n_heads) break;
      const bool is_q = hd < P.Hq;
      uint16_t *dst = is_q ? P.q + ((size_t)row * P.Hq + hd) * P.D : P.k + ((size_t)row * P.Hkv + (hd - P.Hq)) * P.D;
      const uint16_t *gain = is_q ? P.qnorm_w : P.knorm_w;
      float x1[2] = {bf16lo(lo[c]), bf16hi(lo[c])}, x2[2] = {bf16lo(hi[c]), bf16hi(hi[c])};
      if (P.use_norm) {
        float ss = x1[0] * x1[0] + x2[0] * x2[0] + x1[1] * x1[1] + x2[1] * x2[1];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float rs = rsqrtf(ss / (float)P.D + P.eps);
        if (active) {
          const uint32_t g1 = gain ? *reinterpret_cast<const uint32_t *>(gain + 2 * lane) : 0x3f803f80u;          // bf16 1.0 twice
          const uint32_t g2 = gain ? *reinterpret_cast<const uint32_t *>(gain + half + 2 * lane) : 0x3f803f80u;
          x1[0] = __bfloat162float(__float2bfloat16_rn(x1[0] * rs * bf16lo(g1)));
          x1[1] = __bfloat162float(__float2bfloat16_rn(x1[1] * rs * bf16hi(g1)));
          x2[0] = __bfloat162float(__float2bfloat16_rn(x2[0] * rs * bf16lo(g2)));
          x2[1] = __bfloat162float(__float2bfloat16_rn(x2[1] * rs * bf16hi(g2)));
        }
      }
      if (active) {
        float y1[2] = {x1[0], x1[1]}, y2[2] = {x2[0], x2[1]};
        if (P.use_rope) {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float cs = s_cs[2 * lane + e], sn = s_cs[half + 2 * lane + e];
            y1[e] = x1[e] * cs - x2[e] * sn;
            y2[e] = x2[e] * cs + x1[e] * sn;
          }
        }
        *reinterpret_cast<uint32_t *>(dst + 2 * lane) = pack_bf16(y1[0], y1[1]);
        *reinterpret_cast<uint32_t *>(dst + half + 2 * lane) = pack_bf16(y2[0], y2[1]);
      }
    }
  }
  // v: plain copy into its own contiguous tensor
  const uint16_t *vsrc = P.qkv + qkv_row + (size_t)(P.Hq + P.Hkv) * P.D;
  uint16_t *vdst = P.v + (size_t)row * P.Hkv * P.D;
  for (int c = (part * 128 + tid) * 8; c < P.Hkv * P.D; c += 32 * 8 * stride) *reinterpret_cast<uint4 *>(vdst + c) = *reinterpret_cast<const uint4 *>(vsrc + c);
}

// ------------------------------------------------------------------------------------------------ host
namespace {
struct LayerWs {
  size_t xn, qkv, q, k, v, a, h1, hn, act, angles, attn, planes, total;
};

// The chain of a stack of n_blocks; not ok: kernels of their own.  Times of those / with the chain, called one by one, rows 4 to 128:
//   blocks     weights of a block, MB:  2..8         13..21       29..58       74..96       144..233     312..386 (to 48 rows, to 64, more)  477..661
//   five                                1.11..1.21   1.10..1.16   1.06..1.13   1.00..1.06   0.99..1.09   0.95..1.00, 1.00..1.01, 1.00..1.03  1.00..1.09
//   two, three                          1.05..1.18   1.05..1.13   1.01..1.12   0.99..1.04   0.98..1.08   0.96..1.00, -, 0.99..1.03           0.97..1.06
//   one                                 0.97..1.11   0.97..1.10   0.94..1.05   0.91..1.04   0.97..1.06   0.94..0.98, 0.96..1.00, 0.96..1.02  0.94..1.14
// A stack's first and last chain have one and three of the four products, so one block is two launches that do not start ahead of the end of the kernel in front, and the
// meetings of all CTAs, against seven that do: worth it where launches are what a block is, or beyond the sizes that the kernels of their own fill the SMs with.  (One block of at
// most 32 rows: 0.97 to 1.06 to 13 MB, 0.94 to 1.03 from 21 to 58.)  In a graph the smallest are 1.03..1.14, the others as they are here.
ChainShape block_chain(const dpara_shape *s, const dpara_layer_io *l, int n_blocks) {
  const long M = (long)s->batch * (s->n_boundaries * s->block + (s->spine_queries ? s->n_spine : 0));
  if (M > kChainRows) return ChainShape{};
  const double weights = 2.0 * l->hidden * ((double)(2 * s->n_q_heads + 2 * s->n_kv_heads) * s->head_dim + 3.0 * l->intermediate);
  if (weights > 256e6 && M <= (n_blocks == 1 ? 64 : 48)) return ChainShape{};
  if (n_blocks == 1 && weights > (M <= 32 ? 16e6 : 64e6) && weights < 128e6) return ChainShape{};
  return chain_shape((int)M, l->hidden, l->intermediate, s->n_q_heads * s->head_dim, s->n_kv_heads * s->head_dim, s->head_dim);
}

LayerWs layer_ws_layout(const dpara_shape *s, const dpara_layer_io *l, size_t attn_bytes) {
  const size_t M = (size_t)s->batch * (s->n_boundaries * s->block + (s->spine_queries ? s->n_spine : 0));
  const size_t H = l->hidden, I = l->intermediate, QD = (size_t)s->n_q_heads * s->head_dim, KD = (size_t)s->n_kv_heads * s->head_dim;
  LayerWs w;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t r = o; o += align_up(bytes, 256); return r; };
  w.xn = take(M * H * 2);
  w.qkv = take(M * (QD + 2 * KD) * 2);
  w.q = take(M * QD * 2);
  w.k = take(M * KD * 2);
  w.v = take(M * KD * 2);
  w.a = take(M * QD * 2);
  w.h1 = take(M * H * 4);
  w.hn = take(M * H * 2);
  w.act = take(M * I * 2);
  w.angles = take(M * s->head_dim * 4);
  w.attn = take(attn_bytes);
  w.planes = take(chain_plane_bytes((long)M, l->hidden, s->n_q_heads * s->head_dim, s->n_kv_heads * s->head_dim));
  w.total = o;
  return w;
}

// A call's counters: of every chain of a stack of n blocks, one in front of each attention and one behind the last.
size_t counter_bytes(int n_blocks) { return (size_t)(n_blocks + 1) * kChainCounterWords * sizeof(uint32_t); }
}  // namespace

void layer_workspace_offsets(const dpara_shape *shape, const dpara_layer_io *layer, size_t attn_bytes, size_t out[9]) {
  const LayerWs w = layer_ws_layout(shape, layer, 0);
  const size_t o[9] = {w.xn, w.qkv, w.q, w.k, w.v, w.a, w.h1, w.hn, w.act};
  for (int i = 0; i < 9; ++i) out[i] = attn_bytes + o[i];
}

template <bool kF32In>
static dpara_status launch_rmsnorm(const void *x, const void *gain, void *out, int M, int H, float eps, const AngleJob &angles, cudaStream_t st) {
  const int angle_blocks = angles.table ? (angles.rows * angles.half + kAnglesPerBlock - 1) / kAnglesPerBlock : 0, blocks = (angles.n_clear || angles.n_copy) && !angle_blocks ? 1 : angle_blocks;
  launch_pdl(blocks ? rmsnorm_kernel<kF32In, true> : rmsnorm_kernel<kF32In, false>, dim3(M + blocks), dim3(128), 0, st, x, static_cast<const uint16_t *>(gain), static_cast<uint16_t *>(out), M, H, eps, angles);
  DPARA_CHECK_LAUNCH();
  count_launches(1);
  return DPARA_OK;
}

dpara_status launch_rmsnorm_bf16(const void *x, const void *gain, void *out, int M, int H, float eps, cudaStream_t st, const int64_t *copy, int64_t *to, int n_copy) {
  if (H % 8) return DPARA_ERR_UNSUPPORTED;
  AngleJob job;
  job.copy = copy;
  job.copy_to = to;
  job.n_copy = copy ? n_copy : 0;
  return launch_rmsnorm<false>(x, gain, out, M, H, eps, job, st);
}

size_t layer_workspace_bytes(const dpara_shape *shape, const dpara_layer_io *layer) {
  if (layer->hidden <= 0 || layer->intermediate <= 0) return 0;
  return layer_ws_layout(shape, layer, 0).total + align_up(counter_bytes(1), 256);  // the attention's own scratch is added by the caller
}

// The block's pointers into its workspace
namespace {
struct BlockBuffers {
  uint16_t *xn, *qkv, *q, *k, *v, *a, *hn, *act;
  float *h1, *angles, *planes;
  BlockBuffers(uint8_t *lw, const LayerWs &w)
      : xn(reinterpret_cast<uint16_t *>(lw + w.xn)), qkv(reinterpret_cast<uint16_t *>(lw + w.qkv)), q(reinterpret_cast<uint16_t *>(lw + w.q)),
        k(reinterpret_cast<uint16_t *>(lw + w.k)), v(reinterpret_cast<uint16_t *>(lw + w.v)), a(reinterpret_cast<uint16_t *>(lw + w.a)),
        hn(reinterpret_cast<uint16_t *>(lw + w.hn)), act(reinterpret_cast<uint16_t *>(lw + w.act)), h1(reinterpret_cast<float *>(lw + w.h1)),
        angles(reinterpret_cast<float *>(lw + w.angles)), planes(reinterpret_cast<float *>(lw + w.planes)) {}
};

// What refuses a block, whichever kernels would run it
dpara_status check_block(const dpara_shape *shape, const dpara_layer_io *L) {
  if (!L->x || !L->w_qkv || !L->w_o || !L->w_gate_up || !L->w_down || !L->y_f32 || L->hidden <= 0 || L->intermediate <= 0) return DPARA_ERR_INVALID_ARG;
  if ((L->qnorm_w == nullptr) != (L->knorm_w == nullptr)) return DPARA_ERR_INVALID_ARG;
  if (shape->boundary_lo != 0 || shape->boundary_hi != shape->n_boundaries) return DPARA_ERR_UNSUPPORTED;   // (the products behind the attention read every row)
  if (L->hidden % 64 || L->intermediate % 64 || shape->n_q_heads * shape->head_dim % 64) return DPARA_ERR_UNSUPPORTED;
  return DPARA_OK;
}

AngleJob angle_job(const dpara_shape *shape, const dpara_attn_io *io, const dpara_layer_io *L, int M, int R, float *table) {
  AngleJob angles;
  angles.table = table;
  angles.ctx_offsets = io->ctx_offsets; angles.ctx_lens = io->ctx_lens;
  angles.rows = M; angles.per_request = R; angles.slot_rows = shape->n_boundaries * shape->block; angles.block = shape->block;
  angles.half = shape->head_dim / 2;
  for (int d = 0; d < shape->head_dim / 2 && d < 64; ++d) angles.inv_freq[d] = pow((double)L->rope_theta, -2.0 * d / shape->head_dim);
  return angles;
}

dpara_status block_attention(const dpara_shape *shape, const dpara_attn_io *io, const BlockBuffers &B, void *workspace, int32_t *status_word, cudaStream_t st) {
  const int Sq = shape->spine_queries ? shape->n_spine : 0, R = shape->n_boundaries * shape->block + Sq;
  dpara_attn_io aio = *io;
  aio.q = B.q; aio.k_blk = B.k; aio.v_blk = B.v; aio.out = B.a; aio.out_dtype = DPARA_BF16; aio.out_lse = nullptr;
  if (Sq) {
    // the spine's keys/values are the block's own: rows J * Bq .. of each request in the k / v buffers
    const size_t at = (size_t)shape->n_boundaries * shape->block * shape->n_kv_heads * shape->head_dim;
    aio.k_spine = B.k + at;
    aio.v_spine = B.v + at;
  }
  return launch_attention(shape, &aio, workspace, status_word, st, Sq ? R : 0, Sq ? R : 0);
}

// Angles of rows that turn by other frequencies than the blocks before
__global__ void __launch_bounds__(128) angles_kernel(const __grid_constant__ AngleJob A) {
  pdl_wait();
  pdl_launch_dependents();
  angle_block(A, blockIdx.x * kAnglesPerBlock);
}

// A stack of n blocks of few rows: the norm of its input, then chains and attentions in turn.  block(l), ctx(l): block l with its input and outputs, and its context.
// DPARA_ERR_UNSUPPORTED: this device cannot hold a chain's grid at once; the caller's other way adds each product's sums in another order and gives the same up to its roundings.
template <typename Block, typename Ctx>
dpara_status launch_chained(const dpara_shape *shape, const ChainShape &sh, int n, Block block, Ctx ctx, uint8_t *attn_ws, uint8_t *lw, uint32_t *counters,
                            int32_t *status_word, cudaStream_t st) {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < kNumSM) return DPARA_ERR_UNSUPPORTED;
  const int Sq = shape->spine_queries ? shape->n_spine : 0, R = shape->n_boundaries * shape->block + Sq, M = shape->batch * R;
  dpara_layer_io L{}, before = block(0);
  const BlockBuffers B(lw, layer_ws_layout(shape, &before, 0));
  const dpara_attn_io first_io = ctx(0);
  AngleJob start = before.use_rope ? angle_job(shape, &first_io, &before, M, R, B.angles) : AngleJob{};
  start.clear = counters;
  start.n_clear = (n + 1) * kChainCounterWords;
  dpara_status s = launch_rmsnorm<false>(before.x, before.rms1_w, B.xn, M, before.hidden, before.rms_eps, start, st);
  if (s != DPARA_OK) return s;
  bool made = before.use_rope;
  float theta = before.rope_theta;   // what the angles were made for
  for (int l = 0; l <= n; ++l) {
    ChainArgs c{};
    c.M = M; c.hidden = before.hidden; c.intermediate = before.intermediate;
    c.n_q_heads = shape->n_q_heads; c.n_kv_heads = shape->n_kv_heads; c.head_dim = shape->head_dim;
    c.xn = B.xn; c.qkv = B.qkv; c.q = B.q; c.k = B.k; c.v = B.v; c.a = B.a; c.h1 = B.h1; c.hn = B.hn; c.act = B.act;
    c.planes = B.planes; c.counters = counters + (size_t)l * kChainCounterWords;
    if (l > 0) {
      c.tail = 1;
      c.x = before.x; c.w_o = before.w_o; c.rms2_w = before.rms2_w; c.w_gate_up = before.w_gate_up; c.w_down = before.w_down; c.eps2 = before.rms_eps;
      c.y_f32 = l == n ? before.y_f32 : nullptr;   // (between blocks the bf16 rows are all that is read)
      c.y_bf16 = before.y_bf16;
    }
    if (l < n) {
      L = block(l);
      c.head = 1;
      c.rms1_w = L.rms1_w; c.w_qkv = L.w_qkv; c.qnorm_w = L.qnorm_w; c.knorm_w = L.knorm_w; c.eps1 = L.rms_eps; c.use_norm = L.qnorm_w != nullptr;
      if (L.use_rope) {
        c.angles = B.angles;
        if (!made || theta != L.rope_theta) {
          const dpara_attn_io io = ctx(l);
          const AngleJob job = angle_job(shape, &io, &L, M, R, B.angles);
          launch_pdl(angles_kernel, dim3((M * job.half + kAnglesPerBlock - 1) / kAnglesPerBlock), dim3(128), 0, st, job);
          DPARA_CHECK_LAUNCH();
          count_launches(1);
        }
        made = true;
        theta = L.rope_theta;
      }
      before = L;
    }
    s = launch_chain(sh, c, status_word, st);
    if (s != DPARA_OK) return s;
    if (l < n) {
      const dpara_attn_io io = ctx(l);
      s = block_attention(shape, &io, B, attn_ws, status_word, st);
      if (s != DPARA_OK) return s;
    }
  }
  return DPARA_OK;
}
}  // namespace

dpara_status launch_layer(const dpara_shape *shape, const dpara_attn_io *io, const dpara_layer_io *L, void *workspace,
                          int32_t *status_word, cudaStream_t st, bool angles_there, bool allow_chain) {
  const dpara_status refused = check_block(shape, L);
  if (refused != DPARA_OK) return refused;
  const int Sq = shape->spine_queries ? shape->n_spine : 0;
  const int R = shape->n_boundaries * shape->block + Sq;  // rows per request: mask slots, then (if they are queries) the spine
  const int M = shape->batch * R;
  const int H = L->hidden, I = L->intermediate, D = shape->head_dim;
  const int QD = shape->n_q_heads * D, KD = shape->n_kv_heads * D;
  const size_t attn_ws = attention_workspace_bytes(shape, io->host_ctx_offsets);
  // layout: [attention scratch (as sized by attention_workspace_bytes)] [layer buffers] [counters]
  uint8_t *base = static_cast<uint8_t *>(workspace);
  const LayerWs w = layer_ws_layout(shape, L, 0);
  uint8_t *lw = base + attn_ws;
  const ChainShape chain = allow_chain ? block_chain(shape, L, 1) : ChainShape{};
  if (chain.ok) {
    const dpara_status cs = launch_chained(shape, chain, 1, [&](int) { return *L; }, [&](int) { return *io; }, base, lw, reinterpret_cast<uint32_t *>(lw + w.total), status_word, st);
    if (cs != DPARA_ERR_UNSUPPORTED) return cs;
  }
  const BlockBuffers B(lw, w);

  // Few rows: several CTAs for a row of the row-wise kernel behind the QKV product, so that a warp has one or two heads.  They would each work out
  // their row's angles, so the angles are made once, by blocks behind the rows of this norm.  With a CTA per row they are made there, behind nothing (a table
  // of 1152 rows made the first norm 3 us longer: two blocks 1579 -> 1586 us), and up to 16 heads are few enough for one CTA's warps.  What several CTAs save a
  // block of 25, 72, 144, 288 or 429 rows: 2.0 to 5.6 us at 40 heads, 1.5 to 4.0 at 32, 0.1 to 2.4 at 24, 0.3 to 1.6 at 20, -0.3 to 0.7 at 16; at 12, 10 and 8 they
  // lose 0.6 to 0.7 at 429 rows and mostly do not show at the others (-1.1 to 0.7, runs differ by up to 1).
  const int n_heads = shape->n_q_heads + shape->n_kv_heads, per_row = n_heads <= 16 ? 1 : std::min((4 * kNumSM + M - 1) / M, (n_heads + 3) / 4);
  AngleJob angles;
  if (L->use_rope) angles = angle_job(shape, io, L, M, R, per_row > 1 ? B.angles : nullptr);
  dpara_status s = launch_rmsnorm<false>(L->x, L->rms1_w, B.xn, M, H, L->rms_eps, angles_there ? AngleJob{} : angles, st);
  if (s != DPARA_OK) return s;
  GemmArgs g{};
  g.a = B.xn; g.w = L->w_qkv; g.M = M; g.N = QD + 2 * KD; g.K = H; g.epi = 0; g.out = B.qkv; g.w_ready = 1;  // the kernels of this chain write no weights
  s = launch_gemm_tc(g, status_word, st);
  if (s != DPARA_OK) return s;

  QkParams qp;
  qp.qkv = B.qkv; qp.qnorm_w = static_cast<const uint16_t *>(L->qnorm_w); qp.knorm_w = static_cast<const uint16_t *>(L->knorm_w);
  qp.q = B.q; qp.k = B.k; qp.v = B.v;
  qp.Hq = shape->n_q_heads; qp.Hkv = shape->n_kv_heads; qp.D = D;
  qp.use_rope = L->use_rope; qp.use_norm = L->qnorm_w != nullptr; qp.eps = L->rms_eps; qp.angles = angles;
  launch_pdl(per_row > 1 ? qk_norm_rope_kernel<true> : qk_norm_rope_kernel<false>, dim3(M, per_row), dim3(128), D * sizeof(float), st, qp);
  DPARA_CHECK_LAUNCH();
  count_launches(1);

  s = block_attention(shape, io, B, base, status_word, st);
  if (s != DPARA_OK) return s;

  g = GemmArgs{};
  g.a = B.a; g.w = L->w_o; g.M = M; g.N = H; g.K = QD; g.epi = 1; g.resid = L->x; g.resid_bf16 = 1; g.out = B.h1; g.w_ready = 1;
  s = launch_gemm_tc(g, status_word, st);
  if (s != DPARA_OK) return s;
  s = launch_rmsnorm<true>(B.h1, L->rms2_w, B.hn, M, H, L->rms_eps, AngleJob{}, st);
  if (s != DPARA_OK) return s;
  g = GemmArgs{};
  g.a = B.hn; g.w = L->w_gate_up; g.M = M; g.N = I; g.K = H; g.epi = 2; g.out = B.act; g.w_ready = 1;
  s = launch_gemm_tc(g, status_word, st);
  if (s != DPARA_OK) return s;
  g = GemmArgs{};
  g.a = B.act; g.w = L->w_down; g.M = M; g.N = H; g.K = I; g.epi = 1; g.resid = B.h1; g.resid_bf16 = 0; g.out = L->y_f32; g.out_bf16 = L->y_bf16; g.w_ready = 1;
  return launch_gemm_tc(g, status_word, st);
}

// ------------------------------------------------------------------------------------------------ stack of blocks
namespace {
struct BackboneWs { size_t x0, x1, yf, layer, counters, total; };
BackboneWs backbone_ws_layout(const dpara_shape *s, const dpara_backbone_io *bb, size_t attn_bytes) {
  const size_t M = (size_t)s->batch * (s->n_boundaries * s->block + (s->spine_queries ? s->n_spine : 0));
  const size_t H = bb->host_layers[0].hidden;
  BackboneWs w;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t r = o; o += align_up(bytes, 256); return r; };
  w.layer = take(attn_bytes + layer_workspace_bytes(s, &bb->host_layers[0]));  // the attention scratch leads the block's scratch
  w.x0 = take(M * H * 2);
  w.x1 = take(M * H * 2);
  w.yf = take(M * H * 4);
  w.counters = take(counter_bytes(bb->n_layers));
  w.total = o;
  return w;
}
}  // namespace

size_t backbone_workspace_bytes(const dpara_shape *shape, const int64_t *host_ctx_offsets, const dpara_backbone_io *bb) {
  return backbone_ws_layout(shape, bb, attention_workspace_bytes(shape, host_ctx_offsets)).total;
}

dpara_status launch_backbone(const dpara_shape *shape, const dpara_attn_io *io, const dpara_backbone_io *bb, void *workspace,
                             int32_t *status_word, cudaStream_t st) {
  const BackboneWs w = backbone_ws_layout(shape, bb, attention_workspace_bytes(shape, io->host_ctx_offsets));
  uint8_t *base = static_cast<uint8_t *>(workspace);
  void *xbuf[2] = {base + w.x0, base + w.x1};
  const int last = bb->n_layers - 1;
  // block l, with the tensors between blocks in the workspace, and its context
  auto block = [&](int l) {
    dpara_layer_io L = bb->host_layers[l];
    L.x = l == 0 ? bb->host_layers[0].x : xbuf[(l - 1) & 1];
    L.y_f32 = l == last ? bb->host_layers[last].y_f32 : reinterpret_cast<float *>(base + w.yf);
    L.y_bf16 = l == last ? bb->host_layers[last].y_bf16 : xbuf[l & 1];
    return L;
  };
  auto context = [&](int l) {
    dpara_attn_io a = *io;
    a.k_ctx = bb->host_k_ctx[l];
    a.v_ctx = bb->host_v_ctx[l];
    return a;
  };
  const ChainShape chain = block_chain(shape, &bb->host_layers[0], bb->n_layers);
  bool chained = chain.ok;
  for (int l = 0; l <= last && chained; ++l) {
    const dpara_layer_io L = block(l);
    chained = check_block(shape, &L) == DPARA_OK;   // (else it is refused below)
  }
  if (chained) {
    const size_t attn_ws = attention_workspace_bytes(shape, io->host_ctx_offsets);
    const dpara_status s = launch_chained(shape, chain, last + 1, block, context, base + w.layer, base + w.layer + attn_ws, reinterpret_cast<uint32_t *>(base + w.counters),
                                          status_word, st);
    if (s != DPARA_ERR_UNSUPPORTED) return s;
  }
  for (int l = 0; l <= last; ++l) {
    const dpara_layer_io L = block(l);
    const dpara_attn_io a = context(l);
    // (the rows' positions are the same in every block: one table for all blocks that turn by the same frequencies, made by the first that turns)
    const dpara_layer_io *made = l > 0 && bb->host_layers[l - 1].use_rope && bb->host_layers[l - 1].rope_theta == L.rope_theta ? &bb->host_layers[l - 1] : nullptr;
    dpara_status s = launch_layer(shape, &a, &L, base + w.layer, status_word, st, made != nullptr, false);
    if (s != DPARA_OK) return s;
  }
  return DPARA_OK;
}

}  // namespace dpara
