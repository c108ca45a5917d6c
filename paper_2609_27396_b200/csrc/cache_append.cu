// Feature-cache append (Alg. 1, the cache update after the head loop: the verified features of t_0..t_r join the
// cache, the rejected suffix is dropped; App. D: the history is projected incrementally, never again).
//
// Per drafter layer: rmsnorm of the candidate feature rows -> one tensor-core GEMM against the layer's [keys | values]
// projection -> a row-wise kernel that applies the per-head key norm and the rotary embedding at the row's position
// and writes the r + 1 accepted rows of every request behind the filled part of that layer's cache.  One layer's product
// is skinny (a few hundred rows against a 2 Hkv D x F weight: 8 output tiles at the benchmark shape), so with more than
// 128 rows up to eight layers go into ONE grouped launch, their K ranges cut in parts where that evens out the rounds;
// the parts leave fp32 partial sums and ONE row-wise launch for the same layers adds them (rounding the sum to bf16, as
// a single product's bf16 store would).  The accepted
// length is read on the device (it is the output of the verify/select call queued before), so no host round trip
// sits between verification and the append.  All d + 1 candidate rows go through the GEMM: it is bound by reading the
// projection weights once (2 Hkv D x F bf16 per layer), not by the row count.
#include <math.h>

#include <algorithm>

#include "gemm.cuh"
#include "layer.cuh"

namespace dpara {

struct AppendParams {
  const uint16_t *kv;       // no parts: layer g of the launch: [b * J][2 * Hkv * D] bf16, [keys | values] of every candidate row, from kv + g * part_stride
  const float *kv_parts;    // layer g of the launch: [parts][b * J][2 * Hkv * D] fp32 partial sums from kv_parts + g * parts * part_stride
  size_t part_stride;       // elements between two parts (two layers' rows)
  // per layer of the launch (blockIdx.y)
  const uint16_t *knorm_w[kGemmMaxGroups];  // [D] or null
  uint16_t *k_cache[kGemmMaxGroups], *v_cache[kGemmMaxGroups];
  const int64_t *row_start, *capacity, *ctx_len;   // (ctx_len: the copy of the old lengths)
  const int32_t *accept_len;
  int32_t *status_word;
  int64_t *new_len;         // the caller's lengths, to be written by the call's last launch (null: not this one)
  int b, J, Hkv, D, use_rope;
  float eps, theta;
  double inv_freq[64];      // theta^(-2 d / D), d < D / 2, worked out on the host in double precision
};

// One CTA per (candidate row (request n, draft position i), layer of the launch); rows above the accepted length leave at once.  What a row takes is
// round trips to memory, so a thread has all it needs of a head (or of its piece of v) in flight before the first addition: kParts is a template
// argument (0: bf16 rows), a lane owns four neighbouring elements of either half of a key head and D / 8 lanes share the head.
// With 4-byte loads in a loop over a run-time number of parts the launch took 18 us of the 256-row call of five layers.  Whole calls that way -> this way,
// back to back, 256 rows x 5120: 8 parts (one layer) 26.0 -> 19.2 us, 4 (two) 29.3 -> 22.9, 2 (three) 35.3 -> 29.1, 4 (five) 51.9 -> 46.2, 1 (eight)
// 55.7 -> 50.8; bf16 rows, 64 x 4096, five layers 28.1 -> 25.9.  The same bits in all.
template <int kParts>
__global__ void __launch_bounds__(128) append_rows_kernel(const AppendParams P) {
  extern __shared__ float s_cs[];  // cos[D/2], sin[D/2]
  const int n = blockIdx.x / P.J, i = blockIdx.x % P.J, tid = threadIdx.x, g = blockIdx.y;
  // Outcome, length and angles before the wait: the kernel in front is the projection, which writes none of them, and it lets this one
  // go only when everything before it has ended (256 rows, five layers: 57.0 -> 54.5 us).
  const uint16_t *knorm_w = P.knorm_w[g];
  const int r = P.accept_len[n];
  const long long L = P.ctx_len[n];
  const bool fits = r >= 0 && r < P.J && L + r + 1 <= P.capacity[n];
  const int half = P.D / 2;
  if (P.use_rope && fits && i <= r) {
    const double pos = (double)(L + i);
    for (int d = tid; d < half; d += 128) {
      double sn, cs;
      sincos(pos * P.inv_freq[d], &sn, &cs);
      s_cs[d] = (float)cs;
      s_cs[half + d] = (float)sn;
    }
  }
  const size_t row = (size_t)((fits ? P.row_start[n] : 0) + L + i);
  pdl_wait();
  pdl_launch_dependents();
  // L_n += r_n + 1 for the requests that fitted: the old lengths are read from the copy that the call's first kernel made, so nobody is waited for (a kernel of its own
  // behind this one took 2 us of an append; a ticket, the last CTA writing, as much).
  if (P.new_len && blockIdx.x == 0 && g == 0)
    for (int m = tid; m < P.b; m += 128) {
      const int rm = P.accept_len[m];
      const long long Lm = P.ctx_len[m];
      if (rm >= 0 && rm < P.J && Lm + rm + 1 <= P.capacity[m]) P.new_len[m] = Lm + rm + 1;
    }
  if (!fits) {  // does not fit (or no valid outcome): the request is left alone
    if (i == 0 && g == 0 && tid == 0 && P.status_word) atomicOr(reinterpret_cast<unsigned int *>(P.status_word), DPARA_STATUS_CACHE_FULL);
    return;
  }
  if (i > r) return;  // rejected suffix: dropped
  const size_t src = (size_t)blockIdx.x * 2 * P.Hkv * P.D;
  const uint16_t *kv = P.kv + (size_t)g * P.part_stride + src;
  const float *kv_parts = P.kv_parts + (size_t)g * kParts * P.part_stride + src;
  constexpr int kLoads = kParts ? kParts : 1;
  struct Raw { float4 v[kLoads]; };
  // four neighbouring elements: their loads ...
  auto fetch = [&](int e, Raw &raw) {
    if (kParts == 0) {
      const uint2 w = *reinterpret_cast<const uint2 *>(kv + e);
      raw.v[0] = make_float4(bf16lo(w.x), bf16hi(w.x), bf16lo(w.y), bf16hi(w.y));
    } else {
#pragma unroll
      for (int s = 0; s < kLoads; ++s) raw.v[s] = __ldg(reinterpret_cast<const float4 *>(kv_parts + (size_t)s * P.part_stride + e));
    }
  };
  // ... and their values as the bf16 the projection stores (split K: the rounded sum of the parts)
  auto value = [&](const Raw &raw, float (&x)[4]) {
    float4 a = raw.v[0];
#pragma unroll
    for (int s = 1; s < kLoads; ++s) { a.x += raw.v[s].x; a.y += raw.v[s].y; a.z += raw.v[s].z; a.w += raw.v[s].w; }
    const float y[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) x[e] = __bfloat162float(__float2bfloat16_rn(y[e]));
  };
  const int per_head = P.D / 8, sub = tid % per_head, step = 128 / per_head;   // lanes of a head; heads of the CTA at a time
  const int vs = P.Hkv * P.D, d = 4 * sub;
  // the first pieces of v are on their way while the keys are worked on
  Raw va, vb;
  const int c0 = tid * 4;
  if (kParts && c0 < vs) fetch(vs + c0, va);
  if (kParts && c0 + 512 < vs) fetch(vs + c0 + 512, vb);
  for (int h0 = 0; h0 < P.Hkv; h0 += step) {
    const int h = h0 + tid / per_head;
    const bool has = h < P.Hkv;      // (all lanes of a warp take part in the sums, also those behind the last head)
    Raw lo, hi;
    float x1[4] = {}, x2[4] = {};
    if (has) { fetch(h * P.D + d, lo); fetch(h * P.D + half + d, hi); }
    uint2 g1 = make_uint2(0x3f803f80u, 0x3f803f80u), g2 = g1;
    if (knorm_w) { g1 = *reinterpret_cast<const uint2 *>(knorm_w + d); g2 = *reinterpret_cast<const uint2 *>(knorm_w + half + d); }
    if (h0 == 0) __syncthreads();   // (the angles)
    if (has) { value(lo, x1); value(hi, x2); }
    if (knorm_w) {
      // The squares are added as 32 lanes with the elements (l, l + 32) of both halves each would, and then over those lanes in halves:
      // that order decides the last bit of the norm, and with it some keys' rounding to bf16.
      float sum[4];
      if (P.D == 128) {
        const bool low = sub < 8;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float o1 = __shfl_xor_sync(0xffffffffu, x1[e], 8), o2 = __shfl_xor_sync(0xffffffffu, x2[e], 8);
          const float a1[2] = {low ? x1[e] : o1, low ? o1 : x1[e]}, a2[2] = {low ? x2[e] : o2, low ? o2 : x2[e]};
          float ss = 0.f;
#pragma unroll
          for (int k = 0; k < 2; ++k) ss += a1[k] * a1[k] + a2[k] * a2[k];
          sum[e] = ss;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float ss = 0.f;
          ss += x1[e] * x1[e] + x2[e] * x2[e];
          sum[e] = ss;
        }
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int e = 0; e < 4; ++e) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
      const float ss = (sum[0] + sum[2]) + (sum[1] + sum[3]);
      const float rs = rsqrtf(ss / (float)P.D + P.eps);
      const float f1[4] = {bf16lo(g1.x), bf16hi(g1.x), bf16lo(g1.y), bf16hi(g1.y)}, f2[4] = {bf16lo(g2.x), bf16hi(g2.x), bf16lo(g2.y), bf16hi(g2.y)};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        x1[e] = __bfloat162float(__float2bfloat16_rn(x1[e] * rs * f1[e]));
        x2[e] = __bfloat162float(__float2bfloat16_rn(x2[e] * rs * f2[e]));
      }
    }
    float y1[4], y2[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      y1[e] = x1[e]; y2[e] = x2[e];
      if (P.use_rope) {
        // (which product is rounded decides the last bit: written out)
        const float cs = s_cs[d + e], sn = s_cs[half + d + e];
        y1[e] = __fmaf_rn(x1[e], cs, -__fmul_rn(x2[e], sn));
        y2[e] = __fmaf_rn(x1[e], sn, __fmul_rn(x2[e], cs));
      }
    }
    if (has) {
      uint16_t *kd = P.k_cache[g] + (row * P.Hkv + h) * P.D;
      *reinterpret_cast<uint2 *>(kd + d) = make_uint2(pack_bf16(y1[0], y1[1]), pack_bf16(y1[2], y1[3]));
      *reinterpret_cast<uint2 *>(kd + half + d) = make_uint2(pack_bf16(y2[0], y2[1]), pack_bf16(y2[2], y2[3]));
    }
  }
  uint16_t *vd = P.v_cache[g] + row * P.Hkv * P.D;
  if (kParts == 0) {
    for (int c = tid * 8; c < vs; c += 128 * 8) *reinterpret_cast<uint4 *>(vd + c) = *reinterpret_cast<const uint4 *>(kv + vs + c);
    return;
  }
  auto put = [&](int c, const Raw &raw) {
    float x[4];
    value(raw, x);
    *reinterpret_cast<uint2 *>(vd + c) = make_uint2(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]));
  };
  if (c0 < vs) put(c0, va);
  if (c0 + 512 < vs) put(c0 + 512, vb);
  for (int c = c0 + 1024; c < vs; c += 512) {
    fetch(vs + c, va);
    put(c, va);
  }
}

// Layers per grouped launch and K parts per layer for `layers_left` remaining layers; parts = 0: bf16 stores (at most 128 rows: the
// kernel for few rows takes all layers at once, one chain of sums over K each; the whole call, 8 rows, five layers of 2048 x 4096: 192 us with a
// product a layer, 38 now).  The parts are chosen to minimise
// rounds x (K slabs per part + ~8 slabs' worth of fixed cost per work unit) over the CTA pairs.  Fewer are not slower (256 rows, back to back:
// five layers four parts 43.9 us, none 43.8; one layer eight 29.2, none 21.9), but the parts' sums decide the roundings of the keys: other parts flip some of them.
static void cache_group_plan(const dpara_cache_io *io, int layers_left, int *group, int *parts) {
  const int M = io->batch * io->n_rows, N = 2 * io->n_kv_heads * io->head_dim;
  *group = layers_left < kGemmMaxGroups ? layers_left : kGemmMaxGroups;
  *parts = 0;
  if (M <= 128) return;
  const int tiles = ((M + 255) / 256) * ((N + 255) / 256), pairs = kNumSM / 2, nkb = io->feat_dim / 64;
  int best = 1;
  long best_cost = -1;
  for (int s = 1; s <= 8; s *= 2) {
    if (s > 1 && nkb / s < 4) break;
    const long units = (long)*group * tiles * s;
    const long cost = ((units + pairs - 1) / pairs) * (nkb / s + 8);
    if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = s; }
  }
  *parts = best;
}

static void (*append_rows_of(int parts))(AppendParams) {
  switch (parts) {
    case 0: return append_rows_kernel<0>;
    case 1: return append_rows_kernel<1>;
    case 2: return append_rows_kernel<2>;
    case 4: return append_rows_kernel<4>;
    default: return append_rows_kernel<8>;
  }
}

// normalised copies of the feature rows: one per run of layers that share the input norm
static int cache_norm_slots(const dpara_cache_io *io) {
  int slots = 1;
  for (int l = 1; l < io->n_layers; ++l)
    if (io->host_norm_w && io->host_norm_w[l] != io->host_norm_w[l - 1]) ++slots;
  return slots;
}

static size_t lengths_bytes(const dpara_cache_io *io) { return align_up((size_t)io->batch * sizeof(int64_t), 256); }

size_t cache_append_workspace_bytes(const dpara_cache_io *io) {
  const size_t M = (size_t)io->batch * io->n_rows, N = (size_t)2 * io->n_kv_heads * io->head_dim;
  int group, parts;
  cache_group_plan(io, io->n_layers, &group, &parts);
  auto rows_bytes = [&](int layers, int p) { return align_up((size_t)layers * M * N * (p ? 4 * p : 2), 256); };
  size_t rows = rows_bytes(group, parts);
  // (the first launch has the most layers, the last (smaller) one may cut K in more parts: sized for the larger of the two)
  const int rest = io->n_layers % kGemmMaxGroups;
  if (io->n_layers > kGemmMaxGroups && rest) {
    cache_group_plan(io, rest, &group, &parts);
    rows = std::max(rows, rows_bytes(group, parts));
  }
  return (size_t)cache_norm_slots(io) * align_up(M * io->feat_dim * 2, 256) + rows + lengths_bytes(io);
}

dpara_status launch_cache_append(const dpara_cache_io *io, void *workspace, int32_t *status_word, cudaStream_t st) {
  const int M = io->batch * io->n_rows, F = io->feat_dim, N = 2 * io->n_kv_heads * io->head_dim;
  const size_t xn_bytes = align_up((size_t)M * F * 2, 256);
  int group0, parts0;
  cache_group_plan(io, io->n_layers, &group0, &parts0);
  const int slots = cache_norm_slots(io);
  uint8_t *ws = static_cast<uint8_t *>(workspace);
  uint16_t *kv = reinterpret_cast<uint16_t *>(ws + (size_t)slots * xn_bytes);
  int64_t *old_len = reinterpret_cast<int64_t *>(ws + cache_append_workspace_bytes(io) - lengths_bytes(io));   // copied by the first norm
  AppendParams P;
  memset(&P, 0, sizeof(P));
  P.row_start = io->row_start; P.capacity = io->capacity; P.ctx_len = old_len; P.accept_len = io->accept_len;
  P.status_word = status_word;
  P.b = io->batch;
  P.J = io->n_rows; P.Hkv = io->n_kv_heads; P.D = io->head_dim; P.use_rope = io->use_rope;
  P.eps = io->rms_eps; P.theta = io->rope_theta;
  for (int d = 0; d < io->head_dim / 2 && d < 64; ++d) P.inv_freq[d] = pow((double)io->rope_theta, -2.0 * d / io->head_dim);
  P.part_stride = (size_t)M * N;
  const void *prev_gain = nullptr;
  int slot = -1;
  for (int l0 = 0; l0 < io->n_layers;) {
    int group, parts;
    cache_group_plan(io, io->n_layers - l0, &group, &parts);
    GemmArgs g{};
    g.M = M; g.N = N; g.K = F; g.epi = parts ? 3 : 0; g.split_k = parts ? parts : 1; g.n_groups = group; g.one_chain = 1; g.w_ready = 1;  // the kernel in front is this call's norm or row-wise kernel
    for (int k = 0; k < group; ++k) {
      const int l = l0 + k;
      const void *gain = io->host_norm_w ? io->host_norm_w[l] : nullptr;
      if (l == 0 || gain != prev_gain) {  // layers that share the input norm share the normalised rows
        ++slot;
        dpara_status s = launch_rmsnorm_bf16(io->features, gain, ws + (size_t)slot * xn_bytes, M, F, io->rms_eps, st, l == 0 ? io->ctx_len : nullptr, old_len, io->batch);
        if (s != DPARA_OK) return s;
        prev_gain = gain;
      }
      void *out = parts ? static_cast<void *>(reinterpret_cast<float *>(kv) + (size_t)k * parts * M * N) : static_cast<void *>(kv + (size_t)k * M * N);
      if (k == 0) { g.a = ws + (size_t)slot * xn_bytes; g.w = io->host_w_kv[l]; g.out = out; }
      g.a_g[k] = ws + (size_t)slot * xn_bytes; g.w_g[k] = io->host_w_kv[l]; g.out_g[k] = out;
      P.knorm_w[k] = static_cast<const uint16_t *>(io->host_knorm_w ? io->host_knorm_w[l] : nullptr);
      P.k_cache[k] = static_cast<uint16_t *>(io->host_k_ctx[l]);
      P.v_cache[k] = static_cast<uint16_t *>(io->host_v_ctx[l]);
    }
    dpara_status s = launch_gemm_tc(g, status_word, st);
    if (s != DPARA_OK) return s;
    P.kv = kv;
    P.kv_parts = reinterpret_cast<const float *>(kv);
    P.new_len = l0 + group == io->n_layers ? io->ctx_len : nullptr;
    void (*const rows)(AppendParams) = append_rows_of(parts);
    launch_pdl(rows, dim3(M, group), dim3(128), io->head_dim * sizeof(float), st, P);
    DPARA_CHECK_LAUNCH();
    count_launches(1);
    l0 += group;
  }
  return DPARA_OK;
}

}  // namespace dpara

using namespace dpara;

static dpara_status validate_cache(const dpara_cache_io *io) {
  if (!io) return DPARA_ERR_INVALID_ARG;
  if (io->batch <= 0 || io->n_rows <= 0 || io->feat_dim <= 0 || io->n_kv_heads <= 0 || io->n_layers <= 0) return DPARA_ERR_INVALID_ARG;
  if (io->head_dim != 64 && io->head_dim != 128) return DPARA_ERR_UNSUPPORTED;
  if (io->feat_dim % 64 != 0) return DPARA_ERR_UNSUPPORTED;
  return DPARA_OK;
}

extern "C" size_t dpara_cache_append_workspace_bytes(const dpara_cache_io *io) {
  return validate_cache(io) == DPARA_OK ? cache_append_workspace_bytes(io) : 0;
}

extern "C" dpara_status dpara_cache_append(const dpara_cache_io *io, void *workspace, size_t workspace_bytes, int32_t *status_word,
                                           void *stream) {
  dpara_status s = validate_cache(io);
  if (s != DPARA_OK) return s;
  if (!io->features || !io->accept_len || !io->host_w_kv || !io->host_k_ctx || !io->host_v_ctx || !io->row_start || !io->capacity ||
      !io->ctx_len)
    return DPARA_ERR_INVALID_ARG;
  for (int l = 0; l < io->n_layers; ++l)
    if (!io->host_w_kv[l] || !io->host_k_ctx[l] || !io->host_v_ctx[l] || !aligned16(io->host_w_kv[l]) || !aligned16(io->host_k_ctx[l]) ||
        !aligned16(io->host_v_ctx[l]) || (io->host_norm_w && !aligned16(io->host_norm_w[l])) || (io->host_knorm_w && !aligned16(io->host_knorm_w[l])))
      return DPARA_ERR_INVALID_ARG;
  if (!aligned16(io->features)) return DPARA_ERR_INVALID_ARG;
  if (!workspace || workspace_bytes < cache_append_workspace_bytes(io) || !aligned16(workspace)) return DPARA_ERR_WORKSPACE;
  return launch_cache_append(io, workspace, status_word, static_cast<cudaStream_t>(stream));
}
