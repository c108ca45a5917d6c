// What lies between two attentions of a stack of blocks, for few rows, in ONE launch:
//   O product (+x) -> RMS norm -> gate/up product, SiLU * up -> down product (+h1) -> RMS norm -> QKV product -> per-head norm + rotary embedding.
//
// With few rows each of these steps is a pass over its weights, or nothing but round trips, and a step reads what all SMs wrote in the step before.  As eight
// kernels a block of a small model was launches, set-up and tails (~7 us a kernel), and one of a large model had HBM idle around each of its products.  Here the
// CTAs are persistent (one per SM, cooperative launch) and the steps are separated by counters in memory: ~3 us from a product's last sum to the next one's first
// product, ~7 with a row step in between, and the warp that streams WEIGHTS does not wait for a step: behind its own CTA's sums it goes on to the next product's.
//   * Every product is one round: a CTA has one tile (R <= 128 weight rows, any multiple of 4; gate/up: R gate and R up rows) and one part of K, so
//     tiles are cut to fill the SMs (4096 columns of K 12288: 49 tiles x 3 parts on 148 SMs).
//   * Parts of K leave fp32 sums in planes [part][row][column]; the row step behind the product adds them in the order of the parts,
//     whatever the timing.  No clusters and no exchange through shared memory: those rows have to be read back for their norm anyway.
//   * Activations have a ring and a warp of their own (they wait for the step before; the weights do not).  A slab of them is read for every slab of weights (half as many
//     bytes in gate/up) and takes ~1.1 us on its way.
// Warps: 0-15 sums, row steps (short chains of dependent instructions: eight warps took twice as long); 16 weights; 17 activations; 18 and 19 products (weights
// as the rows, M = 128; activation rows as the columns).  A stage is two operands of weights, gate and up of one slab of K or two slabs in turn, and each of the two warps has one
// of them and an accumulator of its own (two slabs: the sums are added at the end): a single warp took ~750 clocks per stage, two take 500 to 700.
// Measured, whole stacks of blocks, kernels of their own -> this (us): five blocks of 72 rows, hidden 4096 (386 MB of weights each) 592 -> 584; three blocks of 64 to 128 rows: hidden 512
// 151 -> 130 and 169 -> 144, 1024 184 -> 172 and 193 -> 179, 2048 209 -> 201 and 266 -> 256, 3072 257 -> 245, 5120 407 -> 392 and 507 -> 480.  A block of 72 rows of hidden 4096 is
// 60 us of HBM; the rest is the attention (16), ~4 around it (a cooperative launch does not start ahead of the end of the kernel in front), and the four times that HBM
// waits for a step.  Tried: asking for the next product's weights in L2 while the ring is full, at once or one stage each 0.5 us, and for the O product's while the attention runs
// (the row steps, or the attention, get longer by what the product wins); parts of K that start at different slabs in different tiles (no change: the activations are not what a stage waits
// for); weights of the next product while others still work on this one (the slowest CTA sets the pace).
// Beside another stream the wait for all SMs shows: six stacks of five blocks of 72 rows beside six passes of library products that read 1 GB of weights (us alone, the other's alone,
// both together): hidden 4096 3479, 1247, 4806 (kernels of their own 3638, 1242, 4661), 2048 2100, 1256, 3431 (2296, 1248, 3245), 512 1358, 1248, 2526 (1611, 1242, 2518); beside small
// products (64 x 1024 x 4096) 5602, 4244 and 3436 (5365, 4121, 3551).  Short kernels of another stream wait for a chain's end: twelve runs of six scans of one CTA done after 2890, 1728 and 1182
// (1121, 708, 705).  Which call takes the chain: layer.cu.
// All waits are bounded by wall time and give up with DPARA_STATUS_TIMEOUT; the launch is cooperative, so all CTAs are resident.
#include "chain.cuh"
#include "gemm.cuh"
#include "sm100_ptx.cuh"

namespace dpara {
using namespace ptx;

namespace {
constexpr int kThreads = 640, kEpiThreads = 512, kEpiWarps = kEpiThreads / 32;
constexpr int kWeightWarp = 16, kActWarp = 17, kMmaWarp = 18;   // (18 and 19)
constexpr int kSlabK = 64;                 // K columns per slab (one 128-byte swizzle row)
constexpr int kMaxWStages = 8, kMaxASlots = 4;
constexpr int kSmemMax = 227 * 1024;
constexpr int kBarBytes = 1024;
constexpr int kMaxSplit = 8;
constexpr int kHeld = (kChainHidden + 4 * kEpiThreads - 1) / (4 * kEpiThreads);   // groups of four elements of a row that a thread holds
constexpr int kAccCols = 256;              // TMEM columns of one accumulator buffer
enum { kO = 0, kGateUp = 1, kDown = 2, kQkv = 3, kProducts = 4 };
// counters: CTAs that are through with ...
enum { kCountO = 0, kCountNorm2 = 1, kCountGateUp = 2, kCountDown = 3, kCountRow = 4, kCountQkv = 5 };
}  // namespace

struct ChainProduct {
  int N, rows, tiles, split, units;
  int stages;        // of the whole K range: two slabs of K each, gate/up: one
};

// Read from a copy in shared memory: a line of the parameter bank costs a step ~700 clocks when it is first met.
struct ChainInfo {
  ChainProduct p[kProducts];
  int tail, head;
  int M, T, H, I, n_q, n_kv, D;
  int use_norm;
  float eps1, eps2;
  int op_bytes, w_stages, a_slots, on_way;
  const uint16_t *x, *rms2_w, *rms1_w, *qnorm_w, *knorm_w;
  float *h1, *y_f32;
  uint16_t *hn, *act, *y_bf16, *xn, *qkv, *q, *k, *v;
  const float *angles;
  float *planes;
  uint32_t *counters;
  int32_t *status;
};
struct ChainParams {
  CUtensorMap map_w[kProducts], map_a[kProducts];
  ChainInfo info;
  int bar_offset;
};
static_assert(kChainRows <= kNumSM, "a row step has a CTA for each row");
constexpr int kInfoWords = sizeof(ChainInfo) / 4;
static_assert(kInfoWords <= kThreads && sizeof(ChainInfo) + 512 <= kBarBytes, "");

__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

// Waits (the whole warp) until `count` CTAs have signalled; what they wrote before is then visible, to the asynchronous proxy too.
__device__ __forceinline__ bool wait_count(const uint32_t *counter, uint32_t count, volatile int *abort_flag, int site) {
  uint64_t t0 = 0;
  for (unsigned int tries = 0;; ++tries) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    if (__all_sync(0xffffffffu, v >= count)) break;
    if (tries == 0) t0 = global_timer_ns();
    if (tries % 64 == 63 && __any_sync(0xffffffffu, *abort_flag || global_timer_ns() - t0 > kWaitLimitNs)) {
      if (*abort_flag == 0) *abort_flag = site;
      return false;
    }
  }
  fence_async_global();
  return true;
}

// Barrier 1 among the 512 threads of the sums' and row steps' warps; `live` is true behind it where it was in all of them.
__device__ __forceinline__ bool epi_bar_all(bool live) {
  uint32_t all;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "barrier.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(all) : "r"((uint32_t)live), "n"(kEpiThreads) : "memory");
  return all != 0;
}
// (those threads; the reader orders its bulk copies behind what it has seen)
__device__ __forceinline__ void signal_count(uint32_t *counter) {
  named_bar_sync(1, kEpiThreads);
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
}

// A row step: v = residual + the sum of the row's parts; kept as fp32 and / or bf16, and normalised (of the bf16 values where `rounded`).  The step is
// round trips to L2, so what does not depend on the product in front, residual and gain, is read ahead of the wait for it, and the parts are
// in flight together.
struct RowStep {
  float4 resid[kHeld];
  uint2 gain[kHeld];
  template <bool kBf16Resid>
  __device__ __forceinline__ void read(const void *residual, const uint16_t *gains, int row, int H) {
#pragma unroll
    for (int i = 0; i < kHeld; ++i) {
      const int c = 4 * threadIdx.x + i * 4 * kEpiThreads;
      resid[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      gain[i] = make_uint2(0x3f803f80u, 0x3f803f80u);   // (no gain: bf16 ones)
      if (c < H) {
        if (kBf16Resid) {
          const uint2 b = *reinterpret_cast<const uint2 *>(static_cast<const uint16_t *>(residual) + (size_t)row * H + c);
          resid[i] = make_float4(bf16lo(b.x), bf16hi(b.x), bf16lo(b.y), bf16hi(b.y));
        } else {
          resid[i] = __ldcg(reinterpret_cast<const float4 *>(static_cast<const float *>(residual) + (size_t)row * H + c));
        }
        if (gains) gain[i] = *reinterpret_cast<const uint2 *>(gains + c);
      }
    }
  }
};
__device__ __forceinline__ void row_step(const RowStep &R, const float *planes, size_t plane, int parts, int row, int H, float *out_f32, uint16_t *out_bf16, bool rounded,
                                         float eps, uint16_t *normed, float *s_red) {
  const int tid = threadIdx.x;
  const size_t base = (size_t)row * H;
  const float *src = planes + base + 4 * tid;
  float4 v[kHeld];
  // four parts in flight, then three at a time
#pragma unroll
  for (int i = 0; i < kHeld; ++i)
    if (4 * tid + i * 4 * kEpiThreads < H) v[i] = __ldcg(reinterpret_cast<const float4 *>(src + i * 4 * kEpiThreads));
#pragma unroll 1
  for (int left = parts - 1; left > 0; left -= 3, src += 3 * plane) {
    float4 x[3][kHeld];
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
      for (int i = 0; i < kHeld; ++i)
        if (s < left && 4 * tid + i * 4 * kEpiThreads < H) x[s][i] = __ldcg(reinterpret_cast<const float4 *>(src + (s + 1) * plane + i * 4 * kEpiThreads));
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
      for (int i = 0; i < kHeld; ++i)
        if (s < left && 4 * tid + i * 4 * kEpiThreads < H) { v[i].x += x[s][i].x; v[i].y += x[s][i].y; v[i].z += x[s][i].z; v[i].w += x[s][i].w; }
  }
  float ss = 0.f;
#pragma unroll
  for (int i = 0; i < kHeld; ++i) {
    const int c = 4 * tid + i * 4 * kEpiThreads;
    if (c >= H) continue;
    v[i].x += R.resid[i].x; v[i].y += R.resid[i].y; v[i].z += R.resid[i].z; v[i].w += R.resid[i].w;
    if (out_f32) *reinterpret_cast<float4 *>(out_f32 + base + c) = v[i];
    const uint2 b = make_uint2(pack_bf16(v[i].x, v[i].y), pack_bf16(v[i].z, v[i].w));
    if (out_bf16) *reinterpret_cast<uint2 *>(out_bf16 + base + c) = b;
    if (rounded) v[i] = make_float4(bf16lo(b.x), bf16hi(b.x), bf16lo(b.y), bf16hi(b.y));
    ss = fmaf(v[i].x, v[i].x, ss); ss = fmaf(v[i].y, v[i].y, ss); ss = fmaf(v[i].z, v[i].z, ss); ss = fmaf(v[i].w, v[i].w, ss);
  }
  if (!normed) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((tid & 31) == 0) s_red[tid >> 5] = ss;
  named_bar_sync(1, kEpiThreads);
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < kEpiWarps; ++w) tot += s_red[w];
  const float rs = rsqrtf(tot / (float)H + eps);
#pragma unroll
  for (int i = 0; i < kHeld; ++i) {
    const int c = 4 * tid + i * 4 * kEpiThreads;
    if (c < H)
      *reinterpret_cast<uint2 *>(normed + base + c) =
          make_uint2(pack_bf16(v[i].x * rs * bf16lo(R.gain[i].x), v[i].y * rs * bf16hi(R.gain[i].x)), pack_bf16(v[i].z * rs * bf16lo(R.gain[i].y), v[i].w * rs * bf16hi(R.gain[i].y)));
  }
}

// Per-head RMS norm (rounded to bf16) and rotary embedding of the rows' q and k heads, v heads as they are.  A warp takes kAtOnce heads of rows at a time; a
// lane owns the element pairs (2 lane, 2 lane + 1) of both halves of a head.  Where the first ones go, their gains and their angles are worked out ahead of the wait.
constexpr int kAtOnce = 2;
struct HeadUnit {
  uint16_t *dst;       // null: no unit
  uint32_t g1, g2;
  float2 cs, sn;
  bool turned, normed;
  __device__ __forceinline__ void read(const ChainInfo &P, int u, int lane) {
    const int heads = P.n_q + 2 * P.n_kv, row = u / heads, hd = u - row * heads, half = P.D / 2;
    dst = nullptr;
    g1 = g2 = 0x3f803f80u;   // bf16 1.0 twice
    cs = make_float2(1.f, 1.f);
    sn = make_float2(0.f, 0.f);
    const bool is_q = hd < P.n_q, is_v = hd >= P.n_q + P.n_kv;
    turned = !is_v && P.angles;
    normed = !is_v && P.use_norm;
    if (row >= P.M || 2 * lane >= half) return;
    dst = (is_q ? P.q + (row * P.n_q + hd) * P.D : is_v ? P.v + (row * P.n_kv + hd - P.n_q - P.n_kv) * P.D : P.k + (row * P.n_kv + hd - P.n_q) * P.D) + 2 * lane;
    const uint16_t *gain = is_q ? P.qnorm_w : P.knorm_w;
    if (normed && gain) {
      g1 = *reinterpret_cast<const uint32_t *>(gain + 2 * lane);
      g2 = *reinterpret_cast<const uint32_t *>(gain + half + 2 * lane);
    }
    if (turned) {
      const float *t = P.angles + row * P.D + 2 * lane;
      cs = *reinterpret_cast<const float2 *>(t);
      sn = *reinterpret_cast<const float2 *>(t + half);
    }
  }
};
struct HeadStep {
  HeadUnit u[kAtOnce];
  __device__ __forceinline__ void read(const ChainInfo &P, int u0, int stride, int lane) {
#pragma unroll
    for (int c = 0; c < kAtOnce; ++c) u[c].read(P, u0 + c * stride, lane);
  }
};
__device__ __forceinline__ void head_step(HeadStep &S, const ChainInfo &P, int first, int stride, int lane) {
  const int D = P.D, half = D / 2, units = P.M * (P.n_q + 2 * P.n_kv), parts = P.p[kQkv].split, plane = P.M * P.p[kQkv].N;
  const float inv = 1.f / (float)D, eps = P.eps1;
  const float *const planes = P.planes + 2 * lane;
  uint16_t *const raw = P.qkv + 2 * lane;
#pragma unroll 1
  for (int u0 = first; u0 < units; u0 += kAtOnce * stride) {
    if (u0 != first) S.read(P, u0, stride, lane);
    float2 lo[kAtOnce], hi[kAtOnce];
#pragma unroll
    for (int c = 0; c < kAtOnce; ++c) lo[c] = hi[c] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int s0 = 0; s0 < parts; s0 += 4) {
      float2 a[kAtOnce][4], b[kAtOnce][4];
#pragma unroll
      for (int c = 0; c < kAtOnce; ++c) {
        const float *const src = planes + s0 * plane + (u0 + c * stride) * D;   // (a row is its heads)
#pragma unroll
        for (int s = 0; s < 4; ++s)
          if (S.u[c].dst && s0 + s < parts) {
            a[c][s] = __ldcg(reinterpret_cast<const float2 *>(src + s * plane));
            b[c][s] = __ldcg(reinterpret_cast<const float2 *>(src + s * plane + half));
          } else {
            a[c][s] = b[c][s] = make_float2(0.f, 0.f);
          }
      }
#pragma unroll
      for (int c = 0; c < kAtOnce; ++c)
#pragma unroll
        for (int s = 0; s < 4; ++s) { lo[c].x += a[c][s].x; lo[c].y += a[c][s].y; hi[c].x += b[c][s].x; hi[c].y += b[c][s].y; }
    }
    uint32_t l16[kAtOnce], h16[kAtOnce];
    float ss[kAtOnce];
#pragma unroll
    for (int c = 0; c < kAtOnce; ++c) {
      l16[c] = pack_bf16(lo[c].x, lo[c].y);
      h16[c] = pack_bf16(hi[c].x, hi[c].y);
      const float x0 = bf16lo(l16[c]), x1 = bf16hi(l16[c]), y0 = bf16lo(h16[c]), y1 = bf16hi(h16[c]);
      ss[c] = x0 * x0 + y0 * y0 + x1 * x1 + y1 * y1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int c = 0; c < kAtOnce; ++c) ss[c] += __shfl_xor_sync(0xffffffffu, ss[c], o);
#pragma unroll
    for (int c = 0; c < kAtOnce; ++c) {
      const HeadUnit &U = S.u[c];
      if (!U.dst) continue;
      uint32_t y1 = l16[c], y2 = h16[c];
      uint16_t *const r = raw + (u0 + c * stride) * D;
      *reinterpret_cast<uint32_t *>(r) = y1;
      *reinterpret_cast<uint32_t *>(r + half) = y2;
      if (U.normed) {
        const float rs = rsqrtf(ss[c] * inv + eps);
        y1 = pack_bf16(bf16lo(y1) * rs * bf16lo(U.g1), bf16hi(y1) * rs * bf16hi(U.g1));
        y2 = pack_bf16(bf16lo(y2) * rs * bf16lo(U.g2), bf16hi(y2) * rs * bf16hi(U.g2));
      }
      if (U.turned) {
        const float a0 = bf16lo(y1), a1 = bf16hi(y1), b0 = bf16lo(y2), b1 = bf16hi(y2);
        y1 = pack_bf16(a0 * U.cs.x - b0 * U.sn.x, a1 * U.cs.y - b1 * U.sn.y);
        y2 = pack_bf16(b0 * U.cs.x + a0 * U.sn.x, b1 * U.cs.y + a1 * U.sn.y);
      }
      *reinterpret_cast<uint32_t *>(U.dst) = y1;
      *reinterpret_cast<uint32_t *>(U.dst + half) = y2;
    }
  }
}

// Stages of the CTA's part of a product's K range.
struct StageRange {
  int from, to;
  __device__ __forceinline__ StageRange(const ChainProduct &p, int cta) {
    const int part = cta / p.tiles;
    from = part * p.stages / p.split;
    to = (part + 1) * p.stages / p.split;
  }
};

__global__ void __launch_bounds__(kThreads, 1) chain_kernel(const __grid_constant__ ChainParams args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *w_full = reinterpret_cast<uint64_t *>(smem + args.bar_offset), *w_empty = w_full + kMaxWStages, *a_full = w_empty + kMaxWStages,
           *a_empty = a_full + kMaxASlots, *acc_full = a_empty + kMaxASlots, *w_go = acc_full + 1;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(w_go + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  float *s_red = reinterpret_cast<float *>(tmem_slot + 4);
  const ChainInfo &P = *reinterpret_cast<const ChainInfo *>(smem + args.bar_offset + 512);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x < kInfoWords) reinterpret_cast<uint32_t *>(smem + args.bar_offset + 512)[threadIdx.x] = reinterpret_cast<const uint32_t *>(&args.info)[threadIdx.x];
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxWStages; ++s) { mbar_init(w_full + s, 1); mbar_init(w_empty + s, 2); }
    for (int s = 0; s < kMaxASlots; ++s) { mbar_init(a_full + s, 1); mbar_init(a_empty + s, 2); }
    mbar_init(acc_full, 2);
    mbar_init(w_go, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kMmaWarp) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const int stage_bytes = 2 * P.op_bytes, a_off = P.w_stages * stage_bytes, a_bytes = P.T * 128;
  const int first = P.tail ? kO : kQkv, end = P.head ? kProducts : kQkv;
  const int cta = blockIdx.x;
  const uint32_t row_ctas = (uint32_t)P.M;   // CTAs that have a row

  if (warp == kWeightWarp) {
    // ------------------------------------------------------------------ weights: no kernel of this call writes them, no wait at all
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int g = first; g < end; ++g) prefetch_tensormap(&args.map_w[g]);
    int done = 0;   // products of this CTA whose weights have been asked for
    int oldest = 0, out = 0;   // stages on their way: the first of them, how many
    uint32_t oldest_ph = 0;
#pragma unroll 1
    for (int g = first; g < end && ok; ++g) {
      const ChainProduct &p = P.p[g];
      if (cta >= p.units) continue;
      const CUtensorMap *map = &args.map_w[g];
      const int wrow = cta % p.tiles * p.rows, n_w = P.w_stages, op_bytes = P.op_bytes;
      const uint32_t tx = (uint32_t)(p.rows * 256);
      const bool gated = g == kGateUp;
      const StageRange range(p, cta);
      // Not while other CTAs still need the bandwidth for the product in front, nor ahead of this one's sums.
      if (done) ok = __all_sync(0xffffffffu, mbar_wait(w_go, (done & 1) ^ 1u, abort_flag, 14));
#pragma unroll 1
      for (int k = range.from; k < range.to && ok; ++k) {
        // Not more on their way than HBM needs to be busy: what queues there is in front of the sums, the rows and the counters too.
        if (out == P.on_way) {
          ok = __all_sync(0xffffffffu, mbar_wait(w_full + oldest, oldest_ph, abort_flag, 16));
          if (!ok) break;
          --out;
          if (++oldest == n_w) { oldest = 0; oldest_ph ^= 1u; }
        }
        ok = __all_sync(0xffffffffu, mbar_wait(w_empty + stage, ph ^ 1u, abort_flag, 2));
        if (!ok) break;
        ++out;
        if (elect_one()) {
          uint8_t *dst = smem + stage * stage_bytes;
          mbar_arrive_expect_tx(w_full + stage, tx);
          tma_load_2d(dst, map, w_full + stage, gated ? k * kSlabK : 2 * k * kSlabK, wrow);
          tma_load_2d(dst + op_bytes, map, w_full + stage, gated ? k * kSlabK : (2 * k + 1) * kSlabK, gated ? p.N + wrow : wrow);
        }
        __syncwarp();
        if (++stage == n_w) { stage = 0; ph ^= 1u; }
      }
      ++done;
    }
  } else if (warp == kActWarp) {
    // ------------------------------------------------------------------ activations, behind the step that makes them
    int slot = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int g = first; g < end; ++g) prefetch_tensormap(&args.map_a[g]);
    pdl_wait();
    pdl_launch_dependents();
#pragma unroll 1
    for (int g = first; g < end && ok; ++g) {
      const ChainProduct &p = P.p[g];
      if (cta >= p.units) continue;
      const StageRange range(p, cta);
      const bool gated = g == kGateUp;
      if (g == kGateUp) ok = wait_count(P.counters + 32 * kCountNorm2, row_ctas, abort_flag, 3);
      else if (g == kDown) ok = wait_count(P.counters + 32 * kCountGateUp, (uint32_t)P.p[kGateUp].units, abort_flag, 4);
      else if (g == kQkv && P.tail) ok = wait_count(P.counters + 32 * kCountRow, row_ctas, abort_flag, 5);
#pragma unroll 1
      for (int k = range.from; k < range.to && ok; ++k) {
        ok = __all_sync(0xffffffffu, mbar_wait(a_empty + slot, ph ^ 1u, abort_flag, 6));
        if (!ok) break;
        if (elect_one()) {
          uint8_t *dst = smem + a_off + slot * 2 * a_bytes;
          mbar_arrive_expect_tx(a_full + slot, (uint32_t)(gated ? a_bytes : 2 * a_bytes));
          tma_load_2d(dst, &args.map_a[g], a_full + slot, gated ? k * kSlabK : 2 * k * kSlabK, 0);
          if (!gated) tma_load_2d(dst + a_bytes, &args.map_a[g], a_full + slot, (2 * k + 1) * kSlabK, 0);
        }
        __syncwarp();
        if (++slot == P.a_slots) { slot = 0; ph ^= 1u; }
      }
    }
  } else if (warp >= kMmaWarp) {
    // ------------------------------------------------------------------ products (the whole warp walks and waits, one lane issues in straight lines)
    const uint32_t idesc = idesc_bf16_f32(128, P.T, false, false);
    const uint64_t desc = smem_desc_sw128(smem_u32(smem), 16, 1024);
    const uint32_t w_lo = (uint32_t)desc, a_lo = w_lo + ((uint32_t)a_off >> 4), hi = (uint32_t)(desc >> 32);
    const uint32_t stage_units = (uint32_t)stage_bytes >> 4, op_units = (uint32_t)P.op_bytes >> 4, a_units = (uint32_t)a_bytes >> 4;
    const uint32_t op = warp - kMmaWarp;
    int stage = 0, slot = 0, done = 0;
    uint32_t w_ph = 0, a_ph = 0;
    bool ok = true;
#pragma unroll 1
    for (int g = first; g < end && ok; ++g) {
      const ChainProduct &p = P.p[g];
      if (cta >= p.units) continue;
      const StageRange range(p, cta);
      const int n = range.to - range.from;
      // (two buffers in turn; the one before the last was read before the counters let this product's activations through)
      const uint32_t acc = tmem + (done & 1) * kAccCols + op * P.T, a_op = g == kGateUp ? 0 : op * a_units;
      const int n_w = P.w_stages, n_a = P.a_slots;
      bool w_there = false, a_there = false;
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        if (!__all_sync(0xffffffffu, w_there)) ok = __all_sync(0xffffffffu, mbar_wait(w_full + stage, w_ph, abort_flag, 7));
        if (!__all_sync(0xffffffffu, a_there)) ok = __all_sync(0xffffffffu, mbar_wait(a_full + slot, a_ph, abort_flag, 8)) && ok;
        if (!ok) break;
        const uint32_t wo = w_lo + stage * stage_units + op * op_units, ao = a_lo + slot * 2 * a_units + a_op;
        const int w_cur = stage, a_cur = slot;
        if (++stage == n_w) { stage = 0; w_ph ^= 1u; }
        if (++slot == n_a) { slot = 0; a_ph ^= 1u; }
        w_there = mbar_test(w_full + stage, w_ph);
        a_there = mbar_test(a_full + slot, a_ph);
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) mma_ss_lo(acc, wo + 2 * kk, ao + 2 * kk, hi, idesc, kk != 0 || i != 0);
          mma_commit(a_empty + a_cur);
          mma_commit(w_empty + w_cur);
        }
        __syncwarp();
      }
      if (ok && elect_one()) mma_commit(acc_full);
      __syncwarp();
      ++done;
    }
  } else {
    // ------------------------------------------------------------------ sums of the products, row steps
    pdl_wait();
    const int quarter = warp & 3, nh = warp >> 2;   // the TMEM lanes this warp may read; every fourth 8 activation rows
    int done = 0;
    bool live = true;
    // A product's sums into its plane (gate/up: the gated activations)
    auto sums = [&](int g) {
      const ChainProduct &p = P.p[g];
      if (cta >= p.units) return;
      const int tile = cta % p.tiles, part = cta / p.tiles, at = quarter * 32 + lane, col = tile * p.rows + at, M = P.M, N = p.N;
      const bool in = at < p.rows && col < N;
      uint32_t taddr = tmem + (done & 1) * kAccCols + ((uint32_t)(quarter * 32) << 16) + nh * 8;
      float *dst = P.planes + (part * M + nh * 8) * N + col;
      uint16_t *dst16 = P.act + nh * 8 * N + col;
      const uint32_t up = (uint32_t)P.T;
      live = epi_bar_all(warp != 0 || __all_sync(0xffffffffu, mbar_wait(acc_full, done & 1, abort_flag, 10)));
      if (!live) return;
      tc_fence_after();
      ++done;
      if (g == kGateUp) {
#pragma unroll 1
        for (int left = M - nh * 8; left > 0; left -= 32, taddr += 32, dst16 += 32 * N) {
          uint32_t r[8], u[8];
          tmem_ld8(taddr, r);
          tmem_ld8(taddr + up, u);
          tmem_wait_ld();
          if (in) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (j < left) dst16[j * N] = (uint16_t)pack_bf16(silu(__uint_as_float(r[j])) * __uint_as_float(u[j]), 0.f);
          }
        }
      } else {
#pragma unroll 1
        for (int left = M - nh * 8; left > 0; left -= 32, taddr += 32, dst += 32 * N) {
          uint32_t r[8], u[8];
          tmem_ld8(taddr, r);
          tmem_ld8(taddr + up, u);
          tmem_wait_ld();
          if (in) {
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (j < left) dst[j * N] = __uint_as_float(r[j]) + __uint_as_float(u[j]);
          }
        }
      }
      tc_fence_before();
      signal_count(P.counters + 32 * (g == kO ? kCountO : g == kGateUp ? kCountGateUp : g == kDown ? kCountDown : kCountQkv));
      if (threadIdx.x == 0) mbar_arrive(w_go);
    };
    auto wait_all = [&](int counter, int count, int site) {
      live = epi_bar_all(warp != 0 || wait_count(P.counters + 32 * counter, (uint32_t)count, abort_flag, site));
    };
    const size_t plane = (size_t)P.M * P.H;
    if (P.tail) {
      sums(kO);
      RowStep R;
      if (live && cta < P.M) {
        R.read<true>(P.x, P.rms2_w, cta, P.H);
        wait_all(kCountO, P.p[kO].units, 11);
        if (live) {
          row_step(R, P.planes, plane, P.p[kO].split, cta, P.H, P.h1, nullptr, false, P.eps2, P.hn, s_red);
          signal_count(P.counters + 32 * kCountNorm2);
        }
      }
      if (live) sums(kGateUp);
      if (live) sums(kDown);
      if (live && cta < P.M) {
        R.read<false>(P.h1, P.head ? P.rms1_w : nullptr, cta, P.H);
        wait_all(kCountDown, P.p[kDown].units, 12);
        if (live) {
          row_step(R, P.planes, plane, P.p[kDown].split, cta, P.H, P.y_f32, P.y_bf16, true, P.eps1, P.head ? P.xn : nullptr, s_red);
          if (P.head) signal_count(P.counters + 32 * kCountRow);
        }
      }
    }
    if (P.head && live) {
      sums(kQkv);
      if (live) {
        HeadStep S;
        const int unit = cta * kEpiWarps + warp, stride = (int)gridDim.x * kEpiWarps;
        S.read(P, unit, stride, lane);
        wait_all(kCountQkv, P.p[kQkv].units, 13);
        if (live) head_step(S, P, unit, stride, lane);
      }
    }
  }
  // ------------------------------------------------------------------ teardown
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      if (P.status) atomicOr(reinterpret_cast<unsigned int *>(P.status), DPARA_STATUS_TIMEOUT);
#pragma unroll 1
      for (int k = 0; k < 4096; ++k) __nanosleep(256);  // copies that may still be in flight get a bounded time to land
    }
    __syncthreads();
  }
  if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------------------ host
namespace {
// The cheapest tiles of a product in one round.  In ns: stages of a part x the longest of: its weights from HBM (6300 bytes per ns over all SMs that
// have a tile, 42 for one), its products, its bytes from L2; and the planes' way to L2 and back.
ChainTiles chain_tiles(int M, int T, int N, int K, bool gated) {
  ChainTiles best{0, 0, 0};
  double best_cost = 0;
  const int stages = gated ? (K + kSlabK - 1) / kSlabK : (K + 2 * kSlabK - 1) / (2 * kSlabK);
  for (int split = 1; split <= (gated ? 1 : kMaxSplit) && split <= stages; ++split) {
    const int most = kNumSM / split;
    int rows = ((N + most - 1) / most + 3) / 4 * 4;
    if (rows > 128) continue;
    if (rows < 16) rows = 16;
    const int tiles = (N + rows - 1) / rows, units = tiles * split;
    double stage = 2.0 * (130.0 + 0.55 * T);
    const double w = rows * 256.0, a = T * 128.0 * (gated ? 1 : 2);
    for (double other : {w / 42.0, w * units / 6300.0, (w + a) * units / 12000.0})
      if (other > stage) stage = other;
    const double cost = (stages + split - 1) / split * stage + (gated ? 0.0 : 8.0 * split * M * N / 6000.0 + 100.0 * split);
    if (best.rows == 0 || cost < best_cost) { best = ChainTiles{rows, tiles, split}; best_cost = cost; }
  }
  return best;
}
}  // namespace

ChainShape chain_shape(int M, int hidden, int intermediate, int q_dim, int kv_dim, int head_dim) {
  ChainShape sh{};
  const int n_qkv = q_dim + 2 * kv_dim;
  if (M < 1 || M > kChainRows || hidden > kChainHidden || hidden % 64 || intermediate % 64 || q_dim % 64 || head_dim % 4 || head_dim > 128) return sh;
  sh.T = (M + 15) / 16 * 16;
  sh.o = chain_tiles(M, sh.T, hidden, q_dim, false);
  sh.gate_up = chain_tiles(M, sh.T, intermediate, hidden, true);
  sh.down = chain_tiles(M, sh.T, hidden, intermediate, false);
  sh.qkv = chain_tiles(M, sh.T, n_qkv, hidden, false);
  if (!sh.o.rows || !sh.gate_up.rows || !sh.down.rows || !sh.qkv.rows) return sh;   // more columns than a round has
  int rows = 0;
  for (const ChainTiles *t : {&sh.o, &sh.gate_up, &sh.down, &sh.qkv}) rows = t->rows > rows ? t->rows : rows;
  sh.op_bytes = (rows * 128 + 1023) / 1024 * 1024;
  // Activations: four stages, three of the largest.  The rest is weights.  (A product reads 128 rows of an operand, however many were filled: the activations' ring
  // lies behind the last one.)
  sh.a_slots = sh.T <= 80 ? 4 : 3;
  const int behind = sh.a_slots * 2 * sh.T * 128, room = kSmemMax - 1024 - kBarBytes - behind;
  sh.w_stages = room / (2 * sh.op_bytes);
  if (sh.w_stages > kMaxWStages) sh.w_stages = kMaxWStages;
  if (sh.w_stages < 2) return sh;
  // On their way at a time: five blocks of 72 rows 631 us with two, 593, 592 and 593 with three to five.
  sh.on_way = sh.w_stages < 4 ? sh.w_stages : 4;
  sh.smem = sh.w_stages * 2 * sh.op_bytes + behind + kBarBytes + 1024;
  const int reach = (sh.w_stages * 2 - 1) * sh.op_bytes + 128 * 128 + kBarBytes + 1024;
  if (sh.smem < reach) sh.smem = reach;
  if (sh.smem < 116 * 1024) sh.smem = 116 * 1024;   // (one per SM: it takes all tensor memory and waits for its whole grid)
  sh.ok = 1;
  return sh;
}

size_t chain_plane_bytes(long M, int hidden, int q_dim, int kv_dim) {
  if (hidden > kChainHidden) return 0;
  // (a product's parts are kMaxSplit at most, and all its tiles in all its parts have an SM each)
  const long n_qkv = q_dim + 2 * kv_dim, widest = hidden > n_qkv ? hidden : n_qkv, of_all_sms = (long)kNumSM * 128;
  const long columns = kMaxSplit * widest < of_all_sms ? kMaxSplit * widest : of_all_sms;
  return (size_t)(M < kChainRows ? M : kChainRows) * columns * sizeof(float);
}

dpara_status launch_chain(const ChainShape &sh, const ChainArgs &a, int32_t *status, cudaStream_t st) {
  const int QD = a.n_q_heads * a.head_dim, KD = a.n_kv_heads * a.head_dim;
  ChainParams P;
  memset(static_cast<void *>(&P), 0, sizeof(P));
  bool ok = true;
  ChainInfo &I = P.info;
  auto product = [&](int g, const ChainTiles &t, const void *w, const void *act, int N, int K) {
    ok = ok && make_tmap_bf16_2d(&P.map_w[g], w, K, g == kGateUp ? 2 * (uint64_t)N : N, (uint64_t)K * 2, kSlabK, t.rows) &&
         make_tmap_bf16_2d(&P.map_a[g], act, K, a.M, (uint64_t)K * 2, kSlabK, sh.T);
    I.p[g] = ChainProduct{N, t.rows, t.tiles, t.split, t.tiles * t.split, g == kGateUp ? (K + kSlabK - 1) / kSlabK : (K + 2 * kSlabK - 1) / (2 * kSlabK)};
  };
  if (a.tail) {
    product(kO, sh.o, a.w_o, a.a, a.hidden, QD);
    product(kGateUp, sh.gate_up, a.w_gate_up, a.hn, a.intermediate, a.hidden);
    product(kDown, sh.down, a.w_down, a.act, a.hidden, a.intermediate);
  }
  if (a.head) product(kQkv, sh.qkv, a.w_qkv, a.xn, QD + 2 * KD, a.hidden);
  if (!ok) return DPARA_ERR_CUDA;
  I.tail = a.tail; I.head = a.head;
  I.M = a.M; I.T = sh.T; I.H = a.hidden; I.I = a.intermediate; I.n_q = a.n_q_heads; I.n_kv = a.n_kv_heads; I.D = a.head_dim;
  I.x = static_cast<const uint16_t *>(a.x); I.rms2_w = static_cast<const uint16_t *>(a.rms2_w); I.rms1_w = static_cast<const uint16_t *>(a.rms1_w);
  I.qnorm_w = static_cast<const uint16_t *>(a.qnorm_w); I.knorm_w = static_cast<const uint16_t *>(a.knorm_w);
  I.eps1 = a.eps1; I.eps2 = a.eps2; I.use_norm = a.use_norm;
  I.h1 = a.h1; I.y_f32 = a.y_f32;
  I.hn = static_cast<uint16_t *>(a.hn); I.act = static_cast<uint16_t *>(a.act); I.y_bf16 = static_cast<uint16_t *>(a.y_bf16);
  I.xn = static_cast<uint16_t *>(a.xn); I.qkv = static_cast<uint16_t *>(a.qkv);
  I.q = static_cast<uint16_t *>(a.q); I.k = static_cast<uint16_t *>(a.k); I.v = static_cast<uint16_t *>(a.v);
  I.angles = a.angles; I.planes = a.planes; I.counters = a.counters; I.status = status;
  I.op_bytes = sh.op_bytes; I.w_stages = sh.w_stages; I.a_slots = sh.a_slots; I.on_way = sh.on_way;
  P.bar_offset = sh.smem - 1024 - kBarBytes;
  if (cudaFuncSetAttribute(chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess) return DPARA_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  cfg.gridDim = dim3(kNumSM);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, chain_kernel, P);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorCooperativeLaunchTooLarge ? DPARA_ERR_UNSUPPORTED : DPARA_ERR_CUDA;
  }
  count_launches(1);
  return DPARA_OK;
}

}  // namespace dpara
