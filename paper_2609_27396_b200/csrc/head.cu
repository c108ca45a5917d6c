// The critical-path remainder T_Head (Alg. 1 after the barrier; Sec. 3.2 "Loss" for the head's form):
//   base logits  l = h W_lm^T  of the SELECTED branch (b * d rows), one tensor-core GEMM with an fp32 store;
//   head loop    z_i = l_i + W E(y_{i-1}),  y_0 = bonus,  i = 1..d;  y_i = argmax z_i (greedy) or y_i ~ softmax(z_i) (App. C:
//                temperature 1, top-p 1) by inverse CDF from a supplied uniform.
//
// The loop is d dependent steps, each a skinny product: all vocab rows of W (vocab x rank, bf16: 78 MB at vocab 151 936, rank 256) against
// the b embedding rows E(y_{i-1}).  ONE persistent cooperative kernel runs all d steps; CTA c owns the vocabulary entries
// [c T R, (c + 1) T R) as T tiles of R <= 128.  What bounds a step is shared memory (a tile of W written by its copy and read by its product takes
// ~1050 clocks, where its products alone would be done in 640) and the chain last product -> maxima of all CTAs -> token -> row of
// E -> first product (~5000 clocks, 850 of them one round trip to L2, 900 the row, and the slowest CTA sets the pace).  So
//   * as many of a CTA's tiles as tensor memory holds (three of nine at rank 256) are put there once and stay: the products read
//     their A operand from it (10 clocks per product of N = 16 against 40 from shared memory), and a step streams the others only.  The
//     ring that streams them is filled while the chain runs;
//   * the CTAs meet through DATA: each publishes its maximum per request as one 64-bit word with the step's tag, and the warp
//     that needs a request's winner polls that request's words of all CTAs.  No atomic, no fence, no counter, no second
//     round trip for the value; the same warp then fetches the row of E, so that no barrier of the CTA lies in between;
//   * sampling takes the same launch: z stays on the SM, and what a step exchanges is a sum per CTA and request and the token drawn (before: z
//     through memory and a second launch for the draw).
// Measured (16 steps, vocabulary 151 936, rank 256, this kernel before -> now): 16 requests greedy 233 -> 178 us, 8 requests sampling
// 330 -> 230 us (213 with weights as powers of two and their sums in fixed point, which lost light entries and failed for logits above 2^23);
// one request, 8 steps 85 -> 73 us.  Tried: a pause between the copies of the next step's tiles (the polls are not slowed down by
// them: 13.1 -> 13.5 thousand clocks a step); maxima of 16 requests per warp in place of 8 (the exchange is bound by its instructions: +1000).
// Warps:
//   8           streams the tiles of W that do not stay (they do not depend on the tokens: it runs ahead across steps);
//   10          streams the base logits, [b][R] per tile, on a ring of its own (plain loads of those from the epilogue queued behind the
//               deep W stream and cost 1.6 us each);
//   9           issues tcgen05.mma: D[128 vocab rows][kNb] = W_tile[128][rank] * Ey[kNb][rank]^T (M = 128, N = kNb = 16 or 32);
//   0-7         epilogue: thread = vocab row; warps w and w + 4 share the 32 rows of a TMEM lane quarter and take the even / odd
//               requests.  Warp w also does what is per request for requests w, w + 8, ...: publishes, polls, draws, builds Ey.
// Order of a CTA's tiles in a step: first as many streamed ones as the ring holds (their slots are refilled from then on), then the ones in
// tensor memory, then the rest; the vocabulary follows that order, so that a thread meets its rows in increasing order and a strict
// compare keeps the lowest index.
// Greedy: a maximum travels as (order-preserving key of z) << 32 | ~index: the largest word is the largest logit, lowest index on ties; NaN
// ranks below every number.
// Sampling: z replaces the base logit where that lies (shared memory; the call's workspace where a step's logits do not fit), each
// CTA publishes its weight sum per request and the maximum it is relative to; every CTA finds the CTA the threshold u * (sum of all) falls into by the
// same arithmetic, and that one finds the crossing entry and publishes the token.  Weights are fp32 exponentials (their argument is rounded: 6e-8 of
// its size, beside the logits' own error), sums fp64.
// All waits are bounded by wall time and give up with DPARA_STATUS_TIMEOUT; the launch is cooperative, so all CTAs are resident.
#include "gemm.cuh"
#include "head.cuh"
#include "sm100_ptx.cuh"

#include <math.h>

namespace dpara {
using namespace ptx;

namespace {
constexpr int kThreads = 352;  // warps 0-7 epilogue, 8 W, 9 MMA issuer, 10 base logits
constexpr int kEpiWarps = 8, kWeightWarp = 8, kMmaWarp = 9, kLogitWarp = 10;
constexpr int kMaxBatch = 32;
constexpr int kResidentCol = 128;                  // accumulators in TMEM columns [0, 128); behind them the tiles of W that stay
constexpr int kMaxAccBufs = kResidentCol / 16;
constexpr int kMaxStages = 4, kMaxLogitSlots = 16;
constexpr int kCtasPerLane = (kNumSM + 31) / 32;
constexpr int kCopies = 8;                         // of every word of the greedy loop
constexpr int kCtaStride = 32 * kCtasPerLane;      // words of one request: a slot per CTA, whole 128-byte lines
// Sampling: lane l looks after CTAs 5 l .. 5 l + 4 (the scan goes through them in the vocabulary's order) and reads slots l, 32 + l, ...
__device__ __forceinline__ int slot_of(int cta) { return cta % kCtasPerLane * 32 + cta / kCtasPerLane; }
constexpr unsigned long long kTagMask = 63;
constexpr int kTagBits = 6;                        // step / 2 + 1 (two buffers in turn, at most 64 steps)
constexpr int kBarBytes = 3072;                    // barriers and the reduction scratch
// Two loops' CTAs never share an SM: each takes all of its tensor memory and waits for its whole grid, so two loops (of calls on two streams) that each
// hold some SMs' would wait for one another.  The other kernels that take tensor memory need too many registers to come beside one.
constexpr int kMoreThanHalfAnSM = 116 * 1024;

__device__ __forceinline__ uint32_t head_key(float f) {
  if (f != f) return 0u;                    // NaN below everything
  if (f == 0.0f) f = 0.0f;                  // -0 == +0
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ unsigned long long load_word(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void publish(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// Polls until each of the lane's words (at(i) null: none) carries the step's tag; the whole warp calls it.
template <int kN, typename At>
__device__ __forceinline__ bool poll_words(At at, uint32_t tag, unsigned long long (&v)[kN], volatile int *abort_flag) {
  constexpr uint32_t kMask = (uint32_t)kTagMask;
#pragma unroll
  for (int i = 0; i < kN; ++i) v[i] = 0ull;
  uint64_t t0 = 0;
#pragma unroll 1
  for (unsigned int tries = 0;; ++tries) {
    bool all = true;
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      const unsigned long long *p = at(i);
      if (p && ((uint32_t)v[i] & kMask) != tag) v[i] = load_word(p);
    }
#pragma unroll
    for (int i = 0; i < kN; ++i) all = all && (!at(i) || ((uint32_t)v[i] & kMask) == tag);
    if (__all_sync(0xffffffffu, all)) return true;
    if (tries == 0) t0 = global_timer_ns();
    if (tries % 64 == 63 && __any_sync(0xffffffffu, *abort_flag || global_timer_ns() - t0 > kWaitLimitNs)) {
      *abort_flag = 7;
      return false;
    }
  }
}

// ---- sampling.  A logit's weight is exp(z - m) against the maximum m of its CTA's entries, in fp32 where that is a normal number and in fp64 below;
// every sum is fp64.  A CTA's sum travels with its m, and exp(m - largest m) in fp64 brings it beside the others'.
constexpr float kDeep = -87.f;
__device__ __noinline__ double deep_weight(float z, float m) { return exp((double)z - (double)m); }
// (NaN: no weight)
__device__ __forceinline__ double weight(float z, float m) {
  z = fmaxf(z, -INFINITY);
  return z - m < kDeep ? deep_weight(z, m) : (double)expf(z - m);
}
__device__ __forceinline__ double warp_scan(double v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}
// The sum of the lanes before this one, from the sums up to each: the next lane starts where this one ends, so that no threshold falls between two.
__device__ __forceinline__ double before_lane(double inclusive, int lane) {
  const double t = __shfl_up_sync(0xffffffffu, inclusive, 1);
  return lane ? t : 0.0;
}

template <int kCols>
__device__ __forceinline__ void load_acc(uint32_t taddr, uint32_t (&r)[kCols]) {
  if constexpr (kCols == 8) tmem_ld8(taddr, r);
  else tmem_ld16(taddr, r);
}
}  // namespace

struct ArParams {
  CUtensorMap map_w;
  CUtensorMap map_l;              // base logits [block * b][vocab] fp32 (the rows one step reads are contiguous), box = R columns x b rows
  const uint16_t *ar_w, *ar_e;    // [vocab][rank]
  const int32_t *bonus;           // [b]
  const float *uniforms;          // [b][block]
  int32_t *next_tokens;           // [b][block]
  // What the CTAs exchange, zero before the launch: words [2 (step parity)], greedy [kCopies][b][CTA], sampling [b][2][slot of a CTA]; drawn [2][kMaxBatch]
  unsigned long long *words, *drawn;
  float *z;                       // sampling where z does not fit in shared memory: [b][vocab]
  int32_t *status;
  int b, block, vocab;
  int rows, tiles;                // R (a multiple of 4), T
  int resident;                   // tiles that stay in tensor memory
  int stages, logit_slots, slab_bytes, logit_bytes, logit_off, e_off, bar_off;
  int z_in_place;                 // sampling: a step's base logits all have slots, z replaces them there
};

template <bool kSample, int kSlabs, int kNb>
__global__ void __launch_bounds__(kThreads, 1) ar_head_kernel(const __grid_constant__ ArParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int kRank = kSlabs * 64, kHalf = kNb / 2, kPer = kNb / kEpiWarps, kTileCols = kRank / 2, kAccBufs = kResidentCol / kNb;
  uint8_t *sW = smem;                                    // ring of tiles of W, [slab][R rounded up to 8][128 B]
  uint8_t *sE = smem + P.e_off;                          // Ey: [slab][kNb rows][128 B]
  uint8_t *sL = smem + P.logit_off;                      // slots of base logits, [b][R] fp32 each
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + P.bar_off);
  uint64_t *full = bars, *empty = full + kMaxStages, *l_full = empty + kMaxStages, *l_empty = l_full + kMaxLogitSlots,
           *acc_full = l_empty + kMaxLogitSlots, *acc_empty = acc_full + kMaxAccBufs, *e_ready = acc_empty + kMaxAccBufs;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(e_ready + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  unsigned long long *s_red = reinterpret_cast<unsigned long long *>(bars + 64);  // [kEpiWarps][kMaxBatch]

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
    for (int s = 0; s < kMaxLogitSlots; ++s) { mbar_init(l_full + s, 1); mbar_init(l_empty + s, kEpiWarps); }
    for (int a = 0; a < kAccBufs; ++a) { mbar_init(acc_full + a, 1); mbar_init(acc_empty + a, kEpiWarps); }
    mbar_init(e_ready, kEpiWarps);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == kMmaWarp) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  const int v0 = (int)blockIdx.x * P.tiles * P.rows;      // this CTA's first vocabulary entry
  const int count = min(P.vocab - v0, P.tiles * P.rows);  // its entries (>= 1: the grid ends with the vocabulary)
  const int my_tiles = (count + P.rows - 1) / P.rows;
  const int n_res = min(P.resident, my_tiles), n_str = my_tiles - n_res;
  const int lead = min(P.stages, n_str);                  // positions [lead, lead + n_res) of a step are the tiles that stay
  const int n_ctas = gridDim.x;
  const int slots = P.z_in_place ? my_tiles : P.logit_slots;   // in place: tile k of a step in slot k

  if (warp == kWeightWarp) {
    // ------------------------------------------------------------------ W (no kernel of this call writes it: no wait for the one in front)
    prefetch_tensormap(&P.map_w);
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    const uint32_t tx = (uint32_t)(kSlabs * P.rows * 128);
#pragma unroll 1
    for (int step = 0; step < P.block && ok; ++step)
#pragma unroll 1
      for (int k = 0; k < n_str; ++k) {
        ok = __all_sync(0xffffffffu, mbar_wait(empty + stage, ph ^ 1u, abort_flag, 2));
        if (!ok) break;
        const int row0 = v0 + (k < lead ? k : k + n_res) * P.rows;
        if (elect_one()) {
          uint8_t *dst = sW + stage * kSlabs * P.slab_bytes;
          mbar_arrive_expect_tx(full + stage, tx);
#pragma unroll
          for (int sb = 0; sb < kSlabs; ++sb) tma_load_2d(dst + sb * P.slab_bytes, &P.map_w, full + stage, sb * 64, row0);
        }
        __syncwarp();
        if (++stage == P.stages) { stage = 0; ph ^= 1u; }
      }
  } else if (warp == kLogitWarp) {
    // ------------------------------------------------------------------ base logits
    prefetch_tensormap(&P.map_l);
    pdl_wait();
    int slot = 0;
    uint32_t ph = 0;
    bool ok = true;
    const uint32_t tx = (uint32_t)(P.b * P.rows * 4);
#pragma unroll 1
    for (int step = 0; step < P.block && ok; ++step)
#pragma unroll 1
      for (int k = 0; k < my_tiles; ++k) {
        ok = __all_sync(0xffffffffu, mbar_wait(l_empty + slot, ph ^ 1u, abort_flag, 3));
        if (!ok) break;
        if (elect_one()) {
          mbar_arrive_expect_tx(l_full + slot, tx);
          tma_load_2d(sL + slot * P.logit_bytes, &P.map_l, l_full + slot, v0 + k * P.rows, step * P.b);
        }
        __syncwarp();
        if (++slot == slots) { slot = 0; ph ^= 1u; }
      }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------------ MMA issuer (the whole warp walks and waits, one lane issues: a wait
    // inside a one-lane branch costs two to three times as many clocks)
    const uint32_t idesc = idesc_bf16_f32(128, kNb, false, false);
    const uint64_t desc = smem_desc_sw128(smem_u32(sW), 16, 1024);
    const uint32_t w_lo0 = (uint32_t)desc, e_lo = w_lo0 + ((uint32_t)P.e_off >> 4), hi = (uint32_t)(desc >> 32);
    constexpr uint32_t e_slab = (uint32_t)(kNb * 128) >> 4;
    const uint32_t w_slab = (uint32_t)P.slab_bytes >> 4;
    int stage = 0, buf = 0;
    uint32_t ph = 0, ph_acc = 0;
    bool ok = true, there = false;
#pragma unroll 1
    for (int step = 0; step < P.block && ok; ++step) {
      ok = __all_sync(0xffffffffu, mbar_wait(e_ready, step & 1, abort_flag, 4));   // Ey of this step is in shared memory
#pragma unroll 1
      for (int k = 0; k < my_tiles && ok; ++k) {
        const bool stays = k >= lead && k < lead + n_res;
        // (Ey of a step is there when the accumulators of the step before have all been read)
        if (k >= kAccBufs) ok = __all_sync(0xffffffffu, mbar_wait(acc_empty + buf, ph_acc ^ 1u, abort_flag, 5));
        const uint32_t acc = tmem + buf * kNb;
        if (stays) {
          tc_fence_after();
          if (ok && elect_one()) {
            const uint32_t a = tmem + kResidentCol + (k - lead) * kTileCols;
#pragma unroll
            for (int kk = 0; kk < kSlabs * 4; ++kk) mma_ts_lo(acc, a + kk * 8, e_lo + (kk >> 2) * e_slab + (kk & 3) * 2, hi, idesc, kk > 0);
            mma_commit(acc_full + buf);
          }
          __syncwarp();
        } else {
          if (!__all_sync(0xffffffffu, there)) ok = __all_sync(0xffffffffu, mbar_wait(full + stage, ph, abort_flag, 6)) && ok;
          if (!ok) break;
          const int cur = stage;
          if (++stage == P.stages) { stage = 0; ph ^= 1u; }
          there = mbar_test(full + stage, ph);    // (the next one's barrier is asked before this one's products go out)
          tc_fence_after();
          if (elect_one()) {
            const uint32_t w_lo = w_lo0 + cur * kSlabs * w_slab;
#pragma unroll
            for (int kk = 0; kk < kSlabs * 4; ++kk)
              mma_ss_lo(acc, w_lo + (kk >> 2) * w_slab + (kk & 3) * 2, e_lo + (kk >> 2) * e_slab + (kk & 3) * 2, hi, idesc, kk > 0);
            mma_commit(empty + cur);
            mma_commit(acc_full + buf);
          }
          __syncwarp();
        }
        if (++buf == kAccBufs) { buf = 0; ph_acc ^= 1u; }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue, exchange, Ey
    const int quarter = warp & 3, nh = warp >> 2;  // TMEM lane quarter; column nh * kHalf + j holds request 2 j + nh
    const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
    // The tiles that stay: thread = row, 32 words (64 of K) at a time, in the layout of a bf16 A operand (lane = row, column = two
    // neighbouring elements).  Rows behind the tile or the vocabulary only make accumulator lanes that nobody reads.
#pragma unroll 1
    for (int i = 0; i < n_res; ++i) {
      const int row = min(v0 + (lead + i) * P.rows + min(quarter * 32 + lane, P.rows - 1), P.vocab - 1);
      const uint4 *src = reinterpret_cast<const uint4 *>(P.ar_w + (size_t)row * kRank);
#pragma unroll 1
      for (int sb = nh; sb < kSlabs; sb += 2) {
        uint32_t r[32];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const uint4 x = __ldg(src + sb * 8 + q);
          r[4 * q] = x.x; r[4 * q + 1] = x.y; r[4 * q + 2] = x.z; r[4 * q + 3] = x.w;
        }
        tmem_st32(lanes + kResidentCol + i * kTileCols + sb * 32, r);
      }
    }
    tmem_wait_st();
    tc_fence_before();
    // Ey[pos][k] = E[tok][k] in the K-major 128-byte-swizzle layout the MMA reads: slab = k / 64, row at 128 B pitch, 16-byte chunk c of the
    // row stored at chunk position c ^ (row & 7)
    auto put_row = [&](int n, bool live, int tok) {
      const int pos = (n & 1) * kHalf + (n >> 1);
      if (lane < kRank / 8) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (live) v = __ldg(reinterpret_cast<const uint4 *>(P.ar_e + (size_t)tok * kRank + lane * 8));
        *reinterpret_cast<uint4 *>(sE + (lane >> 3) * (kNb * 128) + pos * 128 + (((lane & 7) ^ (pos & 7)) << 4)) = v;
      }
    };
    pdl_wait();
    pdl_launch_dependents();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int n = warp + kEpiWarps * q;
      int tok = 0;
      if (n < P.b) {
        tok = P.bonus[n];
        if (tok < 0 || tok >= P.vocab) {
          if (P.status && lane == 0) atomicOr(reinterpret_cast<unsigned int *>(P.status), DPARA_STATUS_BAD_TOKEN);
          tok = 0;
        }
      }
      put_row(n, n < P.b, tok);
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(e_ready);

    const int z_row = kSample && !P.z_in_place ? P.vocab : P.rows;   // floats between two requests' z of a tile
    const int z_tile = P.z_in_place ? P.logit_bytes / 4 : P.rows;      // ... and between two tiles'
    const int mine_n = (P.b - nh + 1) / 2;                           // this warp's requests 2 j + nh
    int buf = 0, slot = 0;
    uint32_t ph_acc = 0, ph_l = 0;
    bool ok = true;
#pragma unroll 1
    for (int step = 0; step < P.block && ok; ++step) {
      float bz[kHalf];
      int bv[kHalf];
#pragma unroll
      for (int j = 0; j < kHalf; ++j) { bz[j] = -INFINITY; bv[j] = -1; }
#pragma unroll 1
      for (int k = 0; k < my_tiles; ++k) {
        ok = __all_sync(0xffffffffu, mbar_wait(l_full + slot, ph_l, abort_flag, 9) && mbar_wait(acc_full + buf, ph_acc, abort_flag, 8));
        if (!ok) break;
        tc_fence_after();
        uint32_t acc[kHalf];
        load_acc<kHalf>(lanes + buf * kNb + nh * kHalf, acc);
        const int r = quarter * 32 + lane, v = v0 + k * P.rows + r;
        const bool live = r < P.rows && v < P.vocab;
        float *sl = reinterpret_cast<float *>(sL + slot * P.logit_bytes) + nh * P.rows + min(r, P.rows - 1);
        float *zt = kSample && !P.z_in_place ? P.z + (size_t)nh * P.vocab + v : sl;
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty + buf);
        if (++buf == kAccBufs) { buf = 0; ph_acc ^= 1u; }
        // four requests at a time: their loads and compares in flight together
#pragma unroll
        for (int j4 = 0; j4 < kHalf; j4 += 4) {
          if (j4 >= mine_n) break;
          float l[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) l[u] = sl[2 * min(j4 + u, mine_n - 1) * P.rows];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = j4 + u;
            const float z = __uint_as_float(acc[j]) + l[u];
            if (kSample) {
              if (live && j < mine_n) zt[(size_t)(2 * j) * z_row] = z;
              bz[j] = live ? fmaxf(bz[j], z) : bz[j];   // (fmaxf drops NaN)
            } else if (live && (z > bz[j] || (bv[j] < 0 && z == z))) {
              // larger, or the first number this thread sees (NaN never wins; -inf can, at the lowest index)
              bz[j] = z; bv[j] = v;
            }
          }
        }
        if (!kSample || !P.z_in_place) {
          __syncwarp();
          if (lane == 0) mbar_arrive(l_empty + slot);
        }
        if (++slot == slots) { slot = 0; ph_l ^= 1u; }
      }
      // ---- maxima of the CTA: by warp, then over the four quarters
#pragma unroll
      for (int j4 = 0; j4 < kHalf; j4 += 4) {
        if (j4 >= mine_n) break;
        uint32_t key[4], best[4], low[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) key[u] = !kSample && bv[j4 + u] < 0 ? 0u : head_key(bz[j4 + u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) best[u] = __reduce_max_sync(0xffffffffu, key[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) low[u] = kSample ? 0u : __reduce_max_sync(0xffffffffu, key[u] == best[u] && key[u] ? 0xffffffffu - (uint32_t)bv[j4 + u] : 0u);
        if (lane < 4) {
          const unsigned long long x = lane == 0 ? ((unsigned long long)best[0] << 32) | low[0] : lane == 1 ? ((unsigned long long)best[1] << 32) | low[1]
                                     : lane == 2 ? ((unsigned long long)best[2] << 32) | low[2] : ((unsigned long long)best[3] << 32) | low[3];
          s_red[quarter * kMaxBatch + min(2 * (j4 + lane) + nh, kMaxBatch - 1)] = x;
        }
      }
      // (a warp whose wait ran out takes the others along)
      ok = named_bar_all_256(ok);
      if (!ok) break;
      const bool last = step + 1 == P.block;
      unsigned long long top[kPer];
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int n = warp + kEpiWarps * q;
        const unsigned long long x = s_red[(lane & 3) * kMaxBatch + n];
        const uint32_t hi32 = __reduce_max_sync(0xffffffffu, (uint32_t)(x >> 32));
        top[q] = (unsigned long long)hi32 << 32;
        if (!kSample) top[q] |= __reduce_max_sync(0xffffffffu, (uint32_t)(x >> 32) == hi32 ? (uint32_t)x : 0u);
      }
      // this step's words: the two buffers in turn (a CTA writes a step's words when it has seen all of the step before, so those two steps
      // older have been read), in kCopies copies of which a CTA polls one.  (Sampling: one copy, read in whole lines; eight, read with a stride of
      // five words, took 16 us more over 16 steps of 8 requests.)
      const uint32_t tag = (uint32_t)(step >> 1) + 1u;
      constexpr int kWords = kSample ? 2 : 1, copies = kSample ? 1 : kCopies;
      const size_t copy_words = (size_t)P.b * kWords * kCtaStride;
      unsigned long long *const words = P.words + (size_t)(step & 1) * copies * copy_words;
      const unsigned long long *const my_words = words + blockIdx.x % copies * copy_words;
      int tok[kPer];
#pragma unroll
      for (int q = 0; q < kPer; ++q) tok[q] = 0;
      if (!kSample) {
        unsigned long long got[kPer * kCtasPerLane];
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          const int n = warp + kEpiWarps * q;
          // key << 32 | ~(entry of the CTA's range) << 6 | tag
          const uint32_t entry = 0xffffffffu - (uint32_t)top[q] - (uint32_t)v0;
          if (n < P.b && lane < copies)
            publish(words + lane * copy_words + (size_t)n * kCtaStride + blockIdx.x, (top[q] >> 32 << 32) | (uint32_t)(~entry << kTagBits) | tag);
        }
        if (last && blockIdx.x != 0) break;     // (CTA 0 writes the last winners)
        ok = poll_words([&](int i) -> const unsigned long long * {
          const int n = warp + kEpiWarps * (i / kCtasPerLane), c = lane + 32 * (i % kCtasPerLane);
          return n < P.b && c < n_ctas ? my_words + (size_t)n * kCtaStride + c : nullptr;
        }, tag, got, abort_flag);
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          unsigned long long x = 0ull;
#pragma unroll
          for (int i = 0; i < kCtasPerLane; ++i) {
            const unsigned long long w = got[q * kCtasPerLane + i];
            const uint32_t v = ((~(uint32_t)w) >> kTagBits) + (uint32_t)((lane + 32 * i) * P.tiles * P.rows);
            const unsigned long long y = w >> 32 ? (w >> 32 << 32) | (0xffffffffu - v) : 0ull;
            x = y > x ? y : x;
          }
          const uint32_t hi32 = __reduce_max_sync(0xffffffffu, (uint32_t)(x >> 32));
          const uint32_t lo32 = __reduce_max_sync(0xffffffffu, (uint32_t)(x >> 32) == hi32 ? (uint32_t)x : 0u);
          const int n = warp + kEpiWarps * q;
          tok[q] = hi32 ? (int)(0xffffffffu - lo32) : 0;      // (no number in the row: 0)
          if (blockIdx.x == 0 && n < P.b && lane == 0 && ok) P.next_tokens[(size_t)n * P.block + step] = tok[q];
        }
      } else {
        // weight sums: lane l has the groups of four entries [l per_lane, (l + 1) per_lane) of the CTA's range (an odd number of them: no bank
        // conflicts), three groups at a time
        const int groups = count >> 2, tile_groups = P.rows >> 2, per_lane = ((groups + 31) >> 5) | 1, seg = 4 * per_lane;
        double mine[kPer];
        float own_m[kPer];
        unsigned long long got[kPer * 2 * kCtasPerLane];   // per request: the lane's CTAs' sums, then their maxima
        const float *const z0 = P.z_in_place ? reinterpret_cast<const float *>(sL) : P.z + v0;
        auto z_at = [&](int n, int e) { const int t = e / P.rows; return z0 + (size_t)n * z_row + (size_t)t * z_tile + (e - t * P.rows); };
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          const int n = warp + kEpiWarps * q;
          mine[q] = 0.0;
          own_m[q] = -INFINITY;
          if (n < P.b) {
            const uint32_t key = (uint32_t)(top[q] >> 32);
            const float m = __uint_as_float(key & 0x80000000u ? key & 0x7fffffffu : ~key);
            own_m[q] = m;
            if (m > -INFINITY && m < INFINITY) {
              int g = lane * per_lane, t = g / tile_groups, r = g - t * tile_groups;
              const int g1 = min(groups, g + per_lane);
              const float *const zn = z0 + (size_t)n * z_row;
              double sum[2] = {0.0, 0.0};
#pragma unroll 1
              for (; g < g1; g += 3) {
                float4 x[3];
                float low = m;
#pragma unroll
                for (int u = 0; u < 3; ++u) {
                  x[u] = make_float4(m, m, m, m);
                  if (g + u < g1) x[u] = *reinterpret_cast<const float4 *>(zn + (size_t)t * z_tile + 4 * r);
                  if (++r == tile_groups) { r = 0; ++t; }
                  x[u].x = fmaxf(x[u].x, -INFINITY); x[u].y = fmaxf(x[u].y, -INFINITY); x[u].z = fmaxf(x[u].z, -INFINITY); x[u].w = fmaxf(x[u].w, -INFINITY);
                  low = fminf(low, fminf(fminf(x[u].x, x[u].y), fminf(x[u].z, x[u].w)));
                }
                if (low - m >= kDeep) {
#pragma unroll
                  for (int u = 0; u < 3; ++u) {
                    const double w0 = expf(x[u].x - m), w1 = expf(x[u].y - m), w2 = expf(x[u].z - m), w3 = expf(x[u].w - m);
                    if (g + u < g1) { sum[0] += w0; sum[1] += w1; sum[0] += w2; sum[1] += w3; }
                  }
                } else {
#pragma unroll 1
                  for (int e = 0; e < 12 && g + (e >> 2) < g1; ++e) {
                    const float4 y = e < 4 ? x[0] : e < 8 ? x[1] : x[2];
                    sum[0] += weight((e & 3) == 0 ? y.x : (e & 3) == 1 ? y.y : (e & 3) == 2 ? y.z : y.w, m);
                  }
                }
              }
              mine[q] = sum[0] + sum[1];
            }
            double s = mine[q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane < copies) {
              unsigned long long *const to = words + lane * copy_words + (size_t)(2 * n) * kCtaStride + slot_of(blockIdx.x);
              const unsigned long long bits = (unsigned long long)__double_as_longlong(s);
              // (the sum's lowest bits travel with the maximum)
              publish(to, (bits & ~kTagMask) | tag);
              publish(to + kCtaStride, (unsigned long long)__float_as_uint(m) << 32 | (bits & kTagMask) << kTagBits | tag);
            }
          }
        }
        ok = poll_words([&](int i) -> const unsigned long long * {
          const int q2 = i / kCtasPerLane, n = warp + kEpiWarps * (q2 / 2), c = lane * kCtasPerLane + i % kCtasPerLane;
          return n < P.b && c < n_ctas ? my_words + (size_t)(2 * n + (q2 & 1)) * kCtaStride + i % kCtasPerLane * 32 + lane : nullptr;
        }, tag, got, abort_flag);
        if (ok) {
#pragma unroll
          for (int q = 0; q < kPer; ++q) {
            const int n = warp + kEpiWarps * q;
            if (n >= P.b) break;
            double s_all[kCtasPerLane];
            float m_all[kCtasPerLane], top_m = -INFINITY;
#pragma unroll
            for (int i = 0; i < kCtasPerLane; ++i) {
              const bool has = lane * kCtasPerLane + i < n_ctas;
              const unsigned long long sum = got[(2 * q) * kCtasPerLane + i], max = got[(2 * q + 1) * kCtasPerLane + i];
              s_all[i] = has ? __longlong_as_double((long long)((sum & ~kTagMask) | (max >> kTagBits & kTagMask))) : 0.0;
              m_all[i] = has ? __uint_as_float((uint32_t)(max >> 32)) : -INFINITY;
              top_m = fmaxf(top_m, m_all[i]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) top_m = fmaxf(top_m, __shfl_xor_sync(0xffffffffu, top_m, o));
            int owner = 0, pick = 0;    // (no number above -inf, or an infinite one: token 0)
            if (top_m > -INFINITY && top_m < INFINITY) {
              double run = 0.0;
#pragma unroll
              for (int i = 0; i < kCtasPerLane; ++i) {
                s_all[i] *= exp((double)m_all[i] - (double)top_m);
                run += s_all[i];
              }
              const double inc = warp_scan(run, lane), total = __shfl_sync(0xffffffffu, inc, 31);
              // (a uniform that is not in [0, 1) makes the last entry with weight the one drawn)
              const float u = P.uniforms[(size_t)n * P.block + step];
              const double T = u >= 0.f && u < 1.f ? (double)u * total : (double)INFINITY;
              // the first CTA whose end lies above the threshold; if rounding left none, the last one with weight.  (There is one: the sum of
              // the CTA with the largest m is at least 1.)
              double from = before_lane(inc, lane), base = 0.0, tail_base = 0.0;
              int found = -1, tail = -1;
#pragma unroll
              for (int i = 0; i < kCtasPerLane; ++i) {
                const double to = from + s_all[i];
                if (s_all[i] > 0.0) {
                  tail = lane * kCtasPerLane + i; tail_base = from;
                  if (found < 0 && to > T) { found = tail; base = from; }
                }
                from = to;
              }
              unsigned int who = __ballot_sync(0xffffffffu, found >= 0);
              int src = __ffs(who) - 1;
              if (!who) {
                found = tail; base = tail_base;
                src = 31 - __clz(__ballot_sync(0xffffffffu, tail >= 0));
              }
              owner = __shfl_sync(0xffffffffu, found, src);
              base = __shfl_sync(0xffffffffu, base, src);
              if (owner == (int)blockIdx.x) {
                // the lane whose entries the threshold falls into, then the entry, by the same rule
                const double scale = exp((double)own_m[q] - (double)top_m), w = mine[q] * scale, lane_inc = warp_scan(w, lane), lane_from = before_lane(lane_inc, lane);
                unsigned int hit = __ballot_sync(0xffffffffu, w > 0.0 && base + lane_inc > T);
                int hl = __ffs(hit) - 1;
                if (!hit) hl = 31 - __clz(__ballot_sync(0xffffffffu, w > 0.0));
                double acc = base + __shfl_sync(0xffffffffu, lane_from, hl);
                const int e0 = hl * seg, e1 = min(count, e0 + seg);
                pick = -1;
                int last_entry = e0;                                     // the last entry with weight
#pragma unroll 1
                for (int c0 = e0; c0 < e1 && pick < 0; c0 += 32) {
                  double x = 0.0;
                  if (c0 + lane < e1) x = weight(*z_at(n, c0 + lane), own_m[q]);
                  const double in = warp_scan(x * scale, lane);
                  const unsigned int some = __ballot_sync(0xffffffffu, x > 0.0), over = __ballot_sync(0xffffffffu, x > 0.0 && acc + in > T);
                  if (over) pick = c0 + __ffs(over) - 1;
                  if (some) last_entry = c0 + 31 - __clz(some);
                  acc += __shfl_sync(0xffffffffu, in, 31);
                }
                if (pick < 0) pick = last_entry;
                pick += v0;
              }
            }
            if (owner == (int)blockIdx.x && lane == 0) {
              publish(P.drawn + (step & 1) * kMaxBatch + n, (unsigned long long)pick << kTagBits | tag);
              P.next_tokens[(size_t)n * P.block + step] = pick;
            }
          }
        }
        if (P.z_in_place) {
          // z has been read: the slots go back (they were written here, and copies will write them next)
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) for (int k = 0; k < my_tiles; ++k) mbar_arrive(l_empty + k);
        }
        if (last) break;
        unsigned long long token[1] = {0ull};
        const unsigned long long *const mine_drawn =
            lane < kPer && warp + kEpiWarps * lane < P.b ? P.drawn + (step & 1) * kMaxBatch + warp + kEpiWarps * lane : nullptr;
        ok = ok && poll_words([&](int) { return mine_drawn; }, tag, token, abort_flag);
#pragma unroll
        for (int q = 0; q < kPer; ++q) tok[q] = __shfl_sync(0xffffffffu, (int)(token[0] >> kTagBits), q);
      }
      if (last) break;
      if (ok) {
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
          const int n = warp + kEpiWarps * q;
          if (n < P.b) put_row(n, true, tok[q]);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(e_ready);
      } else {
        named_bar_all_256(false);   // (this warp's part of the next step's barrier: the others leave there)
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

namespace {
// Clears the words that the loop's CTAs exchange.  A kernel and not a memset: the LM head then starts behind it without a gap, and may read its weights
// ahead of its wait.
__global__ void __launch_bounds__(256) head_clear_kernel(uint4 *words, size_t n) {
  pdl_wait();
  pdl_launch_dependents();
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) words[i] = make_uint4(0, 0, 0, 0);
}

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
constexpr size_t kDrawnWords = 2 * kMaxBatch;
size_t words_bytes(int b) { return ((size_t)2 * kCopies * b * kCtaStride + kDrawnWords) * sizeof(unsigned long long); }
}  // namespace

size_t head_workspace_bytes(int b, int block, int vocab) {
  if (b <= 0 || block <= 0 || vocab <= 0) return 0;
  return align256((size_t)b * block * vocab * sizeof(float)) + words_bytes(b) + align256((size_t)b * vocab * sizeof(float));
}

template <int kNb>
static void (*ar_kernel(bool sample, int slabs))(ArParams) {
  static void (*const k[2][4])(ArParams) = {{ar_head_kernel<false, 1, kNb>, ar_head_kernel<false, 2, kNb>, ar_head_kernel<false, 3, kNb>, ar_head_kernel<false, 4, kNb>},
                                           {ar_head_kernel<true, 1, kNb>, ar_head_kernel<true, 2, kNb>, ar_head_kernel<true, 3, kNb>, ar_head_kernel<true, 4, kNb>}};
  return k[sample][slabs - 1];
}

dpara_status launch_head(const HeadArgs &h, void *workspace, int32_t *status, cudaStream_t st) {
  if (h.b <= 0 || h.block <= 0 || h.hidden <= 0 || h.vocab <= 0 || h.rank <= 0) return DPARA_ERR_INVALID_ARG;
  if (h.b > kMaxBatch || h.rank % 64 != 0 || h.rank > 256 || h.hidden % 64 != 0 || h.vocab % 8 != 0 || h.block > 64) return DPARA_ERR_UNSUPPORTED;
  if (!h.sel_reps || !h.w_lm || !h.ar_w || !h.ar_e || !h.bonus || !h.next_tokens || !workspace) return DPARA_ERR_INVALID_ARG;
  if (!aligned16(h.sel_reps) || !aligned16(h.w_lm) || !aligned16(h.ar_w) || !aligned16(h.ar_e) || !aligned16(workspace)) return DPARA_ERR_INVALID_ARG;
  uint8_t *ws = static_cast<uint8_t *>(workspace);
  float *logits = reinterpret_cast<float *>(ws);
  unsigned long long *words = reinterpret_cast<unsigned long long *>(ws + align256((size_t)h.b * h.block * h.vocab * sizeof(float)));

  ArParams P;
  memset(&P, 0, sizeof(P));
  int dev = 0, sms = kNumSM;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (sms > kNumSM || sms < 1) sms = kNumSM;
  const int slabs = h.rank / 64, nb = h.b <= 16 ? 16 : 32;
  const bool sample = h.uniforms != nullptr;
  // Tiles per CTA, and with them the number of CTAs.  A step takes ~0.5 us for each tile of a CTA and ~0.012 for each CTA that the others have to hear from: T tiles of 128 rows on n
  // CTAs cost 42 T + n, with as few tiles as the SMs allow and up.  Before, all SMs had as many rows as came out evenly (12 steps, us, that / this): vocabulary 5760 73.2 / 58.5 (45
  // CTAs of 144), 12000 75.8 / 67.0, 30128 90.7 / 87.7; sampling 127.5 / 109.2, 128.6 / 121.9, 145.4 / 137.4; 60000 191 / 178.
  // Where that leaves fewer than four slots of base logits beside the ring of W, tiles of 120 rows are taken if they leave four with as many tiles a CTA.  16 steps of hidden 512, us,
  // 128 rows / 120.  Rank 256: 151936 entries 16 requests 273 / 250, 12 to 15 237..249 / 235..247; 100000 entries 16 requests 220 / 201, 14 199 / 197, 12 189 / 188.  Rank 192: 151936
  // entries, 13 to 16 requests 236..246 / 233..242.  Where they don't leave four they mostly lose (17 to 32 requests, rank 256: 285..358 / 291..362; ranks 64 to 192 of other vocabularies
  // up to 8 %), but not always: 16 requests of 128256 entries 242 / 226, rank 192 of 151936 with 17 to 19 306..317 / 284..300.
  auto plan = [&](int full) {
    const int blocks = (h.vocab + full - 1) / full;
    auto ctas = [&](int t) { return (blocks + t - 1) / t; };
    P.tiles = (blocks + sms - 1) / sms;
    while (42 * (P.tiles + 1) + ctas(P.tiles + 1) < 42 * P.tiles + ctas(P.tiles)) ++P.tiles;
    const int share = ctas(P.tiles) * P.tiles;   // the tiles, evenly filled
    P.rows = ((h.vocab + share - 1) / share + 3) / 4 * 4;
    if (P.rows < 32) P.rows = 32;
    // Tiles that stay: what fits behind the accumulators; one step alone reads W once either way.
    P.resident = h.block > 1 ? (512 - kResidentCol) / (32 * slabs) : 0;
    if (P.resident > P.tiles) P.resident = P.tiles;
    P.slab_bytes = (P.rows + 7) / 8 * 1024;
    P.logit_bytes = (h.b * P.rows * 4 + 127) / 128 * 128;
    const int tile_bytes = slabs * P.slab_bytes, room = 227 * 1024 - 1024 - slabs * nb * 128 - kBarBytes;
    const int streamed = P.tiles - P.resident, most = streamed < 1 ? 1 : (streamed < kMaxStages ? streamed : kMaxStages);
    auto stages_with = [&](int slots) {
      const int n = (room - slots * P.logit_bytes) / tile_bytes;
      return n < 0 ? 0 : (n < most ? n : most);
    };
    P.z_in_place = sample && P.tiles <= kMaxLogitSlots && stages_with(P.tiles) >= (most < 2 ? most : 2);
    if (P.z_in_place) {
      P.logit_slots = P.tiles;
    } else {
      // two to four slots of base logits, as many as cost the ring of W nothing
      P.logit_slots = 2;
      while (P.logit_slots < 4 && stages_with(P.logit_slots + 1) == stages_with(2)) ++P.logit_slots;
    }
    P.stages = stages_with(P.logit_slots);
    return P.z_in_place || P.logit_slots == 4;
  };
  if (!plan(128)) {
    const int tiles = P.tiles;
    if (!plan(120) || P.tiles != tiles) plan(128);
  }
  const int grid = (h.vocab + P.tiles * P.rows - 1) / (P.tiles * P.rows);

  const size_t vecs = (kDrawnWords + (size_t)2 * h.b * (sample ? 2 : kCopies) * kCtaStride) / 2;   // 16 bytes each
  launch_pdl(head_clear_kernel, dim3((unsigned)(vecs < 148 * 256 ? (vecs + 255) / 256 : 148)), dim3(256), 0, st, reinterpret_cast<uint4 *>(words), vecs);
  DPARA_CHECK_LAUNCH();
  count_launches(1);

  // base logits of the selected branches, fp32, stored step-major [block][b][vocab] (GEMM row n * block + i goes
  // to row i * b + n): the b rows a step reads then lie in one contiguous range instead of b ranges
  // block * vocab * 4 bytes apart
  GemmArgs g;
  g.a = h.sel_reps; g.w = h.w_lm; g.M = h.b * h.block; g.N = h.vocab; g.K = h.hidden; g.epi = 3;
  g.resid = nullptr; g.resid_bf16 = 0; g.out = logits; g.out_bf16 = nullptr; g.perm_block = h.block; g.perm_b = h.b;
  g.w_ready = 1;   // the kernel in front clears words of the workspace
  dpara_status rc = launch_gemm_tc(g, status, st);
  if (rc != DPARA_OK) return rc;

  if (!make_tmap_bf16_2d(&P.map_w, h.ar_w, h.rank, h.vocab, (uint64_t)h.rank * 2, 64, P.rows)) return DPARA_ERR_CUDA;
  if (!make_tmap_f32_2d(&P.map_l, logits, h.vocab, (uint64_t)h.block * h.b, (uint64_t)h.vocab * 4, P.rows, h.b)) return DPARA_ERR_CUDA;
  P.ar_w = static_cast<const uint16_t *>(h.ar_w); P.ar_e = static_cast<const uint16_t *>(h.ar_e);
  P.bonus = h.bonus; P.uniforms = h.uniforms; P.next_tokens = h.next_tokens;
  P.drawn = words; P.words = words + kDrawnWords; P.status = status;
  P.z = reinterpret_cast<float *>(reinterpret_cast<uint8_t *>(words) + words_bytes(h.b));
  P.b = h.b; P.block = h.block; P.vocab = h.vocab;
  const int tile_bytes = slabs * P.slab_bytes, e_bytes = slabs * nb * 128;
  P.e_off = P.stages * tile_bytes;
  P.logit_off = P.e_off + e_bytes;
  P.bar_off = P.logit_off + P.logit_slots * P.logit_bytes;
  int smem = P.bar_off + kBarBytes + 1024;
  if (smem < P.e_off + 128 * 128 + 1024) smem = P.e_off + 128 * 128 + 1024;   // (a product reads 128 rows of a slab, however many were filled)
  if (smem < kMoreThanHalfAnSM) smem = kMoreThanHalfAnSM;
  void (*const kernel)(ArParams) = nb == 16 ? ar_kernel<16>(sample, slabs) : ar_kernel<32>(sample, slabs);
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) != cudaSuccess) return DPARA_ERR_CUDA;
  // cooperative: the CTAs wait for one another's words, so every one has to be resident (one per SM fits by construction)
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, kernel, P) != cudaSuccess) {
    cudaGetLastError();
    return DPARA_ERR_CUDA;
  }
  count_launches(1);
  return DPARA_OK;
}

}  // namespace dpara
