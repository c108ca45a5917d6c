// bf16 GEMM  out[M][N] = epilogue( a[M][K] * w[N][K]^T )  on the 5th-generation tensor cores: more than a few activation rows
// (fewer: gemm_skinny.cu).
//
// A pair of CTAs (a cluster of two, tcgen05 cta_group::2) computes a tile of 256 weight rows x nt activation rows (nt <= 256).  The
// WEIGHTS are the rows of the product, so that nt can be any multiple of 16 (256-row tiles of activations computed 1280 rows for 1152
// and 512 for 288); pair_plan chooses it by the weights' shape too: 1152 rows are five tiles of 240 against 17408 x 5120 (SwiGLU) and seven of 176
// against 5120 x 5120, 288 rows two of 144 against 12288 x 4096 (SwiGLU) and three of 96 against 6144 x 4096.  Per 64-wide slab of K each CTA holds 128 of the weight
// rows and HALF of the activation rows (128-byte swizzle) and the accumulator of its own 128 weight rows; the even CTA's thread
// issues M = 256 products that read both halves.  These shapes are bound by the L2 -> shared-memory fill and by power: a pair pulls
// 64 KB per slab for 256 x 256 outputs.  Each CTA's producer fetches its own halves with ordinary tiled copies and counts the bytes
// on the LEADER's barrier; stage and accumulator hand-offs from the MMA thread reach both CTAs through one tcgen05.commit; the
// epilogue warps of both CTAs arrive on the leader's accumulator-empty barrier.
//
// Epilogues (accumulator: lane = output column, TMEM column = activation row):
//   0  bf16 store                                   (QKV projection)
//   1  fp32 out = resid + acc  (+ bf16 copy)        (O and down projections with the residual add)
//   2  bf16 out = silu(gate) * up                   (gate/up projection: 64 of a CTA's weight rows are gate rows and 64 the matching
//                                                    up rows, so the activation never leaves the SM)
//   3  fp32 store                                   (LM head: base logits)
// Every mbarrier wait is bounded; on expiry the CTA sets DPARA_STATUS_TIMEOUT and drains.
#include "gemm.cuh"
#include "gemm_skinny.cuh"
#include "sm100_ptx.cuh"

namespace dpara {
using namespace ptx;

namespace {
constexpr int kBK = 64;
constexpr int kRows = 128;                      // weight rows per CTA
constexpr int kWBytes = kRows * kBK * 2;        // 16 KB
constexpr int kThreads = 320;                   // warps 0-3 and 6-9: epilogue; 4: TMA; 5: MMA
constexpr int kEpiWarps = 8;
constexpr int kMaxStages = 8;
constexpr int kSmemMax = 227 * 1024;
constexpr int kBarBytes = 512;
constexpr int kEpiBytes = kEpiWarps * 16 * 32 * 4;   // 16 activation rows of 32 columns per warp (SwiGLU, fp32 stores)
}  // namespace

struct GemmKernelParams {
  CUtensorMap map_w[kGemmMaxGroups];   // one entry per product of a grouped launch (a plain launch uses entry 0)
  CUtensorMap map_a[kGemmMaxGroups];
  CUtensorMap map_tail[kGemmMaxGroups];   // activations in boxes of a tail unit's rows
  void *out_g[kGemmMaxGroups];
  int n_groups;
  int M, N, K;
  int epi;
  int up_row_offset;
  int nt, t_tiles, n_tiles;            // activation rows per tile; tiles of one product
  int main_units, tail_split, nt_tail; // kTail: tiles from main_units on are cut into tail_split units of nt_tail activation rows
  int stages;
  int w_ready;                         // the first unit's weights may be read ahead of the wait for the kernel in front
  int split_k;                         // > 1 (fp32 store only): the K range in split_k parts, part s writes plane s of [split_k][M][N] partial sums
  const void *resid;
  int resid_bf16;
  void *out_bf16;
  int32_t *status;
  int perm_block, perm_b;
};



// A unit of work: a tile of one of the products, one part of its K range (the parts of a tile are neighbours), or (kTail) some of the activation rows of
// such a part.
template <bool kTail>
struct Unit {
  int grp, tile, ks, kb0, kb1, row0, nt, rows;
  bool tail;
  __device__ __forceinline__ Unit(const GemmKernelParams &P, int unit, int nkb) {
    int sub = 0;
    tail = kTail && unit >= P.main_units;
    if (tail) {
      const int k = (unit - P.main_units) / P.tail_split;
      sub = unit - P.main_units - k * P.tail_split;
      unit = P.main_units + k;
    }
    const int per_group = P.t_tiles * P.n_tiles * P.split_k;
    grp = unit / per_group;
    unit -= grp * per_group;
    tile = unit / P.split_k;
    ks = unit - tile * P.split_k;
    kb0 = ks * nkb / P.split_k;
    kb1 = (ks + 1) * nkb / P.split_k;
    const int first = tile % P.t_tiles * P.nt;
    nt = tail ? P.nt_tail : P.nt;
    row0 = tail ? first + sub * P.nt_tail : first;
    // (a tile's last tail unit may reach behind the tile, the last tile behind the last row; nothing left: no rows)
    rows = min(min(P.M, first + P.nt) - row0, nt);
  }
};

// Epilogue of one accumulator tile.  A thread has one output column (lane) and takes 32 activation rows at a time: an instruction reads or
// writes 32 neighbouring columns of one activation row (fp32: one 128-byte line), straight from and to registers.  Shared memory is
// what these products are short of (per slab the products read 64 bytes and the copies write 64 bytes per clock of the 128 an SM
// has): a transposing buffer here cost 4 % of the whole product.  The two warps of a TMEM quarter take the blocks in turn, and the
// residual rows of a block are on their way while the one before is worked on.
template <bool kTail>
__device__ __forceinline__ void gemm_epilogue(const GemmKernelParams &P, uint32_t taddr, const Unit<kTail> &w, int rank, float *exchange, int quarter, int turn, int lane) {
  const int grp = w.grp, tile = w.tile;
  const int n_tile = tile / P.t_tiles, row0 = w.row0, rows_all = w.rows;
  if (P.epi == 2) {
    // quarters 0 and 1 have gate columns, 2 and 3 the matching up columns: each warp of such a pair hands 16 of the 32 activation rows to the
    // other and finishes the other 16
    const int col = n_tile * 128 + rank * 64 + (quarter & 1) * 32 + lane;
    const bool up_side = quarter >= 2;
    const int bar = 2 + (quarter & 1) + 2 * turn;
    float *mine = exchange + (quarter * 2 + turn) * 512 + lane;
    const float *theirs = exchange + ((quarter ^ 2) * 2 + turn) * 512 + lane;
    uint16_t *out = static_cast<uint16_t *>(P.out_g[grp]) + (size_t)row0 * P.N + col;
#pragma unroll 1
    for (int c0 = turn * 32; c0 < rows_all; c0 += 64) {
      uint32_t r[32];
      tmem_ld32(taddr + c0, r);
      tmem_wait_ld();
      // (selected, not indexed: r stays in registers)
#pragma unroll
      for (int j = 0; j < 16; ++j) mine[j * 32] = __uint_as_float(up_side ? r[j] : r[16 + j]);
      named_bar_sync(bar, 64);
      const int j0 = c0 + (up_side ? 16 : 0);
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float own = __uint_as_float(up_side ? r[16 + j] : r[j]), other = theirs[j * 32];
        const float v = silu(up_side ? other : own) * (up_side ? own : other);
        if (j0 + j < rows_all && col < P.N) out[(size_t)(j0 + j) * P.N] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
      }
      named_bar_sync(bar, 64);
    }
    return;
  }
  if (P.epi == 3) {
    // four bytes per output and nothing else: 16 activation rows at a time through the buffer, so that an instruction writes 512 bytes
    // (a split product of 20 slabs per unit, 42 MB of partial sums: 42 -> 39 us)
    const int sub = lane >> 3, col = n_tile * 256 + rank * 128 + quarter * 32 + (lane & 7) * 4;
    float *mine = exchange + (quarter * 2 + turn) * 512;
    float *out = static_cast<float *>(P.out_g[grp]) + (size_t)w.ks * P.M * P.N + col;
    const int pb = P.perm_block ? P.perm_block : 1 << 30, pm = P.perm_block ? P.perm_b : 0;   // row n * pb + i goes to i * perm_b + n
#pragma unroll 1
    for (int c0 = turn * 32; c0 < rows_all; c0 += 64) {
      uint32_t r[32];
      tmem_ld32(taddr + c0, r);
      tmem_wait_ld();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int j = 0; j < 16; ++j) mine[j * 32 + lane] = __uint_as_float(r[16 * h + j]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int rl = c0 + 16 * h + i * 4 + sub, row = row0 + rl;
          const float4 x = *reinterpret_cast<const float4 *>(mine + (i * 4 + sub) * 32 + (lane & 7) * 4);
          const int orow = P.perm_block ? (row % pb) * pm + row / pb : row;
          if (rl < rows_all && col < P.N) *reinterpret_cast<float4 *>(out + (size_t)orow * P.N) = x;
        }
        __syncwarp();
      }
    }
    return;
  }
  const int col = n_tile * 256 + rank * 128 + quarter * 32 + lane;
  const bool in = col < P.N;
  float rr[32];
  auto fetch = [&](int c0) {
    if (P.epi != 1 || !in) return;
    // (rows behind the last read row M - 1: an unconditional load the compiler can issue early; the value is not used)
    if (P.resid_bf16) {
      const uint16_t *src = static_cast<const uint16_t *>(P.resid) + col;
#pragma unroll
      for (int j = 0; j < 32; ++j) rr[j] = bf16_bits_to_float(src[(size_t)min(row0 + c0 + j, P.M - 1) * P.N]);
    } else {
      const float *src = static_cast<const float *>(P.resid) + col;
#pragma unroll
      for (int j = 0; j < 32; ++j) rr[j] = src[(size_t)min(row0 + c0 + j, P.M - 1) * P.N];
    }
  };
  if (turn * 32 < rows_all) fetch(turn * 32);
#pragma unroll 1
  for (int c0 = turn * 32; c0 < rows_all; c0 += 64) {
    uint32_t r[32];
    tmem_ld32(taddr + c0, r);
    tmem_wait_ld();
    float x[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = P.epi == 1 ? __uint_as_float(r[j]) + rr[j] : __uint_as_float(r[j]);
    if (c0 + 64 < rows_all) fetch(c0 + 64);
    if (!in) continue;
    const int rows = rows_all - c0;
    if (P.epi == 0) {
      uint16_t *out = static_cast<uint16_t *>(P.out_g[grp]) + (size_t)(row0 + c0) * P.N + col;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j < rows) out[(size_t)j * P.N] = __bfloat16_as_ushort(__float2bfloat16_rn(x[j]));
    } else {
      float *out = static_cast<float *>(P.out_g[grp]) + (size_t)(row0 + c0) * P.N + col;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j < rows) out[(size_t)j * P.N] = x[j];
      if (P.out_bf16) {
        uint16_t *o16 = static_cast<uint16_t *>(P.out_bf16) + (size_t)(row0 + c0) * P.N + col;
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (j < rows) o16[(size_t)j * P.N] = __bfloat16_as_ushort(__float2bfloat16_rn(x[j]));
      }
    }
  }
}

template <bool kTail>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1) gemm_pair_kernel(const __grid_constant__ GemmKernelParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int stage_bytes = kWBytes + P.nt * 64;   // 128 weight rows, nt / 2 activation rows
  float *exchange = reinterpret_cast<float *>(smem + P.stages * stage_bytes);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + P.stages * stage_bytes + kEpiBytes);   // used in the leader only
  uint64_t *empty = full + kMaxStages;                                            // local copy in each CTA
  uint64_t *acc_full = empty + kMaxStages;                                        // [2] local copy in each CTA
  uint64_t *acc_empty = acc_full + 2;                                             // [2] used in the leader only
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_empty + 2);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  // (through shuffles: the compiler then knows that these are the same in the whole warp)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int rank = __shfl_sync(0xffffffffu, (int)cluster_ctarank(), 0);
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  const int nkb = P.K / kBK;
  const int tiles = P.t_tiles * P.n_tiles * P.split_k * P.n_groups, units = kTail ? P.main_units + (tiles - P.main_units) * P.tail_split : tiles;

  if (threadIdx.x == 0) {
    for (int s = 0; s < P.stages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full + b, 1);
      mbar_init(acc_empty + b, 2 * kEpiWarps);   // of both CTAs
    }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 5) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers exist before anything signals across the pair
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  // (nothing above touches global memory: the set-up overlaps the tail of the kernel before)

  // Warps 4 and 5: the whole warp walks the loop and waits, one lane issues, and the barrier of the next stage is asked before this
  // stage's instructions go out (a wait inside a one-lane branch costs two to three times as many clocks, and the tensor pipe
  // takes only one product ahead of the running one: what the loop does between two stages' products is idle time of the pipe).
  if (warp == 4) {
    for (int gi = 0; gi < P.n_groups; ++gi) {
      prefetch_tensormap(&P.map_w[gi]);
      prefetch_tensormap(&P.map_a[gi]);
    }
    const bool swiglu = P.epi == 2;
    // (worked out once per unit: a division per stage is what the loop has no time for)
    struct Source {
      const CUtensorMap *map_w, *map_a;
      int wrow, arow;
      uint32_t tx;
    };
    auto source = [&](const Unit<kTail> &w) {
      const int n_tile = w.tile / P.t_tiles;
      return Source{&P.map_w[w.grp], w.tail ? &P.map_tail[w.grp] : &P.map_a[w.grp], swiglu ? n_tile * 128 + rank * 64 : n_tile * 256 + rank * 128,
                    w.row0 + rank * (w.nt / 2), 2u * (uint32_t)(kWBytes + w.nt * 64)};
    };
    auto load_w = [&](const Source &s, int kb, int stage) {
      uint8_t *sw = smem + stage * stage_bytes;
      if (rank == 0) mbar_arrive_expect_tx(full + stage, s.tx);
      tma_load_2d_pair(sw, s.map_w, full + stage, kb * kBK, s.wrow);
      if (swiglu) tma_load_2d_pair(sw + kWBytes / 2, s.map_w, full + stage, kb * kBK, P.up_row_offset + s.wrow);
    };
    auto load_a = [&](const Source &s, int kb, int stage) { tma_load_2d_pair(smem + stage * stage_bytes + kWBytes, s.map_a, full + stage, kb * kBK, s.arow); };
    // The weights of the first unit's first stages ahead of the wait, where nothing in front of this kernel writes them (us, without -> with: four blocks of
    // 280 rows of hidden 704 250 -> 242, five of 576 of 1024 375 -> 369, a block of 378 of 1600 82.0 -> 80.9, round of four requests 662.6 -> 659.7; larger products and the LM heads: the same).
    int early = 0;
    if (P.w_ready) {
      const Unit<kTail> first(P, pair, nkb);
      const Source s = source(first);
      early = min(P.stages, first.kb1 - first.kb0);
      if (elect_one())
#pragma unroll 1
        for (int i = 0; i < early; ++i) load_w(s, first.kb0 + i, i);
      __syncwarp();
      pdl_wait();
      if (elect_one())
#pragma unroll 1
        for (int i = 0; i < early; ++i) load_a(s, first.kb0 + i, i);
      __syncwarp();
    }
    pdl_wait();
    pdl_launch_dependents();
    int stage = early == P.stages ? 0 : early, done = early;
    uint32_t ph = early == P.stages ? 1u : 0u;
    bool ok = true, there = false;
    // (tile id = weight tile * t_tiles + activation tile: the pairs running together cover all activation rows of a few weight tiles)
    for (int unit = pair; unit < units && ok; unit += pairs, done = 0) {
      const Unit<kTail> w(P, unit, nkb);
      const Source s = source(w);
#pragma unroll 1
      for (int kb = w.kb0 + done; kb < w.kb1; ++kb) {
        if (!__all_sync(0xffffffffu, there)) ok = __all_sync(0xffffffffu, mbar_wait(empty + stage, ph ^ 1u, abort_flag, 2));
        if (!ok) break;
        const int cur = stage;
        if (++stage == P.stages) { stage = 0; ph ^= 1u; }
        there = mbar_test(empty + stage, ph ^ 1u);
        if (elect_one()) {
          load_w(s, kb, cur);
          load_a(s, kb, cur);
        }
        __syncwarp();
      }
    }
  } else if (warp == 5) {
    if (rank == 0) {
      const uint64_t desc = smem_desc_sw128(smem_u32(smem), 16, 1024);
      const uint32_t w_lo = (uint32_t)desc, a_lo = w_lo + (kWBytes >> 4), hi = (uint32_t)(desc >> 32), stage_units = (uint32_t)stage_bytes >> 4;
      int stage = 0, k = 0;
      uint32_t ph = 0;
      bool ok = true, there = false;
      for (int unit = pair; unit < units && ok; unit += pairs, ++k) {
        const Unit<kTail> w(P, unit, nkb);
        const uint32_t idesc = idesc_bf16_f32(2 * kRows, w.nt, false, false);
        const int buf = k & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(acc_empty + buf, ((k >> 1) & 1) ^ 1u, abort_flag, 3));  // both CTAs' epilogues of tile k - 2 are done
        if (!ok) break;
        const uint32_t acc = tmem + buf * 256;
#pragma unroll 1
        for (int kb = w.kb0; kb < w.kb1; ++kb) {
          if (!__all_sync(0xffffffffu, there)) ok = __all_sync(0xffffffffu, mbar_wait(full + stage, ph, abort_flag, 4));
          if (!ok) break;
          const int cur = stage;
          if (++stage == P.stages) { stage = 0; ph ^= 1u; }
          there = mbar_test(full + stage, ph);
          tc_fence_after();
          if (elect_one()) {
            const uint32_t so = cur * stage_units;
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk) mma2_ss_lo(acc, w_lo + so + 2 * kk, a_lo + so + 2 * kk, hi, idesc, kk != 0 || kb != w.kb0);
            mma2_commit_both(empty + cur);
          }
          __syncwarp();
        }
        if (ok && elect_one()) mma2_commit_both(acc_full + buf);
        __syncwarp();
      }
    }
  } else {
    pdl_wait();
    const int quarter = warp & 3, turn = warp >= 4;   // the TMEM lanes a warp may read; which of the two warps that may
    int k = 0;
    bool live = true;
    for (int unit = pair; unit < units && live; unit += pairs, ++k) {
      const int buf = k & 1;
      // one warp asks for the accumulator, the others sleep on the named barrier
      live = named_bar_all_256(warp != 0 || __all_sync(0xffffffffu, mbar_wait(acc_full + buf, (k >> 1) & 1, abort_flag, 5)));
      tc_fence_after();
      const uint32_t taddr = tmem + buf * 256 + ((uint32_t)(quarter * 32) << 16);
      if (live) gemm_epilogue<kTail>(P, taddr, Unit<kTail>(P, unit, nkb), rank, exchange, quarter, turn, lane);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_leader(acc_empty + buf);
    }
  }
  // ---------------- teardown
  __syncwarp();
  if (threadIdx.x == 0 && *abort_flag && P.status) atomicOr(reinterpret_cast<unsigned int *>(P.status), DPARA_STATUS_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer may still signal this CTA's barriers or read its shared memory until here
  if (warp == 5) tmem_dealloc_pair(tmem, 512);
}

// ------------------------------------------------------------------------------------------------ host
namespace {
int sm_count() {
  int dev = 0, sms = kNumSM;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 1 ? sms : kNumSM;
}

// Activation tiles for n_all weight tiles on `most` pairs.  A slab of a tile takes 0.12 + 0.21 nt / 256 us (fill and products; 0.33 at 256
// rows), or what its weights take from HBM (all pairs running: 0.385, 0.405 above 208 rows; 0.255 where two pairs read the same weights and
// 0.21 where more do, which does not fetch them only once), and a launch 6 us beside them.  Up to four slabs the last tile's epilogue
// decides, 0.013 us a row.  Narrower tiles are taken where that evens out the rounds or uses more pairs.  Measured (us):
//   200 x 6144 x 4096               24 tiles of 208 rows 21.9, 72 of 80 rows 18.5
//   1152 x 5120 x 5120              100 tiles of 240 rows (two rounds of 74, the second a third full) 61, 140 of 176 rows (two of 0.8 the length) 53
//   129 x 151936 x 2048             9 rounds of 144 rows 114, 17 of 80 rows 143
//   200 x 20480 x 8192              2 rounds of 208 rows 85, 3 of 112 rows 91
//   256 x 12288 x 4096, SwiGLU      2 rounds of 256 rows 57.8, 3 of 128 rows 55.3;  200 rows: 2 rounds of 208 rows 52.4, 3 of 112 rows 54.3
//   256 x 264 x 64                  one tile of 256 rows 7.2, three of 96 rows 5.1;  288 x 1536 x 1024 SwiGLU: three of 96 rows 10.9, four of 80 12.4
// Also tried: the tiles of the last rounds shared out by K, their pieces added through L2 by whoever finished last: never faster
// than this (1152 x 5120 x 17408 165 us against 163, 256 x 151936 x 5120 360 against 355: what the chip saves in idle time it gives back in
// clocks and in the pieces' traffic).
PairPlan pair_plan(int M, int n_all, int nkb, int most) {
  PairPlan best{};
  best.us = -1;
  double best_whole = 0;
  const int t0 = (M + 255) / 256;
  for (int t = t0; t < t0 + 4 && (t == t0 || (M + t - 1) / t > 64); ++t) {
    const int nt = ((M + t - 1) / t + 15) / 16 * 16;
    const long tiles = (long)n_all * t, rounds = (tiles + most - 1) / most;
    double slab = 0.12 + 0.21 * nt / 256.0;
    const double hbm = (tiles < most ? (double)tiles / most : 1.0) * (t == 1 ? (nt > 208 ? 0.405 : 0.385) : t == 2 ? 0.255 : 0.21);
    if (hbm > slab) slab = hbm;
    const double us = 6.0 + rounds * nkb * slab, whole = nkb <= 4 ? us + 0.013 * nt : us;
    if (best.us < 0 || whole < 0.97 * best_whole) { best.t_tiles = t; best.nt = nt; best.us = us; best_whole = whole; }
  }
  return best;
}

// The tiles of a last round that has few of them (at most a third of the pairs): each in up to `at_once` / left parts of its activation rows, on pairs that
// would have nothing to do.  Every part reads the tile's weights again (from L2), so only about two thirds of the pairs are given one.  Against whole
// tiles, 109 products of 129 to 1152 rows with 1 to 24 tiles left of 74, stores and SwiGLU, weights from HBM: 1.057x (geometric mean), faster by
// more than the spread in all but three, slower by more than it in none.  1.13 behind one round of tiles, 1.07 behind two or three, 1.035 behind four to nine (the pairs drift
// apart, and the whole tiles of a last round start early on some); 1.068 with 1 to 8 tiles left, 1.058 with 9 to 16, 1.044 with 17 to 24.  For
// instance 207 x 23112 x 1088 22.0 -> 19.7 us, 498 x 9920 x 2752 SwiGLU 54.9 -> 48.6, 1014 x 14784 x 4544 SwiGLU 196 -> 190.  Launches of several products or parts
// of K too: the append of five layers, 256 rows (40 tiles in four parts, 12 units behind two rounds) 47.3 -> 43.9, 200 rows 43.3 -> 41.4, 407 rows of half the heads 41.1 -> 39.2,
// 325 rows of 1280 features the same; the same bits.
void tail_plan(GemmRoute &r) {
  const long units = (long)r.pair.t_tiles * r.n_all;
  const int left = (int)(units % r.most), at_once = r.most * 13 / 20;   // 48 of 74 pairs
  r.nt_tail = r.main_units = 0;
  if (units < r.most || left == 0 || 2 * left > at_once) return;
  int nt = (r.pair.nt / (at_once / left) + 15) / 16 * 16;
  if (nt < 32) nt = 32;
  if (nt >= r.pair.nt) return;
  r.nt_tail = nt;
  r.main_units = (int)(units - left);
}
}  // namespace

// Everything about a launch that its sizes decide: refusals, then the kernel and its tiles.
dpara_status gemm_route(const GemmArgs &g, GemmRoute &r) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0 || g.epi < 0 || g.epi > 3) return DPARA_ERR_INVALID_ARG;
  if (g.K % kBK != 0 || g.N % 8 != 0 || g.n_groups > kGemmMaxGroups) return DPARA_ERR_UNSUPPORTED;
  // (one residual, one bf16 copy and one row order for all products of a launch)
  if (g.n_groups > 1 && ((g.epi != 0 && g.epi != 3) || g.perm_block)) return DPARA_ERR_UNSUPPORTED;
  const int nkb = g.K / kBK;
  if (g.split_k > 1 && (g.epi != 3 || g.M <= kManyRows || g.split_k > nkb || g.perm_block)) return DPARA_ERR_UNSUPPORTED;
  const int cols = g.epi == 2 ? 128 : 256;   // output columns per tile
  r.n_tiles = (g.N + cols - 1) / cols;
  r.n_all = r.n_tiles * (g.n_groups > 1 ? g.n_groups : 1) * (g.split_k > 1 ? g.split_k : 1);
  r.most = sm_count() / 2 < kNumSM / 2 ? sm_count() / 2 : kNumSM / 2;
  r.pair = pair_plan(g.M, r.n_all, nkb / (g.split_k > 1 ? g.split_k : 1), r.most);
  tail_plan(r);
  // Few rows: single CTAs that share a tile's K range inside clusters.  Above 128 activation rows by the two models (us, pairs / that:
  // 200 rows, 4096 x 12288 44.8 / 30.8, 4096 x 4096 19.8 / 16.1, 6144 x 4096 18.5 / 23.3; 400 rows, 4096 x 4096 21.1 / 22.8).
  r.few = 0;
  if (g.M <= 512) {
    r.skinny = skinny_shape(g);
    r.few = r.skinny.cost >= 0 && (g.M <= kManyRows || 1e-3 * r.skinny.cost + 3.5 < r.pair.us);
  }
  return DPARA_OK;
}

dpara_status launch_gemm_tc(const GemmArgs &g, int32_t *status, cudaStream_t st) {
  GemmRoute route;
  const dpara_status checked = gemm_route(g, route);
  if (checked != DPARA_OK) return checked;
  if (!g.a || !g.w || !g.out || (g.epi == 1 && !g.resid)) return DPARA_ERR_INVALID_ARG;
  if (!aligned16(g.a) || !aligned16(g.w) || !aligned16(g.out) || !aligned16(g.resid) || !aligned16(g.out_bf16)) return DPARA_ERR_INVALID_ARG;
  if (route.few) return launch_gemm_skinny(g, route.skinny, status, st);
  GemmKernelParams P;
  const int w_rows = g.epi == 2 ? 2 * g.N : g.N;
  P.n_groups = g.n_groups > 1 ? g.n_groups : 1;
  P.split_k = g.split_k > 1 ? g.split_k : 1;
  P.n_tiles = route.n_tiles;
  P.t_tiles = route.pair.t_tiles; P.nt = route.pair.nt;
  const bool tail = route.nt_tail > 0;
  P.nt_tail = route.nt_tail; P.main_units = route.main_units;
  P.tail_split = tail ? (P.nt + P.nt_tail - 1) / P.nt_tail : 1;
  for (int gi = 0; gi < P.n_groups; ++gi) {
    const void *a = gi ? g.a_g[gi] : g.a, *w = gi ? g.w_g[gi] : g.w;
    void *o = gi ? g.out_g[gi] : g.out;
    if (!a || !w || !o || !aligned16(a) || !aligned16(w) || !aligned16(o)) return DPARA_ERR_INVALID_ARG;
    if (!make_tmap_bf16_2d(&P.map_w[gi], w, g.K, w_rows, (uint64_t)g.K * 2, kBK, g.epi == 2 ? kRows / 2 : kRows)) return DPARA_ERR_CUDA;
    if (!make_tmap_bf16_2d(&P.map_a[gi], a, g.K, g.M, (uint64_t)g.K * 2, kBK, P.nt / 2)) return DPARA_ERR_CUDA;
    if (tail && !make_tmap_bf16_2d(&P.map_tail[gi], a, g.K, g.M, (uint64_t)g.K * 2, kBK, P.nt_tail / 2)) return DPARA_ERR_CUDA;
    P.out_g[gi] = o;
  }
  P.w_ready = g.w_ready && P.split_k == 1;   // (split: 192 rows, three layers of 2048 x 4096: an append of 24.6 us 25.0, the norm in front reads slower)
  P.M = g.M; P.N = g.N; P.K = g.K; P.epi = g.epi; P.up_row_offset = g.N;
  P.resid = g.resid; P.resid_bf16 = g.resid_bf16; P.out_bf16 = g.out_bf16; P.status = status;
  P.perm_block = g.epi == 3 ? g.perm_block : 0; P.perm_b = g.perm_b;
  const int stage_bytes = kWBytes + P.nt * 64;
  P.stages = (kSmemMax - 1024 - kBarBytes - kEpiBytes) / stage_bytes;
  if (P.stages > kMaxStages) P.stages = kMaxStages;

  const long units = (long)P.t_tiles * route.n_all;
  const int smem = P.stages * stage_bytes + 1024 + kBarBytes + kEpiBytes;
  void (*const kernel)(GemmKernelParams) = tail ? gemm_pair_kernel<true> : gemm_pair_kernel<false>;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess) return DPARA_ERR_CUDA;
  launch_pdl(kernel, dim3(2 * (unsigned)(units < route.most ? units : route.most)), dim3(kThreads), smem, st, P);
  DPARA_CHECK_LAUNCH();
  count_launches(1);
  return DPARA_OK;
}

}  // namespace dpara
