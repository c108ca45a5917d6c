// bf16 GEMM  out[M][N] = epilogue( a[M][K] * w[N][K]^T )  for few activation rows: the WEIGHTS are the rows of the tensor-core
// product and the activations its columns.
//
// With few rows the product is a pass over the weights, and what bounds it is how many SMs stream them, how evenly, and how few clocks
// the issuing warps spend per byte.  256-column tiles of activations x weights left a 72-row product with 16 CTAs for 4096 output
// columns, each a serial chain over all of K.  Measured at 72 rows (us, weights from HBM; that tiling -> this kernel): 6144 x 4096
// 31.1 -> 14.9, 4096 x 4096 34.0 -> 12.5, 2 x 12288 x 4096 SwiGLU 60.4 -> 39.4 (5.2 TB/s), 4096 x 12288 83.3 -> 23.1.  What is left
// above the weights' 7.7 / 5.1 / 31 / 15 us at the copy rate: ~1.4 us from the wait to the first products, ~3 us behind the last.  Here
//   * a tile is one or two operands of R <= 128 weight rows (any multiple of 8: the 128-row operand behind R only makes
//     accumulator lanes that nobody reads), so that the tiles come out at a whole number of rounds over the SMs;
//   * where all tiles run at once, a CLUSTER of S CTAs shares a tile, each over its part of K; the parts meet through distributed shared
//     memory, in the order of the ranks (the same sum every time), and every CTA stores its share of the activation rows.  Not
//     with several rounds of tiles: the parts' meeting is not hidden behind the next tile (100 rows, 10240 x 5120: 46.0 us in three rounds of
//     four CTAs a tile, 25.2 in one of single CTAs; 128 rows, 20480 x 8192: 93 and 70), and over 31 shapes it gained 4 % at most;
//   * a stage of the ring holds the tile's weight rows and T activation rows (M rounded up to 16) of one or two 64-column slabs of K,
//     one TMA copy per operand.  The stage's barrier and loop cost ~250 clocks of the issuing warp beside 40..60 per product: with one
//     slab (four products) of a small tile that is more than the products themselves (16 rows, 4096 x 4096: 13.0 -> 11.2 us with two);
//   * the weights do not depend on the kernel in front: where the caller says so (w_ready) the ring is filled with them before
//     the wait for that kernel.
// Accumulator: lane = weight row (an output column), TMEM column = activation row.  Eight warps share the epilogue, which goes through
// a shared-memory buffer [activation row][128 outputs] and reads it back with 16 bytes per lane along the outputs.
#include "gemm.cuh"
#include "gemm_skinny.cuh"
#include "sm100_ptx.cuh"

#include <mutex>

namespace dpara {
using namespace ptx;

namespace {
constexpr int kThreads = 320;                 // warps 0-3 and 6-9: epilogue; 4: TMA; 5: MMA
constexpr int kEpiThreads = 256, kEpiWarps = 8;
constexpr int kSlabK = 64;                    // K columns per slab (one 128-byte swizzle row); a stage has one or two
constexpr int kWBytes = 128 * 64 * 2;         // 16 KB: what a product reads of an operand's slab
constexpr int kMaxSplit = 8;
constexpr int kSmemMax = 227 * 1024;
constexpr int kBarBytes = 512;
}  // namespace

struct SkinnyParams {
  CUtensorMap map_w[kGemmMaxGroups];
  CUtensorMap map_a[kGemmMaxGroups];
  void *out_g[kGemmMaxGroups];
  int n_groups;
  int M, N, K, epi, up_row_offset;
  int T;            // columns of the product: M rounded up (16; 32 above 256, then two instructions of T / 2)
  int rows;         // weight rows per operand
  // operands per tile: rows [0, rows) and [rows, 2 rows) of the tile; SwiGLU (always 2): gate rows and up rows
  int out_cols;     // output columns per tile
  int tiles;        // tiles of one product
  int split;        // cluster size; above 1 only with one round
  int stages, chunk;
  int ring_bytes, bar_offset;
  int w_ready;
  int one_round;    // every cluster has one tile: the parts may lie in the ring
  int tmem_cols;
  const void *resid;
  int resid_bf16;
  void *out_bf16;
  int perm_block, perm_b;
  int32_t *status;
};

__device__ __forceinline__ bool mbar_try_cluster(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t *bar, uint32_t parity, volatile int *abort_flag, int site) {
  if (mbar_try_cluster(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (;;) {
    if (mbar_try_cluster(bar, parity)) return true;
    if (*abort_flag) return false;
    if (global_timer_ns() - t0 > kWaitLimitNs) break;
  }
  if (*abort_flag == 0) *abort_flag = site;
  return false;
}
__device__ __forceinline__ void mbar_arrive_rank(uint64_t *bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(map_to_cta(smem_u32(bar), rank)) : "memory");
}

// Sum over the cluster's parts of four outputs of kU activation rows each, rank 0 first: the loads of four parts in flight, then their
// additions.  `addr`: shared-memory addresses in this CTA.
template <int kU, bool kCluster>
__device__ __forceinline__ void sum_parts(const uint32_t (&addr)[kU], int split, float4 (&acc)[kU]) {
  if (!kCluster) {
#pragma unroll
    for (int u = 0; u < kU; ++u)
      asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(acc[u].x), "=f"(acc[u].y), "=f"(acc[u].z), "=f"(acc[u].w) : "r"(addr[u]) : "memory");
    return;
  }
#pragma unroll
  for (int u = 0; u < kU; ++u) acc[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int s0 = 0; s0 < split; s0 += 4) {
    float4 x[4][kU];
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (s0 + s < split) {
#pragma unroll
        for (int u = 0; u < kU; ++u) x[s][u] = ld_dsmem_f4(map_to_cta(addr[u], s0 + s));
      }
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if (s0 + s < split) {
#pragma unroll
        for (int u = 0; u < kU; ++u) { acc[u].x += x[s][u].x; acc[u].y += x[s][u].y; acc[u].z += x[s][u].z; acc[u].w += x[s][u].w; }
      }
  }
}

// What the last step of a tile needs (by value: the kernel's loops keep nothing of it in registers).
struct Finish {
  void *out;
  const void *resid;
  void *out_bf16;
  uint32_t part_addr;
  int split, rank, rows_here, c0, half_bytes, col0, N, rows, n_ops, epi, resid_bf16, perm_block, perm_b;
};

__device__ __forceinline__ void sk_store(const Finish &P, int row, int col, float4 x) {
  void *out = P.out;
  if (P.epi == 0) {
    *reinterpret_cast<uint2 *>(static_cast<uint16_t *>(out) + (size_t)row * P.N + col) = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
    return;
  }
  const int orow = P.perm_block ? (row % P.perm_block) * P.perm_b + row / P.perm_block : row;
  *reinterpret_cast<float4 *>(static_cast<float *>(out) + (size_t)orow * P.N + col) = x;
  if (P.epi == 1 && P.out_bf16)
    *reinterpret_cast<uint2 *>(static_cast<uint16_t *>(P.out_bf16) + (size_t)row * P.N + col) = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
}

// Rows rank, rank + split, ... of a chunk (`rows_here` of them in all): sum of the parts, epilogue, store.  Eight warps, each takes
// every eighth of this CTA's rows, kU at a time.
template <int kU, bool kCluster>
__device__ __forceinline__ void sk_finish(const Finish P) {
  const int S = P.split, rank = P.rank, rows_here = P.rows_here, c0 = P.c0, half_bytes = P.half_bytes;
  const uint32_t part_addr = P.part_addr;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, warp = w < 4 ? w : w - 2;
  if (P.epi == 2) {
    constexpr int kR = (kU + 1) / 2, kA = 2 * kR;   // activation rows at a time, with a gate and an up address each
    const int col = P.col0 + 4 * lane;
    const bool in = 4 * lane < P.rows && col < P.N;
#pragma unroll 1
    for (int i0 = warp; rank + S * i0 < rows_here; i0 += kEpiWarps * kR) {
      uint32_t ad[kA];
#pragma unroll
      for (int u = 0; u < kR; ++u) {
        const int j = rank + S * (i0 + kEpiWarps * u);
        ad[2 * u] = part_addr + ((j < rows_here ? j : rank + S * i0) * 128 + 4 * lane) * 4;
        ad[2 * u + 1] = ad[2 * u] + half_bytes;
      }
      float4 x[kA];
      sum_parts<kA, kCluster>(ad, S, x);
#pragma unroll
      for (int u = 0; u < kR; ++u) {
        const int j = rank + S * (i0 + kEpiWarps * u);
        if (in && j < rows_here) {
          const float4 g = x[2 * u], up = x[2 * u + 1];
          *reinterpret_cast<uint2 *>(static_cast<uint16_t *>(P.out) + (size_t)(c0 + j) * P.N + col) =
              make_uint2(pack_bf16(silu(g.x) * up.x, silu(g.y) * up.y), pack_bf16(silu(g.z) * up.z, silu(g.w) * up.w));
        }
      }
    }
    return;
  }
  const int n_ops = P.n_ops;
#pragma unroll 1
  for (int h = 0; h < n_ops; ++h) {
    const int col = P.col0 + h * P.rows + 4 * lane;
    const bool in = 4 * lane < P.rows && col < P.N;
#pragma unroll 1
    for (int i0 = warp; rank + S * i0 < rows_here; i0 += kEpiWarps * kU) {
      uint32_t ad[kU];
      float4 rr[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int j = rank + S * (i0 + kEpiWarps * u), jj = j < rows_here ? j : rank + S * i0;
        ad[u] = part_addr + h * half_bytes + (jj * 128 + 4 * lane) * 4;
        rr[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (P.epi == 1 && in) {
          const size_t o = (size_t)(c0 + jj) * P.N + col;
          if (P.resid_bf16) {
            const uint2 b = *reinterpret_cast<const uint2 *>(static_cast<const uint16_t *>(P.resid) + o);
            rr[u] = make_float4(bf16lo(b.x), bf16hi(b.x), bf16lo(b.y), bf16hi(b.y));
          } else {
            rr[u] = *reinterpret_cast<const float4 *>(static_cast<const float *>(P.resid) + o);
          }
        }
      }
      float4 x[kU];
      sum_parts<kU, kCluster>(ad, S, x);
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int j = rank + S * (i0 + kEpiWarps * u);
        if (in && j < rows_here) {
          if (P.epi == 1) { x[u].x += rr[u].x; x[u].y += rr[u].y; x[u].z += rr[u].z; x[u].w += rr[u].w; }
          sk_store(P, c0 + j, col, x[u]);
        }
      }
    }
  }
}

// kHalves operands per tile, kInstr instructions across the activation rows (two above 256), kSlabs slabs per stage.
template <int kHalves, int kInstr, int kSlabs>
__global__ void __launch_bounds__(kThreads, 1) gemm_skinny_kernel(const __grid_constant__ SkinnyParams P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int w_slab = P.rows * 128, a_slab = P.T / kInstr * 128;         // bytes of one slab of an operand
  const int stage_bytes = kSlabs * (kHalves * w_slab + kInstr * a_slab);
  const int act_off = kSlabs * kHalves * w_slab;                             // activations behind the weights
  // the parts of a tile, [half][chunk][128]
  float *part = reinterpret_cast<float *>(P.one_round ? smem : smem + P.ring_bytes);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + P.bar_offset);
  uint64_t *empty = full + 16;
  uint64_t *acc_full = empty + 16, *acc_empty = acc_full + 2;
  uint64_t *ready = acc_empty + 2;   // every CTA of the cluster has left its part in its buffer
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(ready + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

  // (through a shuffle: the compiler then knows that these are the same in the whole warp, and works out descriptors and addresses of
  // the issuing warps in uniform registers)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int S = P.split;
  const int rank = __shfl_sync(0xffffffffu, (int)cluster_ctarank(), 0);
  const int cluster = blockIdx.x / S, n_clusters = gridDim.x / S;
  constexpr int kStageK = kSlabs * kSlabK;
  const int nkb = (P.K + kStageK - 1) / kStageK;   // (columns behind K read as zeros)
  const int kb0 = rank * nkb / S, kb1 = (rank + 1) * nkb / S;
  const int total = P.tiles * P.n_groups;
  const int len = kb1 - kb0;
  const int buf_cols = kHalves * P.T;
  const int n_buf = P.one_round || 2 * buf_cols > 512 ? 1 : 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < P.stages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full + b, 1);
      mbar_init(acc_empty + b, kEpiWarps);
    }
    mbar_init(ready, S);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 5) {
    tmem_alloc(tmem_slot, P.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  if (S > 1) cluster_sync_all();  // every CTA's barriers exist before a peer arrives on them
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  // Warps 4 and 5: the whole warp walks the loop and waits, one lane issues, and the barrier of the next stage is asked before this
  // stage's instructions go out.  Both loops issue in straight lines: a branch or a loop inside the one-lane part costs 50 clocks and
  // more, which with four short products per stage is what the loop's time would be.
  if (warp == 4) {
    for (int gi = 0; gi < P.n_groups; ++gi) {
      prefetch_tensormap(&P.map_w[gi]);
      prefetch_tensormap(&P.map_a[gi]);
    }
    const uint32_t tx = (uint32_t)stage_bytes;
    const int second = P.epi == 2 ? P.up_row_offset : P.rows;   // from the first operand's rows to the second's
    const int act_half = P.T / 2;
    auto load_w = [&](const CUtensorMap *map, int wrow, int kb, int stage) {
      uint8_t *sw = smem + stage * stage_bytes;
      mbar_arrive_expect_tx(full + stage, tx);
      tma_load_3d(sw, map, full + stage, 0, wrow, kSlabs * kb);
      if (kHalves == 2) tma_load_3d(sw + kSlabs * w_slab, map, full + stage, 0, second + wrow, kSlabs * kb);
    };
    auto load_a = [&](const CUtensorMap *map, int kb, int stage) {
      uint8_t *sa = smem + stage * stage_bytes + act_off;
      tma_load_3d(sa, map, full + stage, 0, 0, kSlabs * kb);
      if (kInstr == 2) tma_load_3d(sa + kSlabs * a_slab, map, full + stage, 0, act_half, kSlabs * kb);
    };
    // the first tile's first stages: their weights before the wait, if nothing in front of this kernel writes them
    const int early = P.w_ready ? min(P.stages, len) : 0;
    if (elect_one())
#pragma unroll 1
      for (int i = 0; i < early; ++i) load_w(&P.map_w[cluster / P.tiles], cluster % P.tiles * P.out_cols, kb0 + i, i);
    __syncwarp();
    pdl_wait();
    pdl_launch_dependents();
    if (elect_one())
#pragma unroll 1
      for (int i = 0; i < early; ++i) load_a(&P.map_a[cluster / P.tiles], kb0 + i, i);
    __syncwarp();
    int stage = early == P.stages ? 0 : early;
    uint32_t ph = early == P.stages ? 1u : 0u;
    bool ok = true, there = false;
    int first = early;
    for (int unit = cluster; unit < total && ok; unit += n_clusters, first = 0) {
      const int grp = unit / P.tiles, wrow = (unit - grp * P.tiles) * P.out_cols;
      const CUtensorMap *map_w = &P.map_w[grp], *map_a = &P.map_a[grp];
#pragma unroll 1
      for (int i = first; i < len; ++i) {
        if (!__all_sync(0xffffffffu, there)) ok = __all_sync(0xffffffffu, mbar_wait(empty + stage, ph ^ 1u, abort_flag));
        if (!ok) break;
        const int cur = stage;
        if (++stage == P.stages) { stage = 0; ph ^= 1u; }
        there = mbar_test(empty + stage, ph ^ 1u);
        if (elect_one()) {
          load_w(map_w, wrow, kb0 + i, cur);
          load_a(map_a, kb0 + i, cur);
        }
        __syncwarp();
      }
    }
  } else if (warp == 5) {
    const int n_cols = P.T / kInstr;
    const uint32_t idesc = idesc_bf16_f32(128, n_cols, false, false);
    const uint64_t desc = smem_desc_sw128(smem_u32(smem), 16, 1024);
    const uint32_t w_lo = (uint32_t)desc, a_lo = w_lo + ((uint32_t)act_off >> 4), hi = (uint32_t)(desc >> 32);
    const uint32_t stage_units = (uint32_t)stage_bytes >> 4, w_units = (uint32_t)w_slab >> 4, a_units = (uint32_t)a_slab >> 4;
    int stage = 0, k = 0;
    uint32_t ph = 0;
    bool ok = true, there = false;
    for (int unit = cluster; unit < total && ok; unit += n_clusters, ++k) {
      const int buf = n_buf == 2 ? k & 1 : 0;
      const uint32_t use = n_buf == 2 ? k >> 1 : k;
      ok = __all_sync(0xffffffffu, mbar_wait(acc_empty + buf, (use & 1) ^ 1u, abort_flag, 2));
      if (!ok) break;
      const uint32_t acc = tmem + buf * buf_cols;
#pragma unroll 1
      for (int i = 0; i < len; ++i) {
        if (!__all_sync(0xffffffffu, there)) ok = __all_sync(0xffffffffu, mbar_wait(full + stage, ph, abort_flag, 3));
        if (!ok) break;
        const int cur = stage;
        if (++stage == P.stages) { stage = 0; ph ^= 1u; }
        there = mbar_test(full + stage, ph);
        tc_fence_after();
        if (elect_one()) {
          const uint32_t so = cur * stage_units;
          // (the first product of a tile replaces what is in the accumulator)
#pragma unroll
          for (int kk = 0; kk < kStageK / 16; ++kk)
#pragma unroll
            for (int h = 0; h < kHalves; ++h)
#pragma unroll
              for (int q = 0; q < kInstr; ++q)
                mma_ss_lo(acc + h * P.T + q * n_cols, w_lo + so + (kSlabs * h + kk / 4) * w_units + 2 * (kk % 4), a_lo + so + (kSlabs * q + kk / 4) * a_units + 2 * (kk % 4), hi,
                          idesc, kk != 0 || i != 0);
          mma_commit(empty + cur);
        }
        __syncwarp();
      }
      if (ok && elect_one()) mma_commit(acc_full + buf);
      __syncwarp();
    }
  } else {
    pdl_wait();
    const uint32_t part_addr = smem_u32(part);
    const int ew = warp < 4 ? warp : warp - 2, quarter = warp & 3;   // epilogue warp 0..7; the TMEM lanes it may read
    int k = 0;
    bool live = true;
    for (int unit = cluster; unit < total && live; unit += n_clusters, ++k) {
      const int grp = unit / P.tiles, tile = unit - grp * P.tiles;
      const int buf = n_buf == 2 ? k & 1 : 0;
      const uint32_t use = n_buf == 2 ? k >> 1 : k;
      // one warp asks for the accumulator, the others sleep on the named barrier: eight polling warps slow down the two that issue
      live = named_bar_all_256(warp != 0 || __all_sync(0xffffffffu, mbar_wait(acc_full + buf, use & 1, abort_flag, 4)));
      tc_fence_after();
      const uint32_t taddr = tmem + buf * buf_cols + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
      for (int c0 = 0; c0 < P.T; c0 += P.chunk) {
        // ---- this CTA's part of activation rows [c0, c0 + chunk) into its buffer, once the last one has been read
        if (!P.one_round) named_bar_sync(1, kEpiThreads);
        const int n_here = min(P.chunk, P.T - c0);
        int piece = 0;   // 32 columns each, handed out to the two warps of a TMEM quarter in turn
#pragma unroll 1
        for (int h = 0; h < kHalves; ++h)
#pragma unroll 1
          for (int j0 = 0; j0 < n_here; j0 += 32, ++piece) {
            if ((piece & 1) != (ew >> 2)) continue;
            uint32_t r[32];
            tmem_ld32(taddr + h * P.T + c0 + j0, r);
            tmem_wait_ld();
            float *dst = part + (h * P.chunk + j0) * 128 + quarter * 32 + lane;
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (j0 + j < n_here) dst[j * 128] = __uint_as_float(r[j]);
          }
        if (c0 + P.chunk >= P.T) {  // the last of the accumulator has been read
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty + buf);
        }
        live = named_bar_all_256(live);
        if (S > 1) {
          if (threadIdx.x < S) mbar_arrive_rank(ready, threadIdx.x);
          live = named_bar_all_256(live && (warp != 0 || __all_sync(0xffffffffu, mbar_wait_cluster(ready, 0, abort_flag, 6))));
        }
        const int rows_here = min(P.M - c0, n_here);
        if (live) {
          const Finish f = {P.out_g[grp], P.resid, P.out_bf16, part_addr, S, rank, rows_here, c0, P.chunk * 512, tile * P.out_cols, P.N, P.rows,
                            P.epi == 2 ? 1 : kHalves, P.epi, P.resid_bf16, P.perm_block, P.perm_b};
          if (S == 1) sk_finish<4, false>(f);
          else sk_finish<2, true>(f);
        }
      }
    }
  }
  // ---------------- teardown
  __syncwarp();
  if (threadIdx.x == 0 && *abort_flag && P.status) atomicOr(reinterpret_cast<unsigned int *>(P.status), DPARA_STATUS_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  if (S > 1) cluster_sync_all();  // the peers may still read this CTA's buffer or arrive on its barriers until here
  if (warp == 5) tmem_dealloc(tmem, P.tmem_cols);
}

// ------------------------------------------------------------------------------------------------ host
namespace {
// Clusters of each size that are resident together (asked once per device).
const int *cluster_capacity() {
  static std::mutex m;
  static int cap[16][kMaxSplit + 1];
  static bool known[16];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 16) dev = 0;
  std::lock_guard<std::mutex> lock(m);
  if (!known[dev]) {
    if (cudaFuncSetAttribute(gemm_skinny_kernel<1, 1, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess) cudaGetLastError();
    int sms = kNumSM;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (int s = 1; s <= kMaxSplit; ++s) {
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      cfg.gridDim = dim3(sms / s * s);
      cfg.blockDim = dim3(kThreads);
      cfg.dynamicSmemBytes = kSmemMax;
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = s; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int n = 0;
      if (s == 1) n = sms;
      else if (cudaOccupancyMaxActiveClusters(&n, gemm_skinny_kernel<1, 1, 2>, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
      cap[dev][s] = n < sms / s ? n : sms / s;
    }
    known[dev] = true;
  }
  return cap[dev];
}
}  // namespace

// Ring, behind it the parts (in the ring itself when there is one round) or the 16 KB that a product may read behind an operand's
// start (it reads 128 rows, however many were filled), barriers.  false: fewer than two stages fit.
bool skinny_layout(SkinnyShape &sh, int nkb) {
  const int slab = 128 * (sh.rows * sh.halves + sh.T), part_row = sh.halves * 512;   // bytes per slab; bytes of parts per activation row
  sh.chunk = sh.one_round || sh.T * part_row <= 48 * 1024 ? sh.T : 32;
  int behind = sh.one_round ? 0 : sh.chunk * part_row;
  if (behind < kWBytes) behind = kWBytes;
  // Two slabs per stage where that leaves a ring of three, or of four above 64 activation rows, whose products are long enough to cover a stage's
  // loop (three stages of two slabs / six of one, us: 88 rows, 5120 x 17408 39.8 / 36.3; 100 rows, 151936 x 5120 284 / 273; but 13 rows,
  // 151936 x 1664 79.1 / 83.3), and each CTA of a tile at least one stage.
  const int room = kSmemMax - 1024 - kBarBytes - behind;
  sh.slabs = room / (2 * slab) >= (sh.T > 64 ? 4 : 3) && (nkb + 1) / 2 >= sh.split ? 2 : 1;
  const int stage = slab * sh.slabs;
  sh.stages = room / stage;
  if (sh.stages > 16) sh.stages = 16;
  if (sh.stages < 2) return false;
  sh.ring_bytes = sh.stages * stage;
  if (sh.one_round && sh.ring_bytes + behind < sh.T * part_row) return false;
  sh.bar_offset = sh.ring_bytes + behind;
  sh.smem = sh.bar_offset + kBarBytes + 1024;
  int cols = sh.halves * sh.T * (sh.one_round || 2 * sh.halves * sh.T > 512 ? 1 : 2);
  if (sh.T % 32) cols += 16;   // accumulators are read 32 columns at a time
  sh.tmem_cols = 32;
  while (sh.tmem_cols < cols && sh.tmem_cols < 512) sh.tmem_cols *= 2;
  return true;
}

// Shape of one launch: the cheapest of one CTA per tile, in its three smallest numbers of rounds, and two to eight CTAs per tile where all
// tiles run at once, with one or two operands each.  Cost of a candidate in ns: rounds x (slabs of a part x the longest of: issuing
// a slab's products; filling it (95 bytes per ns and SM, 42 of them from HBM); all SMs' weights from HBM (6300 bytes per ns, less for
// short tiles); all SMs' bytes from L2 (12000)) + what a tile costs beside its slabs (more when parts have to meet; an odd number of CTAs per
// cluster is slower than alone where it starts behind another kernel: five blocks of 72 rows 681 us with three CTAs a tile in the
// 4096 x 12288 product, 654 with four).  Over 150 random products of 1 to 288 rows (weights 512 .. 17408 wide, vocabularies to 151936) the launch
// taken is within 2 % of the best of all candidates, the CTA pairs' among them, for 91, within 5 % for 115 and 10 % for 135; the rest, up
// to 15 % off, are products of 7 to 22 us.  Measured (us, weights from HBM, launches back to back; CTAs per tile taken): 72 rows, 6144 x 4096 14.7
// (two; best other 16.7), 4096 x 4096 12.3 (four; 12.6), 2 x 12288 x 4096 SwiGLU 38.8 (one; 42.1), 4096 x 12288 23.2 (four; 24.4).
SkinnyShape skinny_shape(const GemmArgs &g) {
  SkinnyShape best{};
  best.cost = -1;
  if (g.M > 512 || g.split_k > 1) return best;
  const int T = g.M <= 256 ? (g.M + 15) / 16 * 16 : (g.M + 31) / 32 * 32;
  const int nkb = (g.K + kSlabK - 1) / kSlabK, groups = g.n_groups > 1 ? g.n_groups : 1;
  const int *cap = cluster_capacity();
  for (int halves = g.epi == 2 ? 2 : 1; halves <= 2; ++halves) {
    if (halves * T > 512) continue;
    const int per_tile = g.epi == 2 ? 1 : halves;     // output columns per operand row
    for (int s = 1; s <= (g.one_chain ? 1 : kMaxSplit) && s <= nkb; ++s) {
      if (cap[s] <= 0) continue;
      int tried = 0;
      for (long k = 1; tried < 3 && k < 4096; ++k) {
        const long tiles_max = k * cap[s] / groups;   // tiles of one product so that all products take k rounds
        if (tiles_max <= 0) continue;
        const int cols = (int)((g.N + tiles_max - 1) / tiles_max);
        int rows = ((cols + per_tile - 1) / per_tile + 7) / 8 * 8;
        if (rows > 128) continue;
        if (rows < 16) rows = 16;
        ++tried;
        SkinnyShape sh{};
        sh.T = T; sh.rows = rows; sh.halves = halves; sh.split = s;
        sh.tiles = (g.N + rows * per_tile - 1) / (rows * per_tile);
        const long units = (long)sh.tiles * groups;
        sh.clusters = units < cap[s] ? (int)units : cap[s];
        const long rounds = (units + sh.clusters - 1) / sh.clusters;
        sh.one_round = rounds == 1;
        if (!sh.one_round && (s > 1 || g.M > kManyRows)) break;   // (more rows: the caller takes such shapes to the CTA pairs)
        if (!skinny_layout(sh, nkb)) continue;
        const double w_bytes = rows * halves * 128.0, active = (double)sh.clusters * s;
        const double bytes = w_bytes + T * 128.0;
        double slab = halves * ((sh.slabs == 2 ? 130.0 : 180.0) + 0.55 * T);
        for (double other : {bytes / 95.0, w_bytes / 42.0, w_bytes * (1.0 + 16.0 / rows) * active / 6300.0, bytes * active / 12000.0})
          if (other > slab) slab = other;
        const double tail = 1000 + 15.0 * T * halves, more = rounds - 1;
        const int stages_k = (nkb + sh.slabs - 1) / sh.slabs;
        sh.cost = rounds * ((stages_k + s - 1) / s * sh.slabs) * slab + tail * (1.0 + 0.2 * more) + (s > 1 ? 800.0 + 150.0 * s : 0.0) + (s > 1 && s % 2 ? 1500.0 : 0.0);
        if (best.cost < 0 || sh.cost < best.cost) best = sh;
      }
    }
  }
  return best;
}

dpara_status launch_gemm_skinny(const GemmArgs &g, const SkinnyShape &sh, int32_t *status, cudaStream_t st) {
  SkinnyParams P;
  P.n_groups = g.n_groups > 1 ? g.n_groups : 1;
  const int w_rows = g.epi == 2 ? 2 * g.N : g.N;
  for (int gi = 0; gi < P.n_groups; ++gi) {
    const void *a = gi ? g.a_g[gi] : g.a, *w = gi ? g.w_g[gi] : g.w;
    void *o = gi ? g.out_g[gi] : g.out;
    if (!a || !w || !o || !aligned16(a) || !aligned16(w) || !aligned16(o)) return DPARA_ERR_INVALID_ARG;
    // [K / 64][rows][64]: the slabs of an operand in one copy
    if (!make_tmap_bf16_3d(&P.map_w[gi], w, 64, w_rows, g.K / 64, (uint64_t)g.K * 2, 128, 64, sh.rows, sh.slabs)) return DPARA_ERR_CUDA;
    if (!make_tmap_bf16_3d(&P.map_a[gi], a, 64, g.M, g.K / 64, (uint64_t)g.K * 2, 128, 64, sh.T <= 256 ? sh.T : sh.T / 2, sh.slabs)) return DPARA_ERR_CUDA;
    P.out_g[gi] = o;
  }
  P.M = g.M; P.N = g.N; P.K = g.K; P.epi = g.epi; P.up_row_offset = g.N;
  P.T = sh.T; P.rows = sh.rows; P.out_cols = g.epi == 2 ? sh.rows : sh.rows * sh.halves;
  P.tiles = sh.tiles; P.split = sh.split; P.stages = sh.stages; P.chunk = sh.chunk;
  P.ring_bytes = sh.ring_bytes; P.bar_offset = sh.bar_offset; P.one_round = sh.one_round; P.tmem_cols = sh.tmem_cols;
  P.w_ready = g.w_ready;
  P.resid = g.resid; P.resid_bf16 = g.resid_bf16; P.out_bf16 = g.out_bf16;
  P.perm_block = g.epi == 3 ? g.perm_block : 0; P.perm_b = g.perm_b;
  P.status = status;
  // (above 256 rows a ring of four stages of two slabs never fits)
  void (*const kernel)(SkinnyParams) = sh.T > 256       ? gemm_skinny_kernel<1, 2, 1>
                                       : sh.halves == 2 ? (sh.slabs == 2 ? gemm_skinny_kernel<2, 1, 2> : gemm_skinny_kernel<2, 1, 1>)
                                                        : (sh.slabs == 2 ? gemm_skinny_kernel<1, 1, 2> : gemm_skinny_kernel<1, 1, 1>);
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess) return DPARA_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  cfg.gridDim = dim3((unsigned)sh.clusters * sh.split);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = sh.split; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = sh.split > 1 ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, kernel, P) != cudaSuccess) { cudaGetLastError(); return DPARA_ERR_CUDA; }
  DPARA_CHECK_LAUNCH();
  count_launches(1);
  return DPARA_OK;
}

}  // namespace dpara
