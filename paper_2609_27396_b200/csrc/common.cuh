// Shared host/device helpers of the dpara kernels (sm_100a).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/dpara.h"

namespace dpara {

constexpr int kNumSM = 148;  // B200: 2 dies x 74 SMs; grids are sized in multiples of this where it matters

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) { return __uint_as_float(((uint32_t)b) << 16); }

__device__ __forceinline__ float bf16lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Launch-error check used by the host entry points: returns DPARA_ERR_CUDA from the caller.
#define DPARA_CHECK_LAUNCH()                                   \
  do {                                                         \
    cudaError_t e_ = cudaGetLastError();                       \
    if (e_ != cudaSuccess) return DPARA_ERR_CUDA;              \
  } while (0)

// Programmatic dependent launch.  THE RULE for every kernel of this library: a CTA runs pdl_launch_dependents() only after a pdl_wait() of
// its own (which blocks until the kernels before it have completed and their writes are visible), or never.  A kernel launched through launch_pdl behind
// it is then released, and its launch latency and set-up overlap this one's tail, only when everything older than the kernel
// in FRONT of it is complete: ahead of its own pdl_wait() it can race with that one kernel and with nothing else.  Most kernels touch global memory
// only behind their wait.  These read ahead of it, and what they read may not be written by the kernel directly in front:
//   kernel                                  reads ahead of its wait                in front of it, by the order its call launches them
//   gemm_skinny_, gemm_pair_kernel, w_ready  weights                                RMS norm, attention or a product (block); RMS norm or append_rows (append)
//   chain_kernel                            weights                                RMS norm, attention or the kernel that makes angles
//   qk_norm_rope_kernel                     context offsets or lengths, angles     the QKV product
//   append_rows_kernel                      accept_len, old lengths, capacity, row_start   the projection
//   the LM head's product                   weights                                head_clear_kernel
//   ar_head_kernel                          W of the head loop                     the LM head's product
//   verify kernels, early-start form        all but the representations; they also use their workspace   what the caller queued: the flag is its promise
// Moving a trigger ahead of a wait, or a kernel that writes one of these directly in front of its reader, makes a race.
// Without the launch attribute both instructions do nothing.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Process-wide count of kernels this library has launched (evidence for benchmarks; relaxed atomic).
void count_launches(int n);

}  // namespace dpara
