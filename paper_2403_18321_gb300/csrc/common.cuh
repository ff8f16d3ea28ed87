// common.cuh -- small device helpers shared by the kernels of this library.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "internal.h"

namespace gbpca {

constexpr unsigned kFull = 0xffffffffu;

template <typename T>
__device__ __forceinline__ float to_f32(T v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <>
__device__ __forceinline__ float to_f32<__half>(__half v) { return __half2float(v); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
  return v;
}
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Programmatic dependent launch.  The many small kernels of a fit take 2 to 6 us
// each, of which about one is the hand-over from one to the next; launched by
// launch_after, a kernel's CTAs come in while its predecessor still runs and wait
// in pdl_wait (first thing, every thread) for that one to complete and its
// writes to be visible.  Every kernel so launched waits, so that what a kernel has
// seen complete has seen everything before it complete.  pdl_begin also lets the
// next kernel's CTAs in -- for the short kernels only: waiting CTAs take SM slots
// that another stream could use.  100 x 100 x 50 fit 288 -> 239 us, 512 x 217 x 224
// 1434 -> 1410.  Not for the adjoint, whose small kernels ran longer beside the
// waiting CTAs than the hand-overs cost (512 x 512 x 200: 330 -> 347 us).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() {
  pdl_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
cudaError_t launch_after(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Records a data-dependent status in the header; the first non-OK code wins.
__device__ __forceinline__ void set_status(DevHeader* h, int st) {
  atomicCAS(&h->status, (int)PCA_OK, st);
}

}  // namespace gbpca
