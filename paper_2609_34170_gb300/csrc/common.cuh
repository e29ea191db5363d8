// Shared device helpers of the rolling-step kernels (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"

namespace ravel {

typedef __nv_bfloat16 bf16;


__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(bf16 x) { return __bfloat162float(x); }

template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ bf16 from_f32<bf16>(float x) { return __float2bfloat16_rn(x); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// err: the word of an ErrorWord.  The kernel that raises an error also writes it
// to the host's mirror, so that a call without one copies nothing back (a
// 4-byte copy per call cost a batch-1 step 5 of 608 us, a tiny fp32 one 7 of
// 139, and a single projection, M 800 x N 1024 x K 4096, 7 of 22).
__device__ __forceinline__ void raise_error(int* err, int bits) {
  if (!err) return;
  atomicOr(err, bits);
  int* mirror = ((ErrorWord*)err)->mirror;
  if (mirror) atomicOr_system(mirror, bits);
}

// Programmatic Dependent Launch: let the next kernel in the stream start
// launching, and wait until the previous kernel has completed and its memory
// is visible (a no-op when the kernel was not launched programmatically).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float silu_f(float x) { return x / (1.f + expf(-x)); }

__device__ __forceinline__ float gelu_tanh_f(float g) {
  const float k0 = 0.7978845608028654f;   // sqrt(2/pi)
  return 0.5f * g * (1.f + tanhf(k0 * (g + 0.044715f * g * g * g)));
}

// The same with the tanh of the special-function unit (one instruction,
// relative error up to 2^-11), for results that are rounded to bf16: the error
// is up to |g| 2^-12.  For positive gates that is below the rounding (2^-8 of the
// result); for negative ones 1 + t cancels, and from about g = -1.5 on it is the
// larger of the two, absolute and at most 1.2e-3 at g = -5.
__device__ __forceinline__ float gelu_tanh_bf16out(float g) {
  const float k0 = 0.7978845608028654f;   // sqrt(2/pi)
  const float u = k0 * (g + 0.044715f * g * g * g);
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(u));
  return 0.5f * g * (1.f + t);
}

}  // namespace ravel
