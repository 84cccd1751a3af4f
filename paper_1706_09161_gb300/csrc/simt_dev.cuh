// Packed FP32 arithmetic (two lanes per 64-bit register) and guarded 128-bit loads of the
// CUDA-core GEMM kernels.
#pragma once
#include <cuda_runtime.h>

namespace lbm {
namespace {

__device__ __forceinline__ unsigned long long ffma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

__device__ __forceinline__ unsigned long long fadd2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

__device__ __forceinline__ unsigned long long twice(float a) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(a));
  return d;
}

// four consecutive values p[0..3] of which `left` exist (zeros past them)
__device__ __forceinline__ float4 load4(const float* p, int left, bool vec) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (left >= 4 && vec) return *reinterpret_cast<const float4*>(p);
  if (left > 0) v.x = p[0];
  if (left > 1) v.y = p[1];
  if (left > 2) v.z = p[2];
  if (left > 3) v.w = p[3];
  return v;
}

}  // namespace
}  // namespace lbm
