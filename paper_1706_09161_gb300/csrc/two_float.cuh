// Device sums kept in FP64, or in FP32 forms as an unevaluated pair of floats.
#pragma once
#include <cuda_runtime.h>

namespace lbm {
namespace {

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

template <typename real>
struct SumAcc;
template <>
struct SumAcc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ void warp_reduce() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  __device__ __forceinline__ void store(double* slot) const { *slot = s; }
};
template <>
struct SumAcc<float> {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float x) {
    float t, e;
    two_sum(hi, x, t, e);
    hi = t;
    lo = __fadd_rn(lo, e);
  }
  __device__ __forceinline__ void warp_reduce() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float oh = __shfl_xor_sync(0xffffffffu, hi, o), ol = __shfl_xor_sync(0xffffffffu, lo, o);
      float t, e;
      two_sum(hi, oh, t, e);
      hi = t;
      lo = __fadd_rn(__fadd_rn(lo, ol), e);
    }
  }
  // the pair (hi, lo) in the slot's 8 bytes; the final pass adds hi + lo in FP64
  __device__ __forceinline__ void store(double* slot) const { *reinterpret_cast<float2*>(slot) = make_float2(hi, lo); }
};

}  // namespace
}  // namespace lbm
