// df64.cuh -- double-float numbers: a real as the unevaluated sum hi + lo of
// two floats (|lo| <= ulp(hi)/2), ~48 significant bits.  The DF64 form stores
// its links so; the arithmetic between the links is the FP64 form's fixed point
// (link_fx.cuh).
#pragma once
#include <cuda_runtime.h>

namespace clgc {

struct df64 {
  float hi, lo;
  df64() = default;
  __host__ __device__ constexpr df64(float h, float l) : hi(h), lo(l) {}
  // explicit: a double never turns into a df64 (or back) without a visible cast
  __device__ __forceinline__ explicit df64(double d) : hi((float)d), lo((float)(d - (double)(float)d)) {}
  __device__ __forceinline__ explicit operator double() const { return (double)hi + (double)lo; }
};

// s + e = a + b exactly, s = fl(a + b) (Knuth's two-sum).
__device__ __forceinline__ df64 df_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  return df64(s, (a - (s - bb)) + (b - bb));
}

// Storage of a complex df64 number: (re.hi, re.lo, im.hi, im.lo).
__device__ __forceinline__ float4 df_pack(df64 re, df64 im) { return make_float4(re.hi, re.lo, im.hi, im.lo); }

}  // namespace clgc
