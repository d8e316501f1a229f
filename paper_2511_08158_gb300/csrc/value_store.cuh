// Rounding of a stored value of A into the plan's storage type, shared by the plan build and the
// value refresh.
#pragma once

#include <type_traits>

#include "device_common.cuh"

namespace loops {

template <class T>
__device__ __forceinline__ T cvt_rn(float x);
template <>
__device__ __forceinline__ __half cvt_rn<__half>(float x) { return __float2half_rn(x); }
template <>
__device__ __forceinline__ __nv_bfloat16 cvt_rn<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// Out of line: inlined, the compiler computes it for every entry and selects.
template <class TB>
static __device__ __noinline__ TB stored_value_f64(float v, double scale) { return from_f64<TB>((double)v * scale); }

// The plan's power-of-two scale in binary32; 0 where it is outside binary32's normal range.
inline float scale_f32(double scale) { return scale >= 0x1p-126 && scale <= 0x1p127 ? (float)scale : 0.f; }

// Stored value of one input entry: round(scale * v). A binary32 entry's product with the power-of-
// two scale is exact in binary32, so it needs no binary64 arithmetic (a slow pipe here), except
// below binary32's normal range.
template <class TB>
__device__ __forceinline__ TB stored_value(double v, double scale, float) { return from_f64<TB>(v * scale); }
template <class TB>
__device__ __forceinline__ TB stored_value(float v, double scale, float scale_f) {
  if constexpr (std::is_same<TB, double>::value) {
    return (double)v * scale;
  } else if constexpr (std::is_same<TB, float>::value) {
    return v;  // FP32 plans store unscaled values
  } else {
    const float x = v * scale_f;
    if (v != 0.f && !(fabsf(x) >= 0x1p-126f)) return stored_value_f64<TB>(v, scale);
    return cvt_rn<TB>(x);
  }
}

}  // namespace loops
