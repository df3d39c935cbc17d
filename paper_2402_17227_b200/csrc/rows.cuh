// Sum of squares of a row by one warp.
#pragma once

#include "common.cuh"

namespace vcas {
namespace {

__device__ __forceinline__ float sq8(const uint4& v) {
  // eight bf16 values: widen by placing the 16 bits in the top half of a float
  float s = 0.f;
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float lo = __uint_as_float(u[i] << 16);
    const float hi = __uint_as_float(u[i] & 0xffff0000u);
    s = fmaf(lo, lo, s);
    s = fmaf(hi, hi, s);
  }
  return s;
}
__device__ __forceinline__ float sq4(const float4& v) {
  float s = v.x * v.x;
  s = fmaf(v.y, v.y, s);
  s = fmaf(v.z, v.z, s);
  s = fmaf(v.w, v.w, s);
  return s;
}

template <typename T> struct Vec;
template <> struct Vec<__nv_bfloat16> {
  using type = uint4;
  static constexpr int N = 8;
  static __device__ __forceinline__ float sq(const uint4& v) { return sq8(v); }
  static __device__ __forceinline__ float one(__nv_bfloat16 x) { const float f = __bfloat162float(x); return f * f; }
};
template <> struct Vec<float> {
  using type = float4;
  static constexpr int N = 4;
  static __device__ __forceinline__ float sq(const float4& v) { return sq4(v); }
  static __device__ __forceinline__ float one(float x) { return x * x; }
};

// Sum of squares of one row of d elements, accumulated by the 32 lanes of a warp (not yet reduced).
template <typename T>
__device__ __forceinline__ float row_partial(const T* __restrict__ src, int d, int lane) {
  using V = typename Vec<T>::type;
  constexpr int VN = Vec<T>::N;
  float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, acc3 = 0.f;
  if ((d % VN) == 0) {
    const V* v = reinterpret_cast<const V*>(src);
    const int nv = d / VN;
    int i = lane;
    for (; i + 224 < nv; i += 256) {          // eight independent 16-byte loads in flight per lane
      const V x0 = __ldg(v + i), x1 = __ldg(v + i + 32), x2 = __ldg(v + i + 64), x3 = __ldg(v + i + 96);
      const V x4 = __ldg(v + i + 128), x5 = __ldg(v + i + 160), x6 = __ldg(v + i + 192), x7 = __ldg(v + i + 224);
      acc0 += Vec<T>::sq(x0); acc1 += Vec<T>::sq(x1); acc2 += Vec<T>::sq(x2); acc3 += Vec<T>::sq(x3);
      acc0 += Vec<T>::sq(x4); acc1 += Vec<T>::sq(x5); acc2 += Vec<T>::sq(x6); acc3 += Vec<T>::sq(x7);
    }
    for (; i + 96 < nv; i += 128) {
      const V x0 = __ldg(v + i), x1 = __ldg(v + i + 32), x2 = __ldg(v + i + 64), x3 = __ldg(v + i + 96);
      acc0 += Vec<T>::sq(x0); acc1 += Vec<T>::sq(x1); acc2 += Vec<T>::sq(x2); acc3 += Vec<T>::sq(x3);
    }
    for (; i < nv; i += 32) acc0 += Vec<T>::sq(__ldg(v + i));
  } else {
    for (int i = lane; i < d; i += 32) acc0 += Vec<T>::one(src[i]);
  }
  return (acc0 + acc1) + (acc2 + acc3);
}

}  // namespace
}  // namespace vcas
