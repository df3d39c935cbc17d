// Rows of eight consecutive elements in registers, and their cut into bf16 parts.
#pragma once

#include "common.cuh"

namespace vcas {

__device__ __forceinline__ uint32_t bf16x2_rn(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

template <typename T> struct Vec8;
template <> struct Vec8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = __ldg(reinterpret_cast<const float4*>(p));
    b = __ldg(reinterpret_cast<const float4*>(p) + 1);
  }
  __device__ __forceinline__ void get(float (&f)[8]) const {
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
  }
};
template <> struct Vec8<__nv_bfloat16> {
  uint4 v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { v = __ldg(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ void get(float (&f)[8]) const {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(u[i] << 16); f[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u); }
  }
};

__device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&v)[8]) {
  *reinterpret_cast<uint4*>(p) = make_uint4(bf16x2_rn(v[0], v[1]), bf16x2_rn(v[2], v[3]), bf16x2_rn(v[4], v[5]),
                                            bf16x2_rn(v[6], v[7]));
}

// x = x1 + x2 + x3 exactly (eight significant bits each, rounded to nearest: |x2| <= 2^-9 |x|, |x3| <= 2^-18 |x|), the
// parts of eight elements stored at dst, dst + stride, dst + 2 stride.  An infinite, NaN or almost overflowing x, which
// has no finite x1, is all in its third part, which meets one part of the other operand only (inf y = inf y1; beside
// other parts it would give inf - inf).
__device__ __forceinline__ void store_parts3(const float (&f)[8], __nv_bfloat16* dst, size_t stride) {
  uint32_t p1[4], p2[4], p3[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float x0 = f[2 * e], x1 = f[2 * e + 1];
    const bool ok0 = fabsf(x0) < 3.3e38f, ok1 = fabsf(x1) < 3.3e38f;
    p1[e] = bf16x2_rn(ok0 ? x0 : 0.f, ok1 ? x1 : 0.f);
    const float r0 = x0 - __uint_as_float(p1[e] << 16), r1 = x1 - __uint_as_float(p1[e] & 0xffff0000u);
    p2[e] = bf16x2_rn(ok0 ? r0 : 0.f, ok1 ? r1 : 0.f);
    p3[e] = bf16x2_rn(r0 - __uint_as_float(p2[e] << 16), r1 - __uint_as_float(p2[e] & 0xffff0000u));
  }
  *reinterpret_cast<uint4*>(dst) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
  *reinterpret_cast<uint4*>(dst + stride) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
  *reinterpret_cast<uint4*>(dst + 2 * stride) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
}

}  // namespace vcas
