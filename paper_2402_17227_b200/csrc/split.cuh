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

// x = x1 + x2 + x3 in bf16 parts of eight significant bits each, the parts of eight elements stored at dst, dst + stride,
// dst + 2 stride.  Exact down to the smallest bf16, 2^-133 (|x| above 2^-109 keeps its 24 bits; 0 < |x| < 2^-134 has x1 = 0).
//
// ROUND, for a product of two cut operands: rounded to nearest, |x2| <= 2^-9 |x|, |x3| <= 2^-18 |x|, so that what the
// six part products leave out is small.  (x1 of an |x| that would round to infinity is cut instead.)  An infinite or NaN x is
// all in x3, which meets y1 only, beside x1 = +-1 and x2 = 0: inf y = inf y1, inf inf = inf 1 + 1 inf, inf 0 = NaN.
//
// Otherwise, for a product with an operand y that is its own single part, where all three parts meet y: cut, not rounded, so
// that all parts have the sign of x, and none is 0 unless x is: inf y must not become inf - inf or 0 inf.  What is put in
// place of a 0, 2^-126, is below 2^-26 |x|.
__device__ __forceinline__ float cut_bf16(float x) { return __uint_as_float(__float_as_uint(x) & 0xffff0000u); }
__device__ __forceinline__ void store_parts(const uint32_t (&p1)[4], const uint32_t (&p2)[4], const uint32_t (&p3)[4],
                                            __nv_bfloat16* dst, size_t stride) {
  *reinterpret_cast<uint4*>(dst) = make_uint4(p1[0], p1[1], p1[2], p1[3]);
  *reinterpret_cast<uint4*>(dst + stride) = make_uint4(p2[0], p2[1], p2[2], p2[3]);
  *reinterpret_cast<uint4*>(dst + 2 * stride) = make_uint4(p3[0], p3[1], p3[2], p3[3]);
}
// Eight values of which one at least is infinite, NaN or, with ROUND, above 3.38e38: one element after the other, out of the way
// of the others (in line it cost the pass over 4950 rows, 776 + 1000 wide, 3 us).
template <bool ROUND>
__device__ __noinline__ void store_parts3_special(float4 u, float4 v, __nv_bfloat16* dst, size_t stride) {
  const float f[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
  uint32_t p[3][4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float part[3][2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float x = f[2 * e + i];
      if (fabsf(x) <= 3.402823466e38f) {
        part[0][i] = !ROUND || fabsf(x) > 3.38e38f ? cut_bf16(x) : __bfloat162float(__float2bfloat16_rn(x));
        const float r = x - part[0][i];
        part[1][i] = ROUND ? __bfloat162float(__float2bfloat16_rn(r)) : cut_bf16(r);
        part[2][i] = r - part[1][i];
      } else {
        part[0][i] = copysignf(1.f, x);
        part[1][i] = 0.f;
        part[2][i] = x;
      }
      if (!ROUND && fabsf(x) >= 7.9e-31f)
        for (int k = 1; k < 3; ++k)
          if (part[k][i] == 0.f) part[k][i] = copysignf(1.17549435e-38f, x);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k][e] = bf16x2_rn(part[k][0], part[k][1]);
  }
  store_parts(p[0], p[1], p[2], dst, stride);
}
template <bool ROUND>
__device__ __forceinline__ void store_parts3(const float (&f)[8], __nv_bfloat16* dst, size_t stride) {
  uint32_t most = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) most = max(most, __float_as_uint(f[e]) & 0x7fffffffu);
  if (most > (ROUND ? 0x7f7e0000u : 0x7f7fffffu)) {
    store_parts3_special<ROUND>(make_float4(f[0], f[1], f[2], f[3]), make_float4(f[4], f[5], f[6], f[7]), dst, stride);
    return;
  }
  uint32_t p1[4], p2[4], p3[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float x0 = f[2 * e], x1 = f[2 * e + 1];
    if (ROUND) {
      p1[e] = bf16x2_rn(x0, x1);
      const float r0 = x0 - __uint_as_float(p1[e] << 16), r1 = x1 - __uint_as_float(p1[e] & 0xffff0000u);
      p2[e] = bf16x2_rn(r0, r1);
      p3[e] = bf16x2_rn(r0 - __uint_as_float(p2[e] << 16), r1 - __uint_as_float(p2[e] & 0xffff0000u));
    } else {
      // `tiny` vanishes in the rounding of anything that is not 0
      const float t0 = fabsf(x0) >= 7.9e-31f ? copysignf(1.17549435e-38f, x0) : 0.f;
      const float t1 = fabsf(x1) >= 7.9e-31f ? copysignf(1.17549435e-38f, x1) : 0.f;
      const float r0 = x0 - cut_bf16(x0) + t0, r1 = x1 - cut_bf16(x1) + t1;
      const float s0 = r0 - cut_bf16(r0) + t0, s1 = r1 - cut_bf16(r1) + t1;
      p1[e] = __byte_perm(__float_as_uint(x0), __float_as_uint(x1), 0x7632);
      p2[e] = __byte_perm(__float_as_uint(r0), __float_as_uint(r1), 0x7632);
      p3[e] = bf16x2_rn(s0, s1);
    }
  }
  store_parts(p1, p2, p3, dst, stride);
}

}  // namespace vcas
