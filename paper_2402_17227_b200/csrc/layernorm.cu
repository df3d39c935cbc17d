// SampleA in front of a layer that is not a matrix product (Sec. 4: SampleA sits at every layer; App. E: the
// sampled, rescaled gradient is multiplied by the layer's exact Jacobian): the backward of
// Y = LayerNorm(X) * gamma + beta.  Only the rows of kept data are read and computed; rows of dropped data
// get dX = 0.  HBM-bound: every kept row of X and dY is read once and held in registers; fixed summation orders.
#include "common.cuh"

namespace vcas {
namespace {

template <typename T> struct Ld;
template <> struct Ld<__nv_bfloat16> {
  static constexpr int N = 8;
  using V = uint4;
  static __device__ __forceinline__ void unpack(const uint4& v, float (&f)[8]) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(u[i] << 16); f[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u); }
  }
  // rounds to bf16, returns the stored values' sum of squares (not wanted: 0)
  static __device__ __forceinline__ float pack(const float (&f)[8], uint4& v, bool squares = true) {
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 t = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      o[i] = *reinterpret_cast<const uint32_t*>(&t);
    }
    v = make_uint4(o[0], o[1], o[2], o[3]);
    float sq = 0.f;
    if (squares) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float lo = __uint_as_float(o[i] << 16), hi = __uint_as_float(o[i] & 0xffff0000u);
        sq = fmaf(lo, lo, fmaf(hi, hi, sq));
      }
    }
    return sq;
  }
  static __device__ __forceinline__ float one(__nv_bfloat16 x) { return __bfloat162float(x); }
};
template <> struct Ld<float> {
  static constexpr int N = 4;
  using V = float4;
  static __device__ __forceinline__ void unpack(const float4& v, float (&f)[4]) { f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w; }
  static __device__ __forceinline__ float pack(const float (&f)[4], float4& v, bool squares = true) {
    v = make_float4(f[0], f[1], f[2], f[3]);
    if (!squares) return 0.f;
    return fmaf(f[0], f[0], fmaf(f[1], f[1], fmaf(f[2], f[2], f[3] * f[3])));
  }
  static __device__ __forceinline__ float one(float x) { return x; }
};

struct LnParams {
  const void* X; const void* gamma; const void* dY; void* dX;
  const float* scaleA; const int32_t* idxA; const int32_t* dropA; const int32_t* counts;
  float* mu; float* rstd;          // [R] per-row statistics kept for the column pass of wide rows
  float* a_out; int a_parts;       // optional row square-norms of the stored dX (first part; the others 0)
  float* partial;                  // [2][CTAs or row ranges][d] column partial sums
  float* dgamma; float* dbeta;
  int N, T, d, skip_dropped;
  float eps;
};

// Sum of one float over the G warps of a row group, in a fixed order; result in every lane.  slot: G floats per group.
template <int G>
__device__ __forceinline__ void group_sum(float (&v)[3], int n, float* slot, int gw, int group) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
    if (i < n) v[i] = warp_sum(v[i]);
  if (G > 1) {
    if ((threadIdx.x & 31) == 0)
      for (int i = 0; i < n; ++i) slot[gw * 3 + i] = v[i];
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(32 * G) : "memory");
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (i < n) {
        float t = 0.f;
        for (int w = 0; w < G; ++w) t += slot[w * 3 + i];
        v[i] = t;
      }
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(32 * G) : "memory");
  }
}

// G warps per row, VPL vectors of it a lane, the kept rows dealt out to the row groups of the grid in turn.  The row's
// statistics, dX and its share of the column sums dgamma = sum_r G_hat_r x_hat_r, dbeta = sum_r G_hat_r come from one read of X
// and dY; a lane keeps the column sums of its columns in registers over all its rows, the CTA adds its groups in order and
// stores one partial sum per column.  (With a second, column-wise pass over the rows the call on 16384 x 1024 at ratio 0.5
// took 87 us, 17 for the rows and 40 for the columns, one dependent load at a time.)
// Bound by instructions as much as by bytes: the values are widened once and worked on in pairs (f32x2), gamma is widened once
// for all rows.  1/sigma multiplies x - mean and the sum in brackets one after the other: as one factor 1/sigma^2 it left fp32's
// range for x of 1e17 or 1e-18 (16384 x 4096, ratio 0.5 and 1: 102.3 and 137.5 us so, 102.9 and 139.8 now).  A row is also a chain
// of a memory latency and two reductions, so the next row's loads are issued before the present one is worked on, and the zero
// rows of dropped data go out while the first is on its way.  (A row in four vectors a lane, widened in each pass and not loaded
// ahead: bf16, 16384 x 1024, ratio 0.5 35.2 us the call, now 32.6; ratio 1 43.9 and 39.2; 4096 columns 107 and 103, 2048 rows of
// 8192 53.5 and 39.2; fp32, 16384 x 4096 156 and 149.)
template <typename T, int G, int VPL, int WARPS, int CTAS>
__global__ void __launch_bounds__(WARPS * 32, CTAS) ln_kernel(LnParams P) {
  using L = Ld<T>;
  using V = typename L::V;
  constexpr int VN = L::N, GROUPS = WARPS / G;
  static_assert(GROUPS * G == WARPS && (G == 1 || GROUPS < 16), "whole groups, a named barrier each");
  __shared__ float s_slot[GROUPS][G * 3];
  extern __shared__ float s_col[];                   // [GROUPS][2][32 * G * VN] column sums on their way to the CTA's sum
  pdl_wait();      // the kept data come from the SampleA kernel
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, group = warp / G, gw = warp % G;
  const int cntA = P.counts[0], Tn = P.T, d = P.d;
  const int kept_rows = cntA * Tn;
  const int nv = d / VN;
  const float inv_d = 1.0f / (float)d;
  const int v0 = gw * 32 + lane;                     // this lane's vectors: v0, v0 + 32 G
  bool has[VPL];
  uint64_t w[VPL][VN / 2], ag[VPL][VN / 2], ab[VPL][VN / 2];
  auto widen = [](const V& v, uint64_t (&o)[VN / 2]) {
    float f[VN];
    L::unpack(v, f);
#pragma unroll
    for (int e = 0; e < VN / 2; ++e) o[e] = pack2(f[2 * e], f[2 * e + 1]);
  };
#pragma unroll
  for (int q = 0; q < VPL; ++q) {
    has[q] = v0 + q * 32 * G < nv;
#pragma unroll
    for (int e = 0; e < VN / 2; ++e) { w[q][e] = 0; ag[q][e] = 0; ab[q][e] = 0; }
    if (has[q]) widen(__ldg(reinterpret_cast<const V*>((const T*)P.gamma) + v0 + q * 32 * G), w[q]);
  }
  const int groups = gridDim.x * GROUPS, me = blockIdx.x * GROUPS + group;
  V xn[VPL], gn[VPL];                          // the next row, its number and 1/p
  size_t rn = 0;
  float scn = 0.f;
  int k = me / Tn, t = me - k * Tn;                  // the row to be loaded next: token t of the k-th kept datum
  const int dk = groups / Tn, dt = groups - dk * Tn;
  auto fetch = [&]() {
    const int n = P.idxA[k];
    rn = (size_t)n * Tn + t;
    scn = P.scaleA[n];
    k += dk;
    t += dt;
    if (t >= Tn) { t -= Tn; ++k; }
    const V* xv = reinterpret_cast<const V*>((const T*)P.X + rn * d);
    const V* gv = reinterpret_cast<const V*>((const T*)P.dY + rn * d);
#pragma unroll
    for (int q = 0; q < VPL; ++q)
      if (has[q]) xn[q] = __ldg(xv + v0 + q * 32 * G);
#pragma unroll
    for (int q = 0; q < VPL; ++q)
      if (has[q]) gn[q] = __ldg(gv + v0 + q * 32 * G);
  };
  if (me < kept_rows) fetch();
  if (!P.skip_dropped) {
    const int drop_rows = (P.N - cntA) * Tn;
    for (int i = me; i < drop_rows; i += groups) {
      const int kd = i / Tn;
      const size_t r = (size_t)P.dropA[kd] * Tn + (i - kd * Tn);
      V z;
      float zero[VN];
#pragma unroll
      for (int e = 0; e < VN; ++e) zero[e] = 0.f;
      L::pack(zero, z, false);
      for (int j = v0; j < nv; j += 32 * G) reinterpret_cast<V*>((T*)P.dX + r * d)[j] = z;
      if (P.a_out != nullptr && gw == 0)
        for (int j = lane; j < P.a_parts; j += 32) P.a_out[r * P.a_parts + j] = 0.f;
    }
  }
  for (int c = me; c < kept_rows; c += groups) {
    const size_t r = rn;
    const float sc = scn;
    uint64_t x[VPL][VN / 2], g[VPL][VN / 2];
#pragma unroll
    for (int q = 0; q < VPL; ++q)
      if (has[q]) { widen(xn[q], x[q]); widen(gn[q], g[q]); }
    if (c + groups < kept_rows) fetch();
    float sums[3] = {0.f, 0.f, 0.f};
    auto halves = [](uint64_t v) { float a, b; unpack2(v, a, b); return a + b; };
    uint64_t p0 = 0, p1 = 0, p2 = 0;
#pragma unroll
    for (int q = 0; q < VPL; ++q)
      if (has[q]) {
#pragma unroll
        for (int e = 0; e < VN / 2; ++e) p0 = add2(p0, x[q][e]);
      }
    sums[0] = halves(p0);
    group_sum<G>(sums, 1, s_slot[group], gw, group);
    const float mean = sums[0] * inv_d;
    // variance, and the two row sums of g_hat = G_hat * gamma that the Jacobian needs
    const uint64_t nmean = pack2(-mean, -mean), scale = pack2(sc, sc);
    p0 = 0;
#pragma unroll
    for (int q = 0; q < VPL; ++q)
      if (has[q]) {
#pragma unroll
        for (int e = 0; e < VN / 2; ++e) {
          x[q][e] = add2(x[q][e], nmean);
          g[q][e] = mul2(g[q][e], scale);
          const uint64_t gh = mul2(g[q][e], w[q][e]);
          p0 = fma2(x[q][e], x[q][e], p0);
          p1 = add2(p1, gh);
          p2 = fma2(gh, x[q][e], p2);
        }
      }
    sums[0] = halves(p0); sums[1] = halves(p1); sums[2] = halves(p2);
    group_sum<G>(sums, 3, s_slot[group], gw, group);
    const float rstd = rsqrtf(sums[0] * inv_d + P.eps);
    const float m1 = sums[1] * inv_d, m2 = sums[2] * rstd * inv_d;     // mean(g_hat), mean(g_hat * x_hat)
    const uint64_t nm1 = pack2(-m1, -m1), nm2 = pack2(-m2, -m2), inv = pack2(rstd, rstd);
    float sq[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < VPL; ++q)
      if (has[q]) {
        float o[VN];
#pragma unroll
        for (int e = 0; e < VN / 2; ++e) {
          const uint64_t xh = mul2(x[q][e], inv);
          // dX = (g_hat - m1 - x_hat m2) / sigma
          unpack2(mul2(fma2(xh, nm2, fma2(g[q][e], w[q][e], nm1)), inv), o[2 * e], o[2 * e + 1]);
          ag[q][e] = fma2(g[q][e], xh, ag[q][e]);
          ab[q][e] = add2(ab[q][e], g[q][e]);
        }
        V ov;
        sq[0] += L::pack(o, ov, P.a_out != nullptr);
        reinterpret_cast<V*>((T*)P.dX + r * d)[v0 + q * 32 * G] = ov;
      }
    if (P.a_out != nullptr) {                        // the same for the whole grid
      group_sum<G>(sq, 1, s_slot[group], gw, group);
      if (gw == 0)
        for (int j = lane; j < P.a_parts; j += 32) P.a_out[r * P.a_parts + j] = j == 0 ? sq[0] : 0.f;
    }
  }
  // the CTA's column sums, groups in order
  constexpr int W = 32 * G * VN;                     // columns of one q
#pragma unroll
  for (int q = 0; q < VPL; ++q) {
    if (q * 32 * G >= nv) break;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < VN / 2; ++e) {
      float* at = s_col + (gw * 32 + lane) * VN + 2 * e;
      unpack2(ag[q][e], at[(group * 2 + 0) * W], at[(group * 2 + 0) * W + 1]);
      unpack2(ab[q][e], at[(group * 2 + 1) * W], at[(group * 2 + 1) * W + 1]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * W; i += WARPS * 32) {
      const int which = i / W, col = q * W + (i - which * W);
      if (col >= d) continue;
      float t = 0.f;
#pragma unroll
      for (int gr = 0; gr < GROUPS; ++gr) t += s_col[(gr * 2 + which) * W + (i - which * W)];
      P.partial[((size_t)which * gridDim.x + blockIdx.x) * d + col] = t;
    }
  }
}

// Rows wider than sixteen warps hold in registers: two passes, one over rows and one over columns.
// One warp per row.  Work item c < cntA*T: token of a kept datum (compact order); the items after those are the
// rows of dropped data, which are zeroed (unless the caller's consumer never reads them).
template <typename T>
__global__ void __launch_bounds__(256) ln_row_kernel(LnParams P) {
  using L = Ld<T>;
  using V = typename L::V;
  constexpr int VN = L::N;
  pdl_wait();      // the kept data come from the SampleA kernel
  pdl_trigger();
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const int cntA = P.counts[0], Tn = P.T, d = P.d;
  const int kept_rows = cntA * Tn;
  const int total = P.skip_dropped ? kept_rows : P.N * Tn;
  const int nv = d / VN;
  const float inv_d = 1.0f / (float)d;
  for (int c = blockIdx.x * wpb + (threadIdx.x >> 5); c < total; c += gridDim.x * wpb) {
    if (c >= kept_rows) {        // a row of a dropped datum
      const int i = c - kept_rows, k = i / Tn;
      const size_t r = (size_t)P.dropA[k] * Tn + (i - k * Tn);
      V z;
      float zero[VN];
#pragma unroll
      for (int e = 0; e < VN; ++e) zero[e] = 0.f;
      L::pack(zero, z);
      for (int j = lane; j < nv; j += 32) reinterpret_cast<V*>((T*)P.dX + r * d)[j] = z;
      if (P.a_out != nullptr && lane < P.a_parts) P.a_out[r * P.a_parts + lane] = 0.f;
      continue;
    }
    const int k = c / Tn;
    const int n = P.idxA[k];
    const size_t r = (size_t)n * Tn + (c - k * Tn);
    const float sc = P.scaleA[n];
    const V* xv = reinterpret_cast<const V*>((const T*)P.X + r * d);
    const V* gv = reinterpret_cast<const V*>((const T*)P.dY + r * d);
    const V* wv = reinterpret_cast<const V*>((const T*)P.gamma);
    // pass 1: the row's mean
    float s = 0.f;
    for (int j = lane; j < nv; j += 32) {
      float x[VN];
      L::unpack(__ldg(xv + j), x);
#pragma unroll
      for (int e = 0; e < VN; ++e) s += x[e];
    }
    const float mean = warp_sum(s) * inv_d;
    // pass 2: variance, and the two row sums of g_hat = G_hat * gamma that the Jacobian needs
    float v2 = 0.f, s1 = 0.f, s2 = 0.f;
    for (int j = lane; j < nv; j += 32) {
      float x[VN], g[VN], w[VN];
      L::unpack(__ldg(xv + j), x);
      L::unpack(__ldg(gv + j), g);
      L::unpack(__ldg(wv + j), w);
#pragma unroll
      for (int e = 0; e < VN; ++e) {
        const float xc = x[e] - mean, gh = sc * g[e] * w[e];
        v2 = fmaf(xc, xc, v2);
        s1 += gh;
        s2 = fmaf(gh, xc, s2);
      }
    }
    v2 = warp_sum(v2); s1 = warp_sum(s1); s2 = warp_sum(s2);
    const float rstd = rsqrtf(v2 * inv_d + P.eps);
    const float m1 = s1 * inv_d, m2 = s2 * rstd * inv_d;     // mean(g_hat), mean(g_hat * x_hat)
    // pass 3: dX
    float sq = 0.f;
    for (int j = lane; j < nv; j += 32) {
      float x[VN], g[VN], w[VN], o[VN];
      L::unpack(__ldg(xv + j), x);
      L::unpack(__ldg(gv + j), g);
      L::unpack(__ldg(wv + j), w);
#pragma unroll
      for (int e = 0; e < VN; ++e) {
        const float xh = (x[e] - mean) * rstd, gh = sc * g[e] * w[e];
        o[e] = (gh - m1 - xh * m2) * rstd;
      }
      V ov;
      sq += L::pack(o, ov);
      reinterpret_cast<V*>((T*)P.dX + r * d)[j] = ov;
    }
    sq = warp_sum(sq);
    // the first 32 parts; a loop over all of them here left fewer loads in flight above (8192 columns in fp32: 90 us, not 78)
    if (lane == 0) {
      P.mu[r] = mean;
      P.rstd[r] = rstd;
      if (P.a_out != nullptr) P.a_out[r * P.a_parts] = sq;
    } else if (P.a_out != nullptr && lane < P.a_parts) {
      P.a_out[r * P.a_parts + lane] = 0.f;
    }
  }
}

// One thread per column, the kept rows cut into contiguous ranges (blockIdx.y): partial sums of
// dgamma = sum_r G_hat_r * x_hat_r and dbeta = sum_r G_hat_r in row order.
template <typename T>
__global__ void __launch_bounds__(256) ln_col_kernel(LnParams P) {
  pdl_wait();
  pdl_trigger();
  const int col = blockIdx.x * blockDim.x + threadIdx.x;
  const int Tn = P.T, d = P.d;
  const int rows = P.counts[0] * Tn;
  const int per = (rows + (int)gridDim.y - 1) / (int)gridDim.y;
  const int c0 = blockIdx.y * per, c1 = min(rows, c0 + per);
  if (col >= d) return;
  float ag = 0.f, ab = 0.f;
  for (int c = c0; c < c1; ++c) {
    const int k = c / Tn;
    const int n = P.idxA[k];
    const size_t r = (size_t)n * Tn + (c - k * Tn);
    const float g = P.scaleA[n] * Ld<T>::one(((const T*)P.dY)[r * d + col]);
    const float xh = (Ld<T>::one(((const T*)P.X)[r * d + col]) - P.mu[r]) * P.rstd[r];
    ag = fmaf(g, xh, ag);
    ab += g;
  }
  P.partial[(size_t)blockIdx.y * d + col] = ag;
  P.partial[(size_t)((int)gridDim.y + blockIdx.y) * d + col] = ab;
}

// Adds the partial sums of CTAs or row ranges: 32 columns per CTA, 32 warps over 32 ranges of them, the ranges in order.
// Latency-bound (a few hundred partial sums of a column, a row apart): a warp has eight loads in flight.
constexpr int ADD_WARPS = 32;
__global__ void __launch_bounds__(ADD_WARPS * 32) ln_add_kernel(LnParams P, int blocks) {
  __shared__ float s[ADD_WARPS][32];
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tiles = (P.d + 31) / 32;
  const int which = blockIdx.x / tiles, col = (blockIdx.x - which * tiles) * 32 + lane;
  const int per = (blocks + ADD_WARPS - 1) / ADD_WARPS, b0 = warp * per, b1 = min(blocks, b0 + per);
  float t = 0.f;
  if (col < P.d) {
    const float* src = P.partial + (size_t)which * blocks * P.d + col;
    for (int b = b0; b < b1; b += 8) {
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = b + q < b1 ? __ldcg(src + (size_t)(b + q) * P.d) : 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) t += v[q];
    }
  }
  s[warp][lane] = t;
  __syncthreads();
  if (warp == 0 && col < P.d) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < ADD_WARPS; ++w) v += s[w][lane];
    (which == 0 ? P.dgamma : P.dbeta)[col] = v;
  }
}

// The few row ranges of wide rows: one thread per column, the ranges in order.  (ln_add_kernel's CTAs of 1024 threads, 32 columns
// each, took 2 to 5 us longer for 8200 columns of 17 ranges.)  And the parts of the rows' square-norms past the 32 that the row
// kernel writes, which are 0.
__global__ void __launch_bounds__(256) ln_range_add_kernel(LnParams P, int ranges) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x, which = i / P.d, col = i - which * P.d;
  if (P.a_out != nullptr && P.a_parts > 32) {
    const int more = P.a_parts - 32, kept = P.counts[0] * P.T;
    const long total = (long)(P.skip_dropped ? kept : P.N * P.T) * more;
    for (long e = i; e < total; e += (long)gridDim.x * blockDim.x) {
      const int c = (int)(e / more), m = c < kept ? c : c - kept, k = m / P.T;
      const size_t r = (size_t)(c < kept ? P.idxA : P.dropA)[k] * P.T + (m - k * P.T);
      P.a_out[r * P.a_parts + 32 + (e - (long)c * more)] = 0.f;
    }
  }
  if (which > 1) return;
  const float* src = P.partial + (size_t)which * ranges * P.d + col;
  float t = 0.f;
#pragma unroll 8
  for (int r = 0; r < ranges; ++r) t += __ldcg(src + (size_t)r * P.d);
  (which == 0 ? P.dgamma : P.dbeta)[col] = t;
}

// WARPS warps a CTA, CTAS CTAs per SM
template <typename T, int G, int VPL, int WARPS, int CTAS>
cudaError_t run_rows(Handle* h, const LnParams& P, long rows, cudaStream_t st) {
  // fewer when there are fewer rows than row groups or the scratch (4 d^2 floats) is small
  constexpr int GROUPS = WARPS / G;
  long blocks = (rows + GROUPS - 1) / GROUPS;
  if (blocks > CTAS * h->num_sms) blocks = CTAS * h->num_sms;
  if (blocks > 2l * P.d) blocks = 2l * P.d;
  const size_t smem = (size_t)WARPS * 2 * 32 * Ld<T>::N * sizeof(float);
  cudaError_t e = launch_after(ln_kernel<T, G, VPL, WARPS, CTAS>, dim3((unsigned)blocks), dim3(WARPS * 32), smem, st, P);
  if (e == cudaSuccess)
    e = launch_after(ln_add_kernel, dim3(2 * ((P.d + 31) / 32)), dim3(ADD_WARPS * 32), 0, st, P, (int)blocks);
  h->launches += 2;
  return e != cudaSuccess ? e : cudaGetLastError();
}
template <typename T>
cudaError_t run_ln(Handle* h, const LnParams& P, long rows, cudaStream_t st) {
  // The 16-byte vectors of a row decide; a group holds 32 G VPL.  Groups that fit leave no warp with a half-empty row to wait
  // for (powers of two of two vectors a lane, 16384 rows at ratio 0.5 and so: bf16, 576 columns 31.1 and 29.0 us, 1088 47.4 and
  // 41.3, 2560 81.1 and 69.9; fp32, 320 25.2 and 23.6, 1280 72.2 and 61.8, 2560 124 and 104).  Three and four vectors a lane have
  // registers for the next row in fp32 only, in bf16 three with twelve warps an SM; in fp32 they beat more warps a row, which wait for
  // one another (4096 columns by sixteen warps 158 us, by eight 149).  One CTA an SM halves the column sums to be added up (bf16,
  // 2048 rows of 2048 18.8 and 17.8 us); fp32, 2048 columns: in CTAs of one row group, four an SM, 2048 rows take 21.9 us, in one
  // CTA 19.7; 16384 rows at ratio 1 98.8 and 106.3.
  const int nv = P.d / Ld<T>::N;
  // Few rows, of which a group has one at most: more and smaller CTAs start sooner (256 rows of 768 in bf16, the kernels alone: by
  // two warps a row in CTAs of eight 10.4 us, by one in CTAs of twelve 11.3; 512 rows of 3072 in fp32 by sixteen warps 14.2, by eight
  // 15.6; up to 2048 rows of 4096 so).
  const bool few = rows <= 512;
  if constexpr (sizeof(T) == 2) {
    if (nv <= 64) return run_rows<T, 1, 2, 8, 2>(h, P, rows, st);
    if (nv <= 128 && few) return run_rows<T, 2, 2, 8, 2>(h, P, rows, st);
    if (nv <= 96) return run_rows<T, 1, 3, 12, 1>(h, P, rows, st);
    if (nv <= 128) return run_rows<T, 2, 2, 16, 1>(h, P, rows, st);
    if (nv <= 192) return run_rows<T, 3, 2, 12, 1>(h, P, rows, st);
    if (nv <= 256) return few ? run_rows<T, 4, 2, 8, 2>(h, P, rows, st) : run_rows<T, 4, 2, 16, 1>(h, P, rows, st);
    if (nv <= 320) return run_rows<T, 5, 2, 15, 1>(h, P, rows, st);
    if (nv <= 512) return run_rows<T, 8, 2, 8, 2>(h, P, rows, st);
    if (nv <= 1024) return run_rows<T, 16, 2, 16, 1>(h, P, rows, st);
  } else {
    if (nv <= 64) return run_rows<T, 1, 2, 8, 2>(h, P, rows, st);
    if (nv <= 96 && !few) return run_rows<T, 1, 3, 8, 2>(h, P, rows, st);
    if (nv <= 128) return run_rows<T, 2, 2, 8, 2>(h, P, rows, st);
    if (nv <= 192) return run_rows<T, 2, 3, 8, 2>(h, P, rows, st);
    if (nv <= 256) return run_rows<T, 4, 2, 8, 2>(h, P, rows, st);
    if (nv <= 384 && !few) return run_rows<T, 4, 3, 16, 1>(h, P, rows, st);
    if (nv <= 480 && !few) return run_rows<T, 5, 3, 15, 1>(h, P, rows, st);
    if (nv <= 512) return rows > 4096 ? run_rows<T, 4, 4, 4, 4>(h, P, rows, st) : run_rows<T, 8, 2, 16, 1>(h, P, rows, st);
    if (nv <= 768 && !few) return run_rows<T, 8, 3, 8, 2>(h, P, rows, st);
    if (nv <= 1024) return rows > 2048 ? run_rows<T, 8, 4, 8, 2>(h, P, rows, st) : run_rows<T, 16, 2, 16, 1>(h, P, rows, st);
  }
  const int col_blocks = (P.d + 255) / 256;
  const int chunks = 4 * h->num_sms > col_blocks ? 4 * h->num_sms / col_blocks : 1;
  const long blocks = (rows + 7) / 8 < (1l << 20) ? (rows + 7) / 8 : (1l << 20);
  cudaError_t e = launch_after(ln_row_kernel<T>, dim3((unsigned)blocks), dim3(256), 0, st, P);
  if (e == cudaSuccess) e = launch_after(ln_col_kernel<T>, dim3(col_blocks, chunks), dim3(256), 0, st, P);
  if (e == cudaSuccess) e = launch_after(ln_range_add_kernel, dim3((unsigned)((2l * P.d + 255) / 256)), dim3(256), 0, st, P, chunks);
  h->launches += 3;
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_layernorm_bwd(Handle* h, const void* X, const void* gamma, const void* dY, float eps, void* dX,
                                 float* a_out, bool skip_dropped, float* dgamma, float* dbeta, cudaStream_t st) {
  const vcas_layer_desc& d = h->desc;
  const Workspace& ws = h->ws;
  LnParams P;
  P.X = X; P.gamma = gamma; P.dY = dY; P.dX = dX;
  P.scaleA = ws.scaleA; P.idxA = ws.idxA; P.dropA = ws.dropA; P.counts = ws.counts;
  P.mu = ws.w; P.rstd = ws.q;
  P.a_out = a_out; P.a_parts = a_out_parts(d.d_in);
  P.partial = ws.Gs;                                 // Gs, Gact, mean and m2 are neighbours: 4 d^2 floats
  P.dgamma = dgamma; P.dbeta = dbeta;
  P.N = d.N; P.T = d.T; P.d = d.d_in; P.skip_dropped = skip_dropped ? 1 : 0;
  P.eps = eps;
  const long rows = (long)d.N * d.T;
  return d.dtype == VCAS_DTYPE_BF16 ? run_ln<__nv_bfloat16>(h, P, rows, st) : run_ln<float>(h, P, rows, st);
}

}  // namespace vcas
