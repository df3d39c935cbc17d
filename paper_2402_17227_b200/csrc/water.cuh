// Water-filling for q = min(1, c w) by one CTA, shared by SampleW and the variance probe.
#pragma once

#include "common.cuh"

namespace vcas {
namespace {

constexpr int SAMPLER_THREADS = 1024;
constexpr int WATER_ROUNDS = 128;     // rounds of the water-filling before it is reported as not converged
constexpr int SAMPLE_W_SMEM_ROWS = 56 * 1024;     // scores that fit a CTA's shared memory (224 KB)

// How q follows from a row's score once sample_w_kernel has run: fix[1] = mode, fix[0] = c.
constexpr int Q_ZERO = 0;     // nothing to keep (no score is positive, or the budget is 0)
constexpr int Q_ONES = 1;     // the budget covers every positive score: q = [w > 0]
constexpr int Q_CAPPED = 2;   // q = min(1, c w)
constexpr int Q_GIVEN = 3;    // q is read from the caller's q_in

__device__ __forceinline__ float q_of(int mode, float c, float w, const float* q_in, int r) {
  if (mode == Q_CAPPED) {
    if (!(w > 0.f)) return 0.f;
    const float cx = c * w;
    return cx >= 1.0f ? 1.f : cx;
  }
  if (mode == Q_ONES) return w > 0.f ? 1.f : 0.f;
  if (mode == Q_GIVEN) return q_in[r];
  return 0.f;
}
struct WShared {
  float part_f[2][32];
  int part_i[2][32];
  int scan[33];
};

// Block-wide sum of one float and one int in a fixed order (lanes by shuffle tree, then the 32
// warp totals by the same tree, which every warp runs for itself so that one barrier suffices; the
// buffers alternate with `parity`, and a buffer is rewritten only after a later barrier).  fp32 on
// purpose: this is a single-CTA kernel, and double-precision arithmetic concentrated on one SM was
// measured to dominate its run time; a tree sum of non-negative fp32 terms is accurate to about
// 1e-6, inside the 2e-5 the probabilities are specified to.
__device__ __forceinline__ void fast_sum(float& s, int& c, WShared* sh, int parity) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  s = warp_sum(s);
  c = __reduce_add_sync(0xffffffffu, c);
  if (lane == 0) { sh->part_f[parity][warp] = s; sh->part_i[parity][warp] = c; }
  __syncthreads();
  s = warp_sum(sh->part_f[parity][lane]);
  c = __reduce_add_sync(0xffffffffu, sh->part_i[parity][lane]);
}

// The fixed point itself; part(c, Su, ks): sum of the positive scores with c w < 1 and number of the others of a thread.
template <typename Part>
__device__ __forceinline__ bool water_rounds(float S, int nz, float budget, WShared* sh, int& mode, float& c, Part part) {
  int parity = 0;
  fast_sum(S, nz, sh, parity); parity ^= 1;
  c = 0.f;
  if (nz == 0 || budget <= 0.f) { mode = Q_ZERO; return true; }
  if ((float)nz <= budget) { mode = Q_ONES; return true; }
  mode = Q_CAPPED;
  c = budget / S;
  int k = 0;
  for (int iter = 0; iter < WATER_ROUNDS; ++iter) {
    float Su = 0.f;
    int ks = 0;
    part(c, Su, ks);
    fast_sum(Su, ks, sh, parity); parity ^= 1;
    if (ks == k) return true;
    k = ks;
    if (Su > 0.f) {
      const float cn = (budget - (float)k) / Su;
      c = cn > c ? cn : c;
    }
  }
  return false;
}

// c with sum_i min(1, c w_i) = budget over the n scores w by SAMPLER_THREADS threads: every round is one pass over the
// scores and one block-wide sum.  Returns false if it has not converged after WATER_ROUNDS rounds.
__device__ __forceinline__ bool water_fill(const float* w, int n, float budget, WShared* sh, int& mode, float& c) {
  const int tid = threadIdx.x;
  float S = 0.f;
  int nz = 0;
  for (int i = tid; i < n; i += SAMPLER_THREADS) {
    const float x = w[i];
    if (x > 0.f) { S += x; ++nz; }
  }
  return water_rounds(S, nz, budget, sh, mode, c, [&](float at, float& Su, int& ks) {
    for (int i = tid; i < n; i += SAMPLER_THREADS) {
      const float x = w[i];
      if (x > 0.f) {
        if (at * x >= 1.0f) ++ks; else Su += x;
      }
    }
  });
}
// The same over scores in registers, 0 where there are none.
template <int SLOTS>
__device__ __forceinline__ bool water_fill_regs(const float (&w)[SLOTS], float budget, WShared* sh, int& mode, float& c) {
  float S = 0.f;
  int nz = 0;
#pragma unroll
  for (int j = 0; j < SLOTS; ++j)
    if (w[j] > 0.f) { S += w[j]; ++nz; }
  return water_rounds(S, nz, budget, sh, mode, c, [&](float at, float& Su, int& ks) {
#pragma unroll
    for (int j = 0; j < SLOTS; ++j)
      if (w[j] > 0.f) {
        if (at * w[j] >= 1.0f) ++ks; else Su += w[j];
      }
  });
}

}  // namespace
}  // namespace vcas
