// Keep probabilities, Philox Bernoulli masks and compaction for SampleA and SampleW
// (Sec. 4.1, 4.2).  Everything stays on the device: the kept counts are written to the workspace
// and read by the product kernels.  The stage is a chain of small kernels:
//   norms_sample_a_kernel  of few rows: their norms (else score.cu) and what follows in one launch;
//   sample_a_kernel   ||G_n||_F on a few CTAs, the last of which draws: p_n, mask, kept / dropped data (the dX product can
//                     start here);
//   scores_x_kernel   (score.cu) many CTAs: leverage scores and uniforms of the rows of kept data;
//   sample_w_small_kernel, sample_w_kernel  one CTA, scores in registers or in shared memory: the water-filling for q = min(1, c w)
//                     - a handful of block-wide sums - then the masks' counts per chunk of 32 rows and their prefix sums;
//   emit_pack_kernel  many CTAs: kept-row list, 1/(p q), and the compact operands of the dW product (emit_rows_kernel: without).
// Only the scalar fixed point and a scan over R/32 counts run on a single SM.
#include <atomic>

#include "rows.cuh"
#include "split.cuh"
#include "water.cuh"

namespace vcas {
namespace {


struct Scratch {
  double d[32];
  int i[32];
  int scan[33];
  double bd;
  int bi;
};

// Block-wide sum of one double and one int, result in every thread.
__device__ void block_sum(double& s, int& c, Scratch* sc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  s = warp_sum(s);
  c = warp_sum(c);
  if (lane == 0) { sc->d[warp] = s; sc->i[warp] = c; }
  __syncthreads();
  if (warp == 0) {
    double x = lane < (int)(blockDim.x >> 5) ? sc->d[lane] : 0.0;
    int y = lane < (int)(blockDim.x >> 5) ? sc->i[lane] : 0;
    x = warp_sum(x);
    y = warp_sum(y);
    if (lane == 0) { sc->bd = x; sc->bi = y; }
  }
  __syncthreads();
  s = sc->bd;
  c = sc->bi;
  __syncthreads();
}

// Keep probabilities proportional to v, capped at 1, summing to `budget` (the minimiser of
// sum (1-p)/p v^2 under that budget): p = min(1, c v).  The saturated set is grown from
// empty; c only increases, so the iteration reaches the least fixed point, which is the
// unique solution.  Returns false if it has not converged after WATER_ROUNDS rounds.
__device__ bool capped_prop_block(const float* v, int n, double budget, float* p, Scratch* sc) {
  const int tid = threadIdx.x, nt = blockDim.x;
  double S = 0.0;
  int nz = 0;
  for (int i = tid; i < n; i += nt) {
    const float x = v[i];
    if (x > 0.f) { S += (double)x; ++nz; }
  }
  block_sum(S, nz, sc);
  if (nz == 0 || budget <= 0.0) {
    for (int i = tid; i < n; i += nt) p[i] = 0.f;
    return true;
  }
  if ((double)nz <= budget) {
    for (int i = tid; i < n; i += nt) p[i] = v[i] > 0.f ? 1.f : 0.f;
    return true;
  }
  double c = budget / S;
  int k = 0;
  bool converged = false;
  for (int iter = 0; iter < WATER_ROUNDS; ++iter) {
    double Su = 0.0;
    int ks = 0;
    for (int i = tid; i < n; i += nt) {
      const float x = v[i];
      if (x > 0.f) {
        if (c * (double)x >= 1.0) ++ks; else Su += (double)x;
      }
    }
    block_sum(Su, ks, sc);
    if (ks == k) { converged = true; break; }
    k = ks;
    if (Su > 0.0) {
      const double cn = (budget - (double)k) / Su;
      c = cn > c ? cn : c;
    }
  }
  for (int i = tid; i < n; i += nt) {
    const float x = v[i];
    float r = 0.f;
    if (x > 0.f) {
      const double cx = c * (double)x;
      r = cx >= 1.0 ? 1.f : (float)cx;
    }
    p[i] = r;
  }
  return converged;
}

// Ordered compaction of the indices i < n with keep(i): emit(i, position).  Returns the count.
template <typename KeepFn, typename EmitFn>
__device__ int block_compact(int n, KeepFn keep, EmitFn emit, Scratch* sc) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  int base = 0;
  for (int start = 0; start < n; start += blockDim.x) {
    const int i = start + tid;
    const bool k = (i < n) && keep(i);
    const unsigned ballot = __ballot_sync(0xffffffffu, k);
    const int wofs = __popc(ballot & ((1u << lane) - 1u));
    if (lane == 0) sc->scan[warp] = __popc(ballot);
    __syncthreads();
    if (warp == 0) {
      const int v = lane < nw ? sc->scan[lane] : 0;
      int incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      sc->scan[lane] = incl - v;
      if (lane == 31) sc->scan[32] = incl;
    }
    __syncthreads();
    if (k) emit(i, base + sc->scan[warp] + wofs);
    base += sc->scan[32];
    __syncthreads();
  }
  return base;
}

// ------------------------------------------------------------------------------ SampleA
struct SampleAParams {
  const float* a; int a_parts;
  const int32_t* alive; const int32_t* alive_cnt;
  int N, T;
  float rho;
  const float* p_in;
  uint64_t seed;
  float* g; float* p; float* scaleA;
  int32_t* idxA; int32_t* dropA; int32_t* counts;
  int32_t* kept_out; int32_t* kept_cnt_out;
  int32_t* status;
  float* gk;                       // [N] norms of the alive data, in the order of their list
  int32_t* ticket;                 // CTAs that have finished; zero between launches
};

constexpr int SAMPLE_A_THREADS = 256;
constexpr int SAMPLE_A_WARP_LEN = 1024;    // longest sum one warp takes

// Sum of the len floats of one datum by a CTA, in a fixed order; result in thread 0.
__device__ __forceinline__ float datum_sqnorm_cta(const float* an, int len, float* s_part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  int t = threadIdx.x;
  for (; t + 3 * SAMPLE_A_THREADS < len; t += 4 * SAMPLE_A_THREADS)
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] += __ldcg(an + t + k * SAMPLE_A_THREADS);
  for (; t < len; t += SAMPLE_A_THREADS) s[0] += __ldcg(an + t);
  const float w = warp_sum((s[0] + s[1]) + (s[2] + s[3]));
  if (lane == 0) s_part[warp] = w;
  __syncthreads();
  float r = 0.f;
  if (threadIdx.x == 0)
    for (int i = 0; i < SAMPLE_A_THREADS / 32; ++i) r += s_part[i];
  __syncthreads();
  return r;
}

// The number of alive data.  A caller's list is not trusted: a length outside [0, N] or an entry outside [0, N) is reported as
// VCAS_ERR_BAD_ARG in the status word and not followed.
__device__ __forceinline__ int alive_data(const SampleAParams& P) {
  if (P.alive == nullptr) return P.N;
  const int nd = *P.alive_cnt;
  if (nd >= 0 && nd <= P.N) return nd;
  if (threadIdx.x == 0 && blockIdx.x == 0) atomicExch(P.status, (int32_t)VCAS_ERR_BAD_ARG);
  return min(max(nd, 0), P.N);
}
// p, the masks and the lists from the data's norms, by the first warp of a CTA; the others store the norms.
template <int SLOTS>
__device__ __forceinline__ void draw_a(const SampleAParams& P, const float* s_g) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) {
    SampleAOut o;
    o.p = P.p; o.scaleA = P.scaleA; o.idxA = P.idxA; o.dropA = P.dropA; o.idx_copy = P.kept_out;
    const int kept = sample_a_warp<SLOTS>(s_g, P.N, P.rho, P.p_in, P.seed, o, lane);
    if (lane == 0) {
      P.counts[0] = kept;
      if (P.kept_cnt_out != nullptr) *P.kept_cnt_out = kept;
    }
  } else {
    for (int n = threadIdx.x - 32; n < P.N; n += SAMPLE_A_THREADS - 32) P.g[n] = s_g[n];
  }
}

// SampleA (Sec. 4.1) for N <= 32 * SLOTS data.  The CTAs share the data (only the alive ones are read; the others have norm
// 0): one warp sums a datum's T row square-norms, or, where a producer's partial sums make that many more, a CTA.  The CTA
// that finishes last finds p, draws the masks and writes the lists in one warp, whose lanes hold SLOTS data each: the
// smallest SLOTS that fits, since every slot costs a Philox block and a term in every round.  (With one CTA for all sums a
// chained layer's 1 MB of partial sums took 30 us, and 64 data in 32 slots 18 us instead of 5.)
template <int SLOTS>
__global__ void __launch_bounds__(SAMPLE_A_THREADS) sample_a_kernel(SampleAParams P) {
  __shared__ float s_g[32 * SLOTS];
  __shared__ float s_part[SAMPLE_A_THREADS / 32];
  __shared__ int s_last;
  pdl_wait();      // the row norms come from the kernel before this one
  pdl_trigger();   // the dX product kernel may set itself up meanwhile
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nd = alive_data(P);
  const int len = P.T * P.a_parts;
  if (len <= SAMPLE_A_WARP_LEN) {
    for (int k = blockIdx.x * (SAMPLE_A_THREADS / 32) + warp; k < nd; k += gridDim.x * (SAMPLE_A_THREADS / 32)) {
      const int n = P.alive != nullptr ? P.alive[k] : k;
      const float s = (unsigned)n < (unsigned)P.N ? datum_sqnorm_warp(P.a + (size_t)n * len, len, lane) : 0.f;
      if (lane == 0) P.gk[k] = sqrtf(s);
    }
  } else {
    for (int k = blockIdx.x; k < nd; k += gridDim.x) {
      const int n = P.alive != nullptr ? P.alive[k] : k;
      if ((unsigned)n >= (unsigned)P.N) continue;
      const float s = datum_sqnorm_cta(P.a + (size_t)n * len, len, s_part);
      if (threadIdx.x == 0) P.gk[k] = sqrtf(s);
    }
  }
  if (gridDim.x > 1) {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(P.ticket, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) *P.ticket = 0;
  }
  for (int n = threadIdx.x; n < 32 * SLOTS; n += SAMPLE_A_THREADS) s_g[n] = 0.f;
  __syncthreads();
  for (int k = threadIdx.x; k < nd; k += SAMPLE_A_THREADS) {
    const int n = P.alive != nullptr ? P.alive[k] : k;
    if ((unsigned)n < (unsigned)P.N) s_g[n] = __ldcg(P.gk + k);
    else atomicExch(P.status, (int32_t)VCAS_ERR_BAD_ARG);
  }
  __syncthreads();
  draw_a<SLOTS>(P, s_g);
}

// Row square-norms of dY and SampleA of N <= 32 data in one launch, for few rows: a warp per row, and the CTA that finishes last
// sums up the data, a warp each, and draws.  The sums are those of the two kernels, in the same order.  Saves a launch, 2.5 to
// 3.4 us on the host, and its start on the GPU (whole calls, two launches and one: 2048 rows of 4096, 55.3 and 51.0 us; of 3072,
// 38.9 and 36.8; of 1000, 41.8 and 40.8; 3200 of 4096, 50.5 and 46.3; 256 of 256, 25.8 and 23.5).  With more rows the wait for
// the last CTA takes back what it saves (4096 of 3072: 40.7 and 39.6 in bf16, 90.0 and 90.6 in fp32; of 256, 31.2 and 31.6; 8192:
// 46.9 and 48.7), and with more data their sums by one CTA cost more (100 of 16 rows: 28.9 and 35.0).  LayerNorm and scoring calls
// gain the launch on the host (LayerNorm, 256 to 3072 rows of 256 to 1024: 18.2 and 16.0 us; eight scoring calls 0.97 to 1.00 of the
// time, 1576 rows of 768 1.04, the kernels alone 0.94 for 2048 rows of 3072 to 1.07 for 2048 of 1024 in fp32).
constexpr int FUSED_MAX_N = 32, FUSED_MAX_ROWS = 3200;
template <typename T>
__global__ void __launch_bounds__(SAMPLE_A_THREADS) norms_sample_a_kernel(const T* __restrict__ dY, int d_out, float* __restrict__ a,
                                                                          SampleAParams P) {
  __shared__ float s_g[FUSED_MAX_N];
  __shared__ int s_last;
  pdl_trigger();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = gridDim.x * (SAMPLE_A_THREADS / 32);
  const int nd = alive_data(P);
  for (int c = blockIdx.x * (SAMPLE_A_THREADS / 32) + warp; c < nd * P.T; c += warps) {
    const int k = c / P.T, n = P.alive != nullptr ? P.alive[k] : k;
    if ((unsigned)n >= (unsigned)P.N) continue;          // reported below
    const int r = n * P.T + (c - k * P.T);
    const float sq = warp_sum(row_partial<T>(dY + (size_t)r * d_out, d_out, lane));
    if (lane == 0) a[r] = sq;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(P.ticket, 1) == (int)gridDim.x - 1;
  if (threadIdx.x < FUSED_MAX_N) s_g[threadIdx.x] = 0.f;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (threadIdx.x == 0) *P.ticket = 0;
  for (int k = warp; k < nd; k += SAMPLE_A_THREADS / 32) {
    const int n = P.alive != nullptr ? P.alive[k] : k;
    if ((unsigned)n >= (unsigned)P.N) {
      if (lane == 0) atomicExch(P.status, (int32_t)VCAS_ERR_BAD_ARG);
      continue;
    }
    const float s = datum_sqnorm_warp(a + (size_t)n * P.T, P.T, lane);
    if (lane == 0) s_g[n] = sqrtf(s);
  }
  __syncthreads();
  draw_a<1>(P, s_g);
}

// The same for batches of more than 1024 data: one CTA over global memory.
__global__ void __launch_bounds__(SAMPLER_THREADS) sample_a_big_kernel(SampleAParams P) {
  __shared__ Scratch sc;
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int N = P.N;
  for (int n = tid; n < N; n += nt) P.g[n] = 0.f;
  __syncthreads();
  int nd = N;
  if (P.alive != nullptr) {
    nd = *P.alive_cnt;
    if (nd < 0 || nd > N) {
      if (tid == 0) atomicExch(P.status, (int32_t)VCAS_ERR_BAD_ARG);
      nd = min(max(nd, 0), N);
    }
  }
  const int len = P.T * P.a_parts;
  for (int k = warp; k < nd; k += nw) {
    const int n = P.alive != nullptr ? P.alive[k] : k;
    if ((unsigned)n >= (unsigned)N) {
      if (lane == 0) atomicExch(P.status, (int32_t)VCAS_ERR_BAD_ARG);
      continue;
    }
    const float s = datum_sqnorm_warp(P.a + (size_t)n * len, len, lane);
    if (lane == 0) P.g[n] = sqrtf(s);
  }
  __syncthreads();
  if (P.p_in != nullptr) {
    for (int n = tid; n < N; n += nt) P.p[n] = P.p_in[n];
  } else if (!capped_prop_block(P.g, N, (double)N * (double)P.rho, P.p, &sc)) {
    if (tid == 0) atomicExch(P.status, (int32_t)VCAS_ERR_INTERNAL);
  }
  __syncthreads();
  for (int n = tid; n < N; n += nt) {
    const float pn = P.p[n];
    P.scaleA[n] = bernoulli_keep(pn, P.seed, 0u, (uint64_t)n) ? 1.0f / pn : 0.f;
  }
  __syncthreads();
  const int cntA = block_compact(N, [&](int n) { return P.scaleA[n] > 0.f; },
                                 [&](int n, int pos) { P.idxA[pos] = n; if (P.kept_out != nullptr) P.kept_out[pos] = n; },
                                 &sc);
  block_compact(N, [&](int n) { return !(P.scaleA[n] > 0.f); }, [&](int n, int pos) { P.dropA[pos] = n; }, &sc);
  if (tid == 0) {
    P.counts[0] = cntA;
    if (P.kept_cnt_out != nullptr) *P.kept_cnt_out = cntA;
  }
}

// ------------------------------------------------------------------------------ SampleW
__device__ __forceinline__ bool row_kept(int sample_w, float q, uint32_t u) {
  return sample_w ? (q > 0.f && u < (uint32_t)floorf(q * 16777216.0f)) : true;
}

struct SampleWParams {
  const float* wc; const uint32_t* uc;     // compact scores and uniforms of the rows of kept data
  const float* q_in;
  const int32_t* idxA;
  int32_t* counts; int32_t* chunk_off; float* fix;
  double* acc; int32_t* status;
  int T;
  float nu;
  int sample_w, accumulate_vw;
  int smem_rows;                            // scores that fit the kernel's shared memory
  int rows;                                 // N T: entries of wc and uc
};

// SampleW's single-CTA part (Sec. 4.2, Eq. 3) over the n = T * (#kept data) scores.  1. c with sum_r min(1, c w_r) = nu * n by
// water-filling: every round is one pass over the scores and one block-wide sum.  2. Eq. 3 at these probabilities (probe only).
// 3. The number of kept rows in every chunk of 32 rows, and the exclusive prefix sums of these counts: emit_pack_kernel then
// places every chunk's rows without looking at others.
//
// Bound by latencies, not by data.  Up to 16384 scores sit in registers, score j of a thread being entry tid + 1024 j, so that
// a warp's j-th scores are chunk warp + 32 j; they and their uniforms are read before the number of them is known, which takes
// one memory latency for all three, and the counts stay in shared memory until they are summed up.  (With the scores in shared
// memory, the uniforms read when they were needed and the counts written to memory and read back, 1200 scores took 9 us and
// now 6: 4096 rows, 768 -> 3072, 46.1 -> 44.5 us the call; 960 rows of an fp32 layer, 368 -> 80, 39.5 -> 37.)
template <int SLOTS>
__device__ __forceinline__ void sample_w_regs(const SampleWParams& P, const float (&wv)[SLOTS], const uint32_t (&uv)[SLOTS],
                                              int cntA, int n, WShared* sh, int* s_cnt) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = P.T;
  int mode = Q_GIVEN;
  float c = 0.f;
  if (P.q_in == nullptr && !water_fill_regs<SLOTS>(wv, P.nu * (float)T * (float)cntA, sh, mode, c) && tid == 0)
    atomicExch(P.status, (int32_t)VCAS_ERR_INTERNAL);
  const int nchunks = (n + 31) >> 5;
  float vw = 0.f;
#pragma unroll
  for (int j = 0; j < SLOTS; ++j) {
    const int i = tid + SAMPLER_THREADS * j, ch = warp + 32 * j;
    if (ch < nchunks) {                            // warp-uniform
      bool keep = false;
      if (i < n) {
        const int k = P.q_in != nullptr ? i / T : 0;
        const float q = q_of(mode, c, wv[j], P.q_in, P.q_in != nullptr ? P.idxA[k] * T + (i - k * T) : 0);
        keep = row_kept(P.sample_w, q, uv[j]);
        if (q > 0.f) vw += (1.0f - q) / q * wv[j] * wv[j];
      }
      const unsigned b = __ballot_sync(0xffffffffu, keep);
      if (lane == 0) s_cnt[ch] = __popc(b);
    }
  }
  __syncthreads();      // the counts are in place, the reduction buffers free again
  if (P.accumulate_vw) {      // Eq. 3 at these probabilities
    int dummy = 0;
    fast_sum(vw, dummy, sh, 0);
    if (tid == 0) P.acc[1] += (double)vw;
  }
  // exclusive prefix sums over the chunk counts (32 SLOTS of them at most): a thread per chunk
  const int mine = tid < nchunks ? s_cnt[tid] : 0;
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) sh->scan[warp] = incl;
  __syncthreads();
  const int wt = sh->scan[lane];
  const int base = incl - mine + __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0);
  const int total = __reduce_add_sync(0xffffffffu, wt);
  if (tid < nchunks) P.chunk_off[tid] = base;
  if (tid == 0) {
    P.counts[1] = total;
    P.fix[0] = c;
    P.fix[1] = (float)mode;
  }
}
// The scores of the rows that may be among the kept data's (`rows` of them in memory), and their uniforms.
template <int SLOTS>
__device__ __forceinline__ void sample_w_small(const SampleWParams& P, WShared* sh, int* s_cnt) {
  float wv[SLOTS];
  uint32_t uv[SLOTS];
#pragma unroll
  for (int j = 0; j < SLOTS; ++j) {
    const int i = threadIdx.x + SAMPLER_THREADS * j;
    wv[j] = i < P.rows ? __ldcg(P.wc + i) : 0.f;
    uv[j] = i < P.rows && P.sample_w ? __ldcg(P.uc + i) : 0u;
  }
  const int cntA = __ldcg(P.counts), n = cntA * P.T;
#pragma unroll
  for (int j = 0; j < SLOTS; ++j)
    if (threadIdx.x + SAMPLER_THREADS * j >= n) wv[j] = 0.f;
  sample_w_regs<SLOTS>(P, wv, uv, cntA, n, sh, s_cnt);
}

template <int SLOTS>
__global__ void __launch_bounds__(SAMPLER_THREADS) sample_w_small_kernel(SampleWParams P) {
  __shared__ WShared sh;
  __shared__ int s_cnt[32 * SLOTS];
  pdl_wait();      // the scores come from the kernel before this one
  pdl_trigger();   // not before the wait: the emitting kernel reads them ahead
  sample_w_small<SLOTS>(P, &sh, s_cnt);
}

// The same for more scores: in shared memory, or in global memory beyond smem_rows (same code, slower loads).
__global__ void __launch_bounds__(SAMPLER_THREADS) sample_w_kernel(SampleWParams P) {
  extern __shared__ __align__(16) float s_w[];
  __shared__ WShared sh;
  pdl_wait();      // the scores come from the kernel before this one
  pdl_trigger();   // not before the wait: the emitting kernel reads them ahead
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cntA = P.counts[0];
  const int T = P.T;
  const int n = cntA * T;
  const bool in_smem = n <= P.smem_rows;
  if (in_smem) {
    const int n4 = n >> 2;
    for (int i = tid; i < n4; i += SAMPLER_THREADS)
      reinterpret_cast<float4*>(s_w)[i] = reinterpret_cast<const float4*>(P.wc)[i];
    for (int i = (n4 << 2) + tid; i < n; i += SAMPLER_THREADS) s_w[i] = P.wc[i];
    __syncthreads();
  }
  const float* w = in_smem ? s_w : P.wc;

  int mode = Q_GIVEN;
  float c = 0.f;
  if (P.q_in == nullptr) {
    if (!water_fill(w, n, P.nu * (float)T * (float)cntA, &sh, mode, c) && tid == 0)
      atomicExch(P.status, (int32_t)VCAS_ERR_INTERNAL);
  }
  __syncthreads();      // the reduction buffers are free again

  if (P.accumulate_vw) {      // Eq. 3 at these probabilities
    float vw = 0.f;
    int dummy = 0;
    for (int i = tid; i < n; i += SAMPLER_THREADS) {
      const int k = i / T;
      const float x = w[i];
      const float q = q_of(mode, c, x, P.q_in, P.q_in != nullptr ? P.idxA[k] * T + (i - k * T) : 0);
      if (q > 0.f) vw += (1.0f - q) / q * x * x;
    }
    fast_sum(vw, dummy, &sh, 0);
    if (tid == 0) P.acc[1] += (double)vw;
    __syncthreads();
  }

  // kept rows per chunk of 32 compact rows: chunk_off[ch] = count for now.  A warp takes four chunks at a time
  // and issues their loads together (one memory latency per four chunks instead of one per chunk).
  const int nchunks = (n + 31) >> 5;
  for (int ch0 = warp; ch0 < nchunks; ch0 += 4 * (SAMPLER_THREADS / 32)) {
    float wv[4];
    uint32_t uv[4];
#pragma unroll
    for (int k4 = 0; k4 < 4; ++k4) {
      const int i = ((ch0 + k4 * (SAMPLER_THREADS / 32)) << 5) + lane;
      wv[k4] = i < n ? w[i] : 0.f;
      uv[k4] = (i < n && P.sample_w) ? __ldg(P.uc + i) : 0u;
    }
#pragma unroll
    for (int k4 = 0; k4 < 4; ++k4) {
      const int ch = ch0 + k4 * (SAMPLER_THREADS / 32);
      if (ch >= nchunks) break;                    // warp-uniform
      const int i = (ch << 5) + lane;
      bool keep = false;
      if (i < n) {
        const int k = i / T;
        const float q = q_of(mode, c, wv[k4], P.q_in, P.q_in != nullptr ? P.idxA[k] * T + (i - k * T) : 0);
        keep = row_kept(P.sample_w, q, uv[k4]);
      }
      const unsigned b = __ballot_sync(0xffffffffu, keep);
      if (lane == 0) P.chunk_off[ch] = __popc(b);
    }
  }
  __syncthreads();
  // exclusive prefix sums over the chunk counts: every thread owns a contiguous segment
  const int seg = (nchunks + SAMPLER_THREADS - 1) / SAMPLER_THREADS;
  const int lo = tid * seg, hi = min(nchunks, lo + seg);
  int mine = 0;
  for (int ch = lo; ch < hi; ++ch) mine += P.chunk_off[ch];
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) sh.scan[warp] = incl;
  __syncthreads();
  const int wt = sh.scan[lane];
  int base = incl - mine + __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0);
  const int total = __reduce_add_sync(0xffffffffu, wt);
  for (int ch = lo; ch < hi; ++ch) {
    const int cnt = P.chunk_off[ch];
    P.chunk_off[ch] = base;
    base += cnt;
  }
  if (tid == 0) {
    P.counts[1] = total;
    P.fix[0] = c;
    P.fix[1] = (float)mode;
  }
}

struct EmitParams {
  const float* wc; const uint32_t* uc;
  const float* q_in;
  const float* scaleA;
  const int32_t* idxA; const int32_t* dropA;
  const int32_t* counts; const int32_t* chunk_off; const float* fix;
  float* w; float* q; float* scaleW; int32_t* idxW;
  const void* dY; const void* X;                         // operands to pack
  __nv_bfloat16* packG; __nv_bfloat16* packX;            // compact operands
  size_t g_stride, x_stride;                             // elements between the parts of a cut operand
  int N, T, d_in, d_out;
  int ahead;                                             // CTAs that read their first chunk ahead
  int sample_w;
  int parts;                                             // CTAs that share the packing of one chunk's rows
};

// Row k of packG = scaleW[k] * dY[idxW[k]] (G_tilde of Sec. 4.2, rounded to bf16), row k of packX = X[idxW[k]].
__device__ __forceinline__ uint4 scale8(const uint4& v, float sc) {
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
  uint32_t o[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const __nv_bfloat162 t = __floats2bfloat162_rn(sc * __uint_as_float(u[e] << 16), sc * __uint_as_float(u[e] & 0xffff0000u));
    o[e] = *reinterpret_cast<const uint32_t*>(&t);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}
// What emit_rows_kernel hands out of the sampling record (see vcas_score); null pointers: not asked for.
struct RecordOut {
  float* g; float* p; float* w; float* q;
  int32_t* idxA; int32_t* cntA; int32_t* idxW; int32_t* cntW;
};
// A compact row of a chunk of 32, one per lane, as the kernels before SampleW left it.  The first chunk of a CTA is read ahead (see
// pdl_wait), before the wait for SampleW, which started when they had ended and then let this grid start (whole calls: 192 rows,
// 128 -> 192, 22.6 -> 21.5 us on the GPU; 256 rows, 256 -> 256, 21.3 -> 20.5; 8192 rows, 256 -> 1024, 40.9 -> 40.2, of which the
// loads past L1 took back 0.4).  Of a packing grid only the CTAs that may be there by then do so, three an SM; the others read
// after the wait, and find in L1 what the chunk's other CTAs have read (4096 rows, 768 -> 3072: with every CTA past L1 44.6 us, so
// 43.9; 16384, 1024 -> 1024: 71.8 and 70.1).
struct ChunkIn { bool in; int r; float w, sa; uint32_t u; };
template <bool AHEAD>
__device__ __forceinline__ ChunkIn chunk_in(const EmitParams& P, int ch, int lane, int n) {
  auto read = [](const auto* p) { return AHEAD ? __ldcg(p) : *p; };
  ChunkIn o = {};
  const int i = (ch << 5) + lane;
  o.in = i < n;
  if (o.in) {
    const int k = i / P.T;
    const int nd = read(P.idxA + k);
    o.r = nd * P.T + (i - k * P.T);
    o.w = read(P.wc + i);
    o.u = P.sample_w ? read(P.uc + i) : 0u;
    o.sa = read(P.scaleA + nd);
  }
  return o;
}
// Of a kept row: its place j among the chunk's and pos among all, its factor.  The number of them in every lane.
struct ChunkRow { bool keep; int j, pos, count; float q, sc; };
__device__ __forceinline__ ChunkRow chunk_row(const EmitParams& P, const ChunkIn& x, int ch, int lane, int mode, float c) {
  ChunkRow o = {};
  if (x.in) {
    o.q = q_of(mode, c, x.w, P.q_in, x.r);
    o.keep = row_kept(P.sample_w, o.q, x.u);
  }
  const unsigned b = __ballot_sync(0xffffffffu, o.keep);
  o.count = __popc(b);
  o.j = __popc(b & ((1u << lane) - 1u));
  if (o.keep) {
    o.pos = P.chunk_off[ch] + o.j;
    o.sc = P.sample_w ? x.sa / o.q : x.sa;
  }
  return o;
}
constexpr int EMIT_THREADS = 256;
constexpr int EMIT_AHEAD = 3;      // CTAs per SM that fit in every instance (80 registers)
// Without operands to pack: a warp per chunk, and the record into the caller's arrays.  Latency-bound; with an emitting
// launch of a CTA per chunk and a copying one, a scoring call of 16384 rows of 4096 and 1024 columns took 126.4 us, now 121.9.
__global__ void __launch_bounds__(EMIT_THREADS) emit_rows_kernel(EmitParams P, const float* g, const float* p, RecordOut O) {
  const int tid = blockIdx.x * EMIT_THREADS + threadIdx.x, threads = gridDim.x * EMIT_THREADS, lane = threadIdx.x & 31;
  const int cntA = __ldcg(P.counts), T = P.T, n = cntA * T;
  ChunkIn x = chunk_in<true>(P, tid >> 5, lane, n);
  pdl_wait();      // c and the chunk offsets come from the kernel before this one
  pdl_trigger();
  const int cntW = __ldcg(P.counts + 1);
  const float c = P.fix[0];
  const int mode = (int)P.fix[1];
  for (int ch = tid >> 5; ch < (n + 31) >> 5; ch += threads >> 5) {
    if (ch != tid >> 5) x = chunk_in<false>(P, ch, lane, n);
    const ChunkRow o = chunk_row(P, x, ch, lane, mode, c);
    if (x.in) {
      P.w[x.r] = x.w;
      P.q[x.r] = o.q;
      if (O.w != nullptr) O.w[x.r] = x.w;
      if (O.q != nullptr) O.q[x.r] = o.q;
    }
    if (o.keep) {
      P.idxW[o.pos] = x.r;
      P.scaleW[o.pos] = o.sc;
      if (O.idxW != nullptr) O.idxW[o.pos] = x.r;
    }
  }
  // rows of dropped data
  for (int i = tid; i < (P.N - cntA) * T; i += threads) {
    const int k = i / T;
    const int r = P.dropA[k] * T + (i - k * T);
    P.w[r] = 0.f;
    P.q[r] = 0.f;
    if (O.w != nullptr) O.w[r] = 0.f;
    if (O.q != nullptr) O.q[r] = 0.f;
  }
  for (int i = tid; i < P.N; i += threads) {
    if (O.g != nullptr) O.g[i] = g[i];
    if (O.p != nullptr) O.p[i] = p[i];
    if (O.idxA != nullptr && i < cntA) O.idxA[i] = P.idxA[i];
  }
  if (tid == 0) {
    if (O.cntA != nullptr) *O.cntA = cntA;
    if (O.cntW != nullptr) *O.cntW = cntW;
  }
}

// One CTA per (chunk of 32 compact rows, part) (grid-strided): the chunk's kept rows go to positions
// chunk_off[ch]... of the ascending kept-row list with their rescale factors 1/(p_n q_r); q and w are written by
// global row (by part 0); the operands of the chunk's kept rows j with j % parts == part are packed for the dW
// product.  The rows of dropped data get w = q = 0, and the compact operands are padded with zero rows to a
// multiple of 64 (the product's last k-block then adds nothing).
// CUT: the operands for the products of gemm_split.cu: the rescaled rows of dY are kept to fp32 precision in three bf16
// parts, and the rows of an fp32 X likewise (a bf16 X is its own single part).
template <typename E, bool CUT>
__global__ void __launch_bounds__(EMIT_THREADS) emit_pack_kernel(EmitParams P) {
  __shared__ int s_r[32], s_pos[32], s_cnt;
  __shared__ float s_sc[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, parts = P.parts;
  const bool ahead = (int)blockIdx.x < P.ahead;
  const int T = P.T;
  int cntA = 0;
  ChunkIn x = {};
  if (ahead) {
    cntA = __ldcg(P.counts);
    if (warp == 0) x = chunk_in<true>(P, (int)blockIdx.x / parts, lane, cntA * T);
  }
  pdl_wait();      // c and the chunk offsets come from the kernel before this one
  pdl_trigger();   // the dW product kernel may set itself up; it waits for this grid before loading
  if (!ahead) cntA = P.counts[0];
  const int n = cntA * T;
  const int cntW = __ldcg(P.counts + 1);
  const float c = P.fix[0];
  const int mode = (int)P.fix[1];
  const int nchunks = (n + 31) >> 5;
  for (int u = blockIdx.x; u < nchunks * parts; u += gridDim.x) {
    const int ch = u / parts, part = u - ch * parts;
    if (warp == 0) {
      if (!ahead || u != (int)blockIdx.x) x = chunk_in<false>(P, ch, lane, n);
      const ChunkRow o = chunk_row(P, x, ch, lane, mode, c);
      if (part == 0 && x.in) { P.w[x.r] = x.w; P.q[x.r] = o.q; }
      if (o.keep) {
        if (part == 0) { P.idxW[o.pos] = x.r; P.scaleW[o.pos] = o.sc; }
        s_r[o.j] = x.r; s_pos[o.j] = o.pos; s_sc[o.j] = o.sc;
      }
      if (lane == 0) s_cnt = o.count;
    }
    __syncthreads();
    // This part's rows j = part, part + parts, ...  A row's 16-byte pieces (first those of dY, then those of X)
    // are cut into segments of 128; a warp takes (row, segment) items in turn and moves a segment with four
    // independent loads per lane in flight.  One integer division per 2 KB moved, none per piece.
    const int m = s_cnt;
    const int mp = m > part ? (m - part + parts - 1) / parts : 0;
    const int vo = P.d_out / 8, vt = vo + P.d_in / 8;
    const int nseg = (vt + 127) >> 7;
    for (int item = warp; item < mp * nseg; item += EMIT_THREADS / 32) {
      const int jj = item / nseg, seg = item - jj * nseg;
      const int j = part + jj * parts;
      const size_t r = (size_t)s_r[j], pos = (size_t)s_pos[j];
      const float sc = s_sc[j];
      const E* srcG = reinterpret_cast<const E*>(P.dY) + r * P.d_out;
      const E* srcX = reinterpret_cast<const E*>(P.X) + r * P.d_in - (size_t)P.d_out;
      __nv_bfloat16* dstG = P.packG + pos * P.d_out;
      __nv_bfloat16* dstX = P.packX + pos * P.d_in - (size_t)P.d_out;
      const int p0 = (seg << 7) + lane;
      Vec8<E> v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int piece = p0 + 32 * q;
        if (piece < vt) v[q].load((piece < vo ? srcG : srcX) + piece * 8);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int piece = p0 + 32 * q;
        if (piece >= vt) break;
        const bool g = piece < vo;
        __nv_bfloat16* dst = (g ? dstG : dstX) + piece * 8;
        if constexpr (CUT) {
          if (sizeof(E) == 4 || g) {
            float f[8];
            v[q].get(f);
            if (g) {
#pragma unroll
              for (int e = 0; e < 8; ++e) f[e] *= sc;
            }
            store_parts3<sizeof(E) == 4>(f, dst, g ? P.g_stride : P.x_stride);      // a bf16 X is a single part
            continue;
          }
        }
        if constexpr (sizeof(E) == 2)
          *reinterpret_cast<uint4*>(dst) = g ? scale8(v[q].v, sc) : v[q].v;
      }
    }
    __syncthreads();
  }
  // rows of dropped data
  const int ndrop_rows = (P.N - cntA) * T;
  for (int i = blockIdx.x * EMIT_THREADS + tid; i < ndrop_rows; i += gridDim.x * EMIT_THREADS) {
    const int k = i / T;
    const int r = P.dropA[k] * T + (i - k * T);
    P.w[r] = 0.f;
    P.q[r] = 0.f;
  }
  // zero rows up to the next multiple of 64
  const int padded = (cntW + 63) / 64 * 64;
  const uint4 z = make_uint4(0u, 0u, 0u, 0u);
  for (int k = cntW + (int)blockIdx.x; k < padded; k += gridDim.x) {
#pragma unroll
    for (int part = 0; part < (CUT ? 3 : 1); ++part)
      for (int i = tid; i < P.d_out / 8; i += EMIT_THREADS)
        reinterpret_cast<uint4*>(P.packG + part * P.g_stride + (size_t)k * P.d_out)[i] = z;
#pragma unroll
    for (int part = 0; part < (CUT && sizeof(E) == 4 ? 3 : 1); ++part)
      for (int i = tid; i < P.d_in / 8; i += EMIT_THREADS)
        reinterpret_cast<uint4*>(P.packX + part * P.x_stride + (size_t)k * P.d_in)[i] = z;
  }
}

// The sampling record (see vcas_score) into the caller's arrays.  One launch: eight copies of a few KB to 64 KB took 35 us of
// a 150 us scoring call one after the other.
struct CopyParams {
  const float* g; const float* p; const float* w; const float* q;
  const int32_t* idxA; const int32_t* idxW; const int32_t* counts;
  float* og; float* op; float* ow; float* oq;
  int32_t* oidxA; int32_t* ocntA; int32_t* oidxW; int32_t* ocntW;
  int N, R;
};
__global__ void __launch_bounds__(256) copy_out_kernel(CopyParams P) {
  for (int i = blockIdx.x * 256 + threadIdx.x; i < P.R; i += gridDim.x * 256) {
    if (P.ow != nullptr) P.ow[i] = P.w[i];
    if (P.oq != nullptr) P.oq[i] = P.q[i];
    if (P.oidxW != nullptr) P.oidxW[i] = P.idxW[i];
    if (i < P.N) {
      if (P.og != nullptr) P.og[i] = P.g[i];
      if (P.op != nullptr) P.op[i] = P.p[i];
      if (P.oidxA != nullptr) P.oidxA[i] = P.idxA[i];
    }
    if (i == 0) {
      if (P.ocntA != nullptr) *P.ocntA = P.counts[0];
      if (P.ocntW != nullptr) *P.ocntW = P.counts[1];
    }
  }
}

__global__ void __launch_bounds__(SAMPLER_THREADS)
mask_kernel(const float* __restrict__ p, int n, uint64_t seed, int sampler, uint8_t* keep, int32_t* idx,
            int32_t* cnt) {
  __shared__ Scratch sc;
  const int c = block_compact(n,
      [&](int i) {
        const bool k = bernoulli_keep(p[i], seed, (uint32_t)sampler, (uint64_t)i);
        if (keep != nullptr) keep[i] = k ? 1 : 0;
        return k;
      },
      [&](int i, int pos) { if (idx != nullptr) idx[pos] = i; }, &sc);
  if (threadIdx.x == 0 && cnt != nullptr) *cnt = c;
}

}  // namespace

namespace {
SampleAParams sample_a_params(const Handle* h, const SamplerArgs& a) {
  const Workspace& ws = h->ws;
  const vcas_layer_desc& d = h->desc;
  SampleAParams P;
  P.a = a.a_in != nullptr ? a.a_in : ws.a;
  P.a_parts = a.a_in != nullptr ? a.a_parts : 1;
  P.alive = a.alive; P.alive_cnt = a.alive_cnt;
  P.N = d.N; P.T = d.T; P.rho = a.rho; P.p_in = a.p_in; P.seed = a.seed;
  P.g = ws.g; P.p = ws.p; P.scaleA = ws.scaleA; P.idxA = ws.idxA; P.dropA = ws.dropA; P.counts = ws.counts;
  P.kept_out = a.kept_out; P.kept_cnt_out = a.kept_cnt_out;
  P.status = ws.status;
  P.gk = ws.gk; P.ticket = ws.counts + 5;
  return P;
}

template <typename T>
cudaError_t run_norms_sample_a(Handle* h, const void* dY, const SampleAParams& P, cudaStream_t st) {
  const vcas_layer_desc& d = h->desc;
  const dim3 grid((unsigned)((d.N * d.T + SAMPLE_A_THREADS / 32 - 1) / (SAMPLE_A_THREADS / 32))), threads(SAMPLE_A_THREADS);
  const T* y = reinterpret_cast<const T*>(dY);
  norms_sample_a_kernel<T><<<grid, threads, 0, st>>>(y, d.d_out, h->ws.a, P);
  h->launches += 1;
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_norms_sample_a(Handle* h, const void* dY, const SamplerArgs& a, cudaStream_t st) {
  const vcas_layer_desc& d = h->desc;
  if (a.a_in != nullptr || (long)d.N * d.T > FUSED_MAX_ROWS || d.N > FUSED_MAX_N || d.T > SAMPLE_A_WARP_LEN) {
    const cudaError_t e = launch_rownorm_dy(h, dY, a, st);
    return e != cudaSuccess ? e : launch_sample_a(h, a, a.a_in == nullptr, st);
  }
  const SampleAParams P = sample_a_params(h, a);
  return d.dtype == VCAS_DTYPE_BF16 ? run_norms_sample_a<__nv_bfloat16>(h, dY, P, st) : run_norms_sample_a<float>(h, dY, P, st);
}

cudaError_t launch_sample_a(Handle* h, const SamplerArgs& a, bool programmatic, cudaStream_t st) {
  const vcas_layer_desc& d = h->desc;
  const SampleAParams P = sample_a_params(h, a);
  const int per_cta = d.T * P.a_parts <= SAMPLE_A_WARP_LEN ? SAMPLE_A_THREADS / 32 : 1;
  int ctas = (d.N + per_cta - 1) / per_cta;
  const int cap = h->num_sms > 0 ? h->num_sms : 148;
  if (ctas > cap) ctas = cap;
  const dim3 grid((unsigned)ctas), threads(SAMPLE_A_THREADS);
  cudaError_t e;
  if (d.N <= 32)
    e = launch_maybe_after(programmatic, sample_a_kernel<1>, grid, threads, 0, st, P);
  else if (d.N <= 64)
    e = launch_maybe_after(programmatic, sample_a_kernel<2>, grid, threads, 0, st, P);
  else if (d.N <= 128)
    e = launch_maybe_after(programmatic, sample_a_kernel<4>, grid, threads, 0, st, P);
  else if (d.N <= 256)
    e = launch_maybe_after(programmatic, sample_a_kernel<8>, grid, threads, 0, st, P);
  else if (d.N <= WARP_MAX_N)
    e = launch_maybe_after(programmatic, sample_a_kernel<32>, grid, threads, 0, st, P);
  else
    e = launch_maybe_after(programmatic, sample_a_big_kernel, dim3(1), dim3(SAMPLER_THREADS), 0, st, P);
  h->launches += 1;
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_sample_w(Handle* h, const SamplerArgs& a, cudaStream_t st) {
  static std::atomic<bool> attr_set[64];
  const Workspace& ws = h->ws;
  const vcas_layer_desc& d = h->desc;
  const long R = (long)d.N * d.T;
  SampleWParams P;
  P.wc = ws.wc; P.uc = ws.uc; P.q_in = a.q_in; P.idxA = ws.idxA;
  P.counts = ws.counts; P.chunk_off = ws.chunk_off; P.fix = ws.fix; P.acc = ws.acc; P.status = ws.status;
  P.T = d.T; P.nu = a.nu; P.sample_w = a.sample_w; P.accumulate_vw = a.accumulate_vw;
  P.smem_rows = 0;
  P.rows = (int)R;
  h->launches += 1;
  const dim3 threads(SAMPLER_THREADS);
  if (R <= 2 * SAMPLER_THREADS) return launch_after(sample_w_small_kernel<2>, dim3(1), threads, 0, st, P);
  if (R <= 4 * SAMPLER_THREADS) return launch_after(sample_w_small_kernel<4>, dim3(1), threads, 0, st, P);
  if (R <= 8 * SAMPLER_THREADS) return launch_after(sample_w_small_kernel<8>, dim3(1), threads, 0, st, P);
  if (R <= 16 * SAMPLER_THREADS) return launch_after(sample_w_small_kernel<16>, dim3(1), threads, 0, st, P);
  // shared memory for the scores: enough for every row when that fits, else the kernel reads global memory
  // whenever the kept rows exceed it
  int rows = (int)(R < SAMPLE_W_SMEM_ROWS ? R : SAMPLE_W_SMEM_ROWS);
  rows = (rows + 3) & ~3;
  const size_t smem = (size_t)rows * sizeof(float);
  if (smem > 48 * 1024) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dev].load(std::memory_order_acquire)) {
      e = cudaFuncSetAttribute(sample_w_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               SAMPLE_W_SMEM_ROWS * (int)sizeof(float));
      if (e != cudaSuccess) return e;
      attr_set[dev].store(true, std::memory_order_release);
    }
  }
  P.smem_rows = rows;
  const cudaError_t e = launch_after(sample_w_kernel, dim3(1), threads, smem, st, P);
  return e != cudaSuccess ? e : cudaGetLastError();
}

namespace {
EmitParams emit_params(const Handle* h, const SamplerArgs& a) {
  const Workspace& ws = h->ws;
  const vcas_layer_desc& d = h->desc;
  EmitParams P = {};
  P.wc = ws.wc; P.uc = ws.uc; P.q_in = a.q_in; P.scaleA = ws.scaleA; P.idxA = ws.idxA; P.dropA = ws.dropA;
  P.counts = ws.counts; P.chunk_off = ws.chunk_off; P.fix = ws.fix;
  P.w = ws.w; P.q = ws.q; P.scaleW = ws.scaleW; P.idxW = ws.idxW;
  P.N = d.N; P.T = d.T; P.d_in = d.d_in; P.d_out = d.d_out;
  P.sample_w = a.sample_w;
  return P;
}
}  // namespace

cudaError_t launch_emit_record(Handle* h, const SamplerArgs& a, float* g, float* p, float* w, float* q, int32_t* idxA,
                               int32_t* cntA, int32_t* idxW, int32_t* cntW, cudaStream_t st) {
  RecordOut O;
  O.g = g; O.p = p; O.w = w; O.q = q; O.idxA = idxA; O.cntA = cntA; O.idxW = idxW; O.cntW = cntW;
  const long rows = (long)h->desc.N * h->desc.T, cap = (long)(h->num_sms > 0 ? h->num_sms : 148) * 8;
  long blocks = (rows + EMIT_THREADS - 1) / EMIT_THREADS;
  if (blocks > cap) blocks = cap;
  const cudaError_t e = launch_after(emit_rows_kernel, dim3((unsigned)blocks), dim3(EMIT_THREADS), 0, st, emit_params(h, a),
                                     (const float*)h->ws.g, (const float*)h->ws.p, O);
  h->launches += 1;
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_emit_pack(Handle* h, const void* dY, const void* X, const SamplerArgs& a, bool pack, cudaStream_t st) {
  if (!pack) return launch_emit_record(h, a, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, st);
  const Workspace& ws = h->ws;
  const vcas_layer_desc& d = h->desc;
  EmitParams P = emit_params(h, a);
  P.dY = dY; P.X = X;
  P.g_stride = (size_t)h->R_pad * d.d_out; P.x_stride = (size_t)h->R_pad * d.d_in;
  P.packG = ws.packG; P.packX = ws.packX;
  // The number of chunks with kept rows is only known on the device.  The grid has eight CTAs per SM and the rows of a
  // chunk are shared among as many CTAs as the expected number of chunks leaves room for.
  const long R = (long)d.N * d.T;
  const long cap = (long)(h->num_sms > 0 ? h->num_sms : 148) * 8;
  long expected = (long)((double)a.rho * (double)R / 32.0) + 1;
  long parts = cap / expected;
  if (parts < 1) parts = 1;
  if (parts > 16) parts = 16;
  P.parts = (int)parts;
  long blocks = ((R + 31) / 32) * parts;
  if (blocks > cap) blocks = cap;
  P.ahead = (int)(cap / 8) * EMIT_AHEAD;
  const dim3 grid((unsigned)blocks), threads(EMIT_THREADS);
  const cudaError_t e = !h->split_path           ? launch_after(emit_pack_kernel<__nv_bfloat16, false>, grid, threads, 0, st, P)
      : d.dtype == VCAS_DTYPE_F32                ? launch_after(emit_pack_kernel<float, true>, grid, threads, 0, st, P)
                                                 : launch_after(emit_pack_kernel<__nv_bfloat16, true>, grid, threads, 0, st, P);
  h->launches += 1;
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_copy_out(Handle* h, float* g, float* p, float* w, float* q, int32_t* idxA, int32_t* cntA, int32_t* idxW,
                            int32_t* cntW, cudaStream_t st) {
  const Workspace& ws = h->ws;
  CopyParams P;
  P.g = ws.g; P.p = ws.p; P.w = ws.w; P.q = ws.q; P.idxA = ws.idxA; P.idxW = ws.idxW; P.counts = ws.counts;
  P.og = g; P.op = p; P.ow = w; P.oq = q; P.oidxA = idxA; P.ocntA = cntA; P.oidxW = idxW; P.ocntW = cntW;
  P.N = h->desc.N; P.R = h->desc.N * h->desc.T;
  int blocks = (P.R + 255) / 256;
  if (blocks > 592) blocks = 592;
  copy_out_kernel<<<(unsigned)blocks, 256, 0, st>>>(P);
  h->launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_mask_from_probs(Handle* h, const float* p, int n, uint64_t seed, int sampler,
                                   uint8_t* keep, int32_t* idx, int32_t* cnt, cudaStream_t st) {
  mask_kernel<<<1, SAMPLER_THREADS, 0, st>>>(p, n, seed, sampler, keep, idx, cnt);
  h->launches += 1;
  return cudaGetLastError();
}

}  // namespace vcas
