// The variance probe of a tensor-path layer (Alg. 1, App. D) with one product launch per group of batches.
//
// A unit of the product is a tile of the parameter gradient of one batch.  Its CTA forms G_s = dY^T X and beside it, from the
// same loads of X, the gradients of the draws, G_act,j = sum over the data kept in draw j of bf16(dY_n / p_n)^T X_n, each in an
// accumulator of its own, and adds up the squares of G_act,j - G_s: no G_act is ever written.  The rows are rescaled and
// rounded as in the sampled backward, whose gradients V_act speaks about; p_n belongs to the batch and not to the draw, so
// they are made once for all draws, and a draw is only the list of the data that it accumulates.  The accumulators are added
// up in fp32 registers every 1024 rows: tcgen05 truncates, and over 32768 rows in TMEM V_s lost 7e-5 of itself (2e-6 so).
// (G_act,j as a sum of the data's exact products weighted with 1 / p_n needs one product per batch, but its V_act was up to
// 5e-4 off: the rounding moves all values of a datum by the same 1e-4, which does not average out.)
// Measured on B200, against a chain of launches and a product per draw (probe.cu): 4096 rows, 768 -> 3072, M = 4: 709 -> 254 us;
// 16384 rows, 4096 -> 128 of 11008, M = 2: 538 -> 283 us; 640 rows, 128 -> 128, M = 2, rho = 0.8: 145 -> 39 us.
//
// Launches per group: norms of the rows of dY and X (which also gathers the sampled columns of dY), one CTA per draw for p
// and mask, one CTA per draw for Eq. 3 (beside the product, on the side stream), the rescaled rows, the product, the moments
// of G_s.
#include <atomic>

#include "rows.cuh"
#include "split.cuh"
#include "umma.cuh"
#include "water.cuh"

namespace vcas {
namespace {

constexpr int PROBE_MIN_T = 64;              // shortest data served: one step of the contraction
constexpr int PG = 4;                        // most batches a launch serves
constexpr int PROBE_THREADS = 12 * 32;       // warps 0-7 add up, 8 loads, 9 issues, 10 and 11 fill the warpgroup
constexpr int ACC_THREADS = 256;
constexpr int PBN = 128;                     // tile columns
constexpr int PD = 2;                        // draws of a round
constexpr int FLUSH = 16;                    // steps that an accumulator takes before fp32 registers add it up
constexpr int PK = 64;                       // rows of a step
constexpr int PCHUNK = 64 * PK * 2;          // 64 columns of a step
constexpr int PA_BYTES = BM / 64 * PCHUNK;   // 128 columns of dY, or of its rescaled rows
constexpr int PSTAGE = 2 * PA_BYTES + PBN / 64 * PCHUNK;
constexpr int PSTAGES = 4;
constexpr int PMASKS = 28672;                // bytes of the masks of a launch
constexpr int PSMEM = PSTAGES * PSTAGE + 1024 /*alignment slack*/ + 256 /*barriers*/ + PMASKS;

// What a group of batches leaves for its product: a block per batch.
struct ProbeGroup {
  const __nv_bfloat16* dY[PG]; const __nv_bfloat16* X[PG];
  uint8_t* block[PG];
  size_t b_at, p_at, keep_at, scaled_at;
  __nv_bfloat16* sub;              // [batch][R][k] sampled columns of dY
  __device__ __forceinline__ float* a(int g) const { return reinterpret_cast<float*>(block[g]); }             // [R] ||dY_r||^2
  __device__ __forceinline__ float* b(int g) const { return reinterpret_cast<float*>(block[g] + b_at); }      // [R] ||X_r||^2
  __device__ __forceinline__ float* p(int g) const { return reinterpret_cast<float*>(block[g] + p_at); }      // [N]
  __device__ __forceinline__ uint8_t* keep(int g) const { return block[g] + keep_at; }                        // [M][N]
  __host__ __device__ __forceinline__ __nv_bfloat16* scaled(int g) const {                                    // [R][columns]
    return reinterpret_cast<__nv_bfloat16*>(block[g] + scaled_at);
  }
};

// ------------------------------------------------------------------------------------- row norms
// Sum of squares of a row by one warp, and its k elements at the ascending columns `cols` copied to dst.  The columns are
// picked after every 4 KB, from L1: with 48 rows in flight an SM has a megabyte of rows open, so that a pass over the row when
// it ends finds its start neither in L1 nor surely in L2 (16384 rows of 11008 twice, 128 columns, with the rows of X:
// 198 -> 155 us, 6.4 TB/s, which also took the operands' addresses out of local memory).
__device__ __forceinline__ float row_partial_pick(const __nv_bfloat16* __restrict__ row, int d, int lane,
                                                  const int32_t* __restrict__ cols, int k, __nv_bfloat16* __restrict__ dst) {
  const uint4* v = reinterpret_cast<const uint4*>(row);
  const int nv = d / 8;                              // d is a multiple of 64
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int v0 = 0, q = 0; v0 < nv; v0 += 256) {
    uint4 x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int i = v0 + lane + 32 * e;
      x[e] = i < nv ? __ldg(v + i) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e % 4] += sq8(x[e]);
    const int end = min((v0 + 256) * 8, d);
    for (;;) {
      const int col = q + lane < k ? __ldg(cols + q + lane) : INT32_MAX;
      const bool in = col < end;
      if (in) reinterpret_cast<unsigned short*>(dst)[q + lane] = __ldg(reinterpret_cast<const unsigned short*>(row) + col);
      const int n = __popc(__ballot_sync(0xffffffffu, in));
      q += n;
      if (n < 32) break;
    }
  }
  return (acc[0] + acc[1]) + (acc[2] + acc[3]);
}

// One warp per row, HBM-bound: of every batch first the R rows of dY, then those of X.  PICK: the k sampled columns of every
// row of dY are copied out on the way.
template <bool PICK>
__global__ void __launch_bounds__(256) probe_norms_kernel(const __grid_constant__ ProbeGroup G, int batches, int R, int d_out,
                                                          int d_in, const int32_t* __restrict__ cols, int k) {
  pdl_trigger();
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  for (int i = blockIdx.x * wpb + (threadIdx.x >> 5); i < 2 * R * batches; i += gridDim.x * wpb) {
    const int g = i / (2 * R), c = i - g * 2 * R;
    const bool y = c < R;
    const int r = y ? c : c - R, d = y ? d_out : d_in;
    const __nv_bfloat16* row = (y ? G.dY[g] : G.X[g]) + (size_t)r * d;
    const float s = warp_sum(PICK && y ? row_partial_pick(row, d, lane, cols, k, G.sub + ((size_t)g * R + r) * k)
                                       : row_partial<__nv_bfloat16>(row, d, lane));
    if (lane == 0) (y ? G.a(g) : G.b(g))[r] = s;
  }
}

// ------------------------------------------------------------------------------------ the draws
struct DrawParams {
  double* sparsity;                // [2][batch of the probe] p_lo, p_hi
  double* vw;                      // [batch of the probe][M] Eq. 3
  int32_t* status;
  int N, T, M, first_batch;
  float rho, nu;
  double s_lo, s_hi;
  uint64_t seed;
};

// CTA (j, batch), j < M: SampleA of draw j (Sec. 4.1), as in the sampled backward.  CTA (M, batch): Eq. 4's sparsity.
constexpr int DRAW_THREADS = 512;
template <int SLOTS>
__global__ void __launch_bounds__(DRAW_THREADS) probe_draw_kernel(const __grid_constant__ ProbeGroup G, DrawParams P) {
  __shared__ float s_g[32 * SLOTS], s_sorted[32 * SLOTS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x, g = blockIdx.y;
  for (int n = threadIdx.x; n < 32 * SLOTS; n += DRAW_THREADS) s_g[n] = 0.f;
  pdl_wait();
  pdl_trigger();
  __syncthreads();
  for (int n = warp; n < P.N; n += DRAW_THREADS / 32) {
    const float s = datum_sqnorm_warp(G.a(g) + (size_t)n * P.T, P.T, lane);
    if (lane == 0) s_g[n] = sqrtf(s);
  }
  __syncthreads();
  if (j < P.M) {
    if (warp != 0) return;
    float v[SLOTS];
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) v[i] = s_g[lane + 32 * i];
    capped_prop_warp<SLOTS>(v, (float)P.N * P.rho);
    const uint64_t seed = P.seed + (uint64_t)((P.first_batch + g) * P.M + j + 1) * 0x9E3779B97F4A7C15ull;
    float* p = G.p(g);
    uint8_t* keep = G.keep(g) + (size_t)j * P.N;
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
      const int n = lane + 32 * i;
      if (n < P.N) {
        if (j == 0) p[n] = v[i];                     // the same in every draw
        keep[n] = bernoulli_keep(v[i], seed, 0u, (uint64_t)n) ? 1 : 0;
      }
    }
    return;
  }
  // rank of g[i] in descending order (ties broken by index)
  for (int i = threadIdx.x; i < P.N; i += DRAW_THREADS) {
    const float x = s_g[i];
    int rank = 0;
    for (int i2 = 0; i2 < P.N; ++i2) {
      const float y = s_g[i2];
      rank += (y > x) || (y == x && i2 < i);
    }
    s_sorted[rank] = x;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double total = 0.0;
    for (int i = 0; i < P.N; ++i) total += (double)s_sorted[i];
    const double ss[2] = {P.s_lo, P.s_hi};
    for (int k = 0; k < 2; ++k) {
      const double target = ss[k] * total;
      double cum = (double)s_sorted[0];
      int n = 1;
      while (cum < target && n < P.N) { cum += (double)s_sorted[n]; ++n; }
      P.sparsity[k * P.M + P.first_batch + g] = (double)n / (double)P.N;
    }
  }
}

// Eq. 3 of draw (j, batch) at the probabilities q = min(1, c w) of ratio nu: leverage scores of the rows of its kept data (0
// on the others), water-filling, sum of (1 - q) / q w^2.
__global__ void __launch_bounds__(SAMPLER_THREADS) probe_vw_kernel(const __grid_constant__ ProbeGroup G, DrawParams P) {
  extern __shared__ __align__(16) float s_w[];
  __shared__ WShared sh;
  const int tid = threadIdx.x, j = blockIdx.x, g = blockIdx.y, n = P.N * P.T;
  const float* a = G.a(g);
  const float* b = G.b(g);
  const float* p = G.p(g);
  const uint8_t* keep = G.keep(g) + (size_t)j * P.N;
  for (int i = tid; i < n; i += SAMPLER_THREADS) {
    const int d = i / P.T;
    s_w[i] = keep[d] != 0 ? sqrtf(a[i]) * sqrtf(b[i]) / p[d] : 0.f;
  }
  float dummy = 0.f;
  int kept = 0;
  for (int i = tid; i < P.N; i += SAMPLER_THREADS) kept += keep[i];
  fast_sum(dummy, kept, &sh, 1);
  __syncthreads();
  int mode;
  float c;
  if (!water_fill(s_w, n, P.nu * (float)P.T * (float)kept, &sh, mode, c) && tid == 0)
    atomicExch(P.status, (int32_t)VCAS_ERR_INTERNAL);
  __syncthreads();
  float vw = 0.f;
  for (int i = tid; i < n; i += SAMPLER_THREADS) {
    const float x = s_w[i];
    const float q = q_of(mode, c, x, nullptr, 0);
    if (q > 0.f) vw += (1.0f - q) / q * x * x;
  }
  fast_sum(vw, kept, &sh, 0);
  if (tid == 0) P.vw[(P.first_batch + g) * P.M + j] = (double)vw;
}

// --------------------------------------------------------------------------------- rescaled rows
// bf16(dY_r / p_n) for the rows of the data that any draw kept, `cols` columns of each (the sampled ones if SUB); blockIdx.y is
// the batch.  HBM / L2 bound: 16-byte pieces over the whole matrix, four per thread in flight.
constexpr int SCALE_THREADS = 256;
template <bool SUB>
__global__ void __launch_bounds__(SCALE_THREADS) probe_scale_kernel(const __grid_constant__ ProbeGroup G, int N, int T, int M, int cols) {
  extern __shared__ float s_scale[];           // [N] 1/p of the kept data, 0 for the others
  pdl_wait();
  pdl_trigger();
  const int g = blockIdx.y;
  for (int n = threadIdx.x; n < N; n += SCALE_THREADS) {
    const uint8_t* keep = G.keep(g) + n;
    int any = 0;
    for (int j = 0; j < M; ++j) any |= keep[(size_t)j * N];
    s_scale[n] = any != 0 ? 1.0f / G.p(g)[n] : 0.f;
  }
  __syncthreads();
  const int per = T * (cols / 8), total = N * per;        // pieces of a datum, of the batch
  const __nv_bfloat16* src = SUB ? G.sub + (size_t)g * N * T * cols : G.dY[g];
  __nv_bfloat16* dst = G.scaled(g);
  for (int i0 = blockIdx.x * 4 * SCALE_THREADS + threadIdx.x; i0 < total; i0 += gridDim.x * 4 * SCALE_THREADS) {
    Vec8<__nv_bfloat16> v[4];
    float sc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + q * SCALE_THREADS;
      sc[q] = i < total ? s_scale[i / per] : 0.f;
      if (sc[q] == 0.f) continue;
      if (SUB) v[q].v = __ldcg(reinterpret_cast<const uint4*>(src) + i);      // written by a kernel of this call
      else v[q].load(src + (size_t)i * 8);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (sc[q] == 0.f) continue;
      float f[8];
      v[q].get(f);
#pragma unroll
      for (int e = 0; e < 8; ++e) f[e] *= sc[q];
      store8(dst + (size_t)(i0 + q * SCALE_THREADS) * 8, f);
    }
  }
}

// ----------------------------------------------------------------------------------- the product
struct ProbeMaps { CUtensorMap a[PG], e[PG], b[PG]; };      // per batch: dY (or its sampled columns), its rescaled rows, X
struct ProbeParams {
  const uint8_t* keep[PG];         // [M][N]
  float* gs; size_t gs_stride;     // G_s of every batch, d_out x d_in, see gs_at
  double* pact;                    // [batch][tile][warp or part of it]: sum of squares of the differences
  float* partial;                  // [unit][1 + M][128 x 128] when the contraction is cut into slices
  int N, T, d_in, d_out, kT, S, ntiles, tiles, units;    // kT: steps of a datum
  int batches, M;
  int32_t* status;
  unsigned long long wait_limit_ns;
  int stall_once;
};
// Unit u: a slice of the contractions of a tile of a batch.
struct ProbeUnit { int g, tile, slice; };
__device__ __forceinline__ ProbeUnit probe_unit(const ProbeParams& P, int u) {
  ProbeUnit w;
  const int t = u / P.S;
  w.slice = u - t * P.S;
  w.g = t / P.tiles;
  w.tile = t - w.g * P.tiles;
  return w;
}
// A unit works in rounds, two draws at a time, the first beside G_s: the sums that the registers hold.
__device__ __forceinline__ int round_draws(int r, int M) { return min(PD, M - PD * r); }
__host__ __device__ __forceinline__ int rounds_of(int M) { return (M + PD - 1) / PD; }
// The steps of a slice of a round: `left` steps from step kb of datum n on.  Round 0 runs over all data, the others over those
// that any of their draws kept.  mask: [N rounded up to 4] the draws of the round that kept the datum, a bit each; kept: the
// number of data with a mask.
struct RoundSteps { int n, kb, left; };
__device__ __forceinline__ RoundSteps round_steps(const uint8_t* mask, int kept, int N, int kT, int r, int S, int slice) {
  RoundSteps s;
  const int steps = (r == 0 ? N : kept) * kT, per = (steps + S - 1) / S, c0 = min(steps, slice * per);
  s.left = min(steps, c0 + per) - c0;
  int k = c0 / kT;
  s.kb = c0 - k * kT;
  s.n = k;
  if (r == 0 || s.left <= 0) return s;
  s.n = 0;
  for (;; s.n += 4) {                          // the k-th datum with a mask
    const int c = __popc(__vcmpne4(*reinterpret_cast<const uint32_t*>(mask + s.n), 0u)) / 8;
    if (k < c) break;
    k -= c;
  }
  for (;; ++s.n)
    if (mask[s.n] != 0 && k-- == 0) return s;
}

// Welford's update of one element of batch `i` of M: returns its final squared deviation in the last batch, else 0.
__device__ __forceinline__ float welford(float x, int i, int M, float& mean, float& m2) {
  if (i == 0) { mean = x; m2 = 0.f; return 0.f; }
  const float d = x - mean;
  mean = fmaf(d, 1.0f / (float)(i + 1), mean);
  m2 = fmaf(d, x - mean, m2);
  return i == M - 1 ? m2 : 0.f;
}
// Where a tile's columns 4 q .. 4 q + 3 of `row` are in a scratch tile of `rows` rows.  The threads of a warp have consecutive
// rows, so they take 512 consecutive bytes; in rows of columns an instruction would meet 32 cache lines.
__device__ __forceinline__ size_t scratch_at(int q, int rows, int row) { return ((size_t)q * rows + row) * 4; }
// Where columns col .. col + 3 (col a multiple of 4) of row `row` of tile row r0 are in a kept G_s, `rows` = gs_rows(r0).
__device__ __forceinline__ int gs_rows(const ProbeParams& P, int r0) { return min(BM, P.d_out - r0); }
__device__ __forceinline__ size_t gs_at(const ProbeParams& P, int r0, int rows, int row, int col) {
  return (size_t)r0 * P.d_in + scratch_at(col / 4, rows, row);
}
// The sums of THREADS threads, added in a fixed order by thread 0.
template <int THREADS>
__device__ __forceinline__ void block_act(double* out, double act, double* sh) {
  act = warp_sum(act);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) sh[warp] = act;
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < THREADS / 32; ++w) t += sh[w];
    *out = t;
  }
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// Persistent CTAs; a unit is a tile of one batch's gradients, possibly with a slice of the contraction.  Bound by the bytes
// through shared memory (operands in, and out again once per accumulator: 16 KB and 32 KB per 64 rows), for gradients of few
// rows by X from HBM.  The loading and the issuing warp run their loops with uniform control flow, one elected lane acts, and
// what a step does is fixed per datum: with the lists of data walked by one lane a step took 0.8 us whatever it had to do.
__global__ void __launch_bounds__(PROBE_THREADS, 1)
probe_kernel(const __grid_constant__ ProbeMaps maps, const __grid_constant__ ProbeParams P) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint32_t s_begun;               // the accumulators of the round that a product has written, a bit each
  __shared__ int s_kept[PG * 32];            // [batch][round] data with a mask
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(base + PSTAGES * PSTAGE);
  uint64_t* empty = full + PSTAGES;
  uint64_t* acc_full = empty + PSTAGES;      // the accumulators of a round are complete
  uint64_t* acc_empty = acc_full + 1;        // ... have been read
  uint64_t* done = acc_empty + 1;            // see drain_products
  uint32_t* tmem_holder = (uint32_t*)(done + 1);
  volatile int* abort_flag = (int*)(tmem_holder + 1);
  uint8_t* s_mask = base + PSTAGES * PSTAGE + 256;      // [batch][round][N rounded up to 4], see round_steps
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < PSTAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(acc_full, 2);                  // the issuing lane, which has written s_begun, and its products
    mbar_init(acc_empty, ACC_THREADS / 32);
    mbar_init(done, 1);
    *abort_flag = 0;
    *reinterpret_cast<volatile unsigned long long*>(abort_flag + 5) = P.wait_limit_ns;     // read by mbar_wait
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 9) tmem_alloc(tmem_holder, 512);
  const int rounds = rounds_of(P.M), n_pad = (P.N + 3) & ~3;
  pdl_wait();
  for (int i = warp; i < P.batches * rounds; i += PROBE_THREADS / 32) {
    const int g = i / rounds, r = i - g * rounds, draws = round_draws(r, P.M);
    const uint8_t* keep = P.keep[g] + (size_t)(PD * r) * P.N;
    int kept = 0;
    for (int n = lane; n < n_pad; n += 32) {
      uint32_t m = 0;
      if (n < P.N)
        for (int j = 0; j < draws; ++j) m |= (uint32_t)keep[(size_t)j * P.N + n] << j;
      s_mask[i * n_pad + n] = (uint8_t)m;
      kept += m != 0u ? 1 : 0;
    }
    kept = __reduce_add_sync(0xffffffffu, kept);
    if (lane == 0) s_kept[i] = kept;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *(volatile uint32_t*)tmem_holder;

  // The launch gives every thread 168 registers, 64512 in all.  Three sums of 64 columns need more: the two accumulating
  // warpgroups take 2 x 128 x 224 = 57344, the third keeps 128 x 56 = 7168.
  if (warp >= 8) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
  if (warp == 8) {
    // ------------------------------------------------------------------------- TMA producer
    const bool leader = elect_one();
    int stage = 0; uint32_t phase = 0, filled = 0;
    bool ok = true, stalled = P.stall_once == 0 || blockIdx.x != 0;
    for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
      const ProbeUnit w = probe_unit(P, u);
      const int row0 = w.tile / P.ntiles * BM, col0 = w.tile % P.ntiles * PBN;
      const CUtensorMap* ma = &maps.a[w.g];
      const CUtensorMap* me = &maps.e[w.g];
      const CUtensorMap* mb = &maps.b[w.g];
      for (int r = 0; r < rounds && ok; ++r) {
        const uint8_t* mask = s_mask + (w.g * rounds + r) * n_pad;
        RoundSteps it = round_steps(mask, s_kept[w.g * rounds + r], P.N, P.kT, r, P.S, w.slice);
        while (it.left > 0 && ok) {
          const bool kept = __any_sync(0xffffffffu, mask[it.n] != 0);
          const uint32_t bytes = PSTAGE - (r == 0 ? 0 : PA_BYTES) - (kept ? 0 : PA_BYTES);
          const int end = min(P.kT, it.kb + it.left);
          it.left -= end - it.kb;
          for (int kb = it.kb; kb < end; ++kb) {
            ok = __all_sync(0xffffffffu, mbar_wait(&empty[stage], phase ^ 1u, abort_flag, P.status));
            if (!ok) break;
            uint8_t* sa = base + stage * PSTAGE;
            if (stalled) {                       // otherwise nothing will ever arrive for this stage: a wait runs out
              if (leader) {
                mbar_expect_tx(&full[stage], bytes);
                if (r == 0) {
                  tma_load_3d(sa, ma, row0, kb * PK, it.n, &full[stage]);              // rows past T are zero-filled
                  tma_load_3d(sa + PCHUNK, ma, row0 + 64, kb * PK, it.n, &full[stage]);
                }
                if (kept) {
                  tma_load_3d(sa + PA_BYTES, me, row0, kb * PK, it.n, &full[stage]);
                  tma_load_3d(sa + PA_BYTES + PCHUNK, me, row0 + 64, kb * PK, it.n, &full[stage]);
                }
                tma_load_3d(sa + 2 * PA_BYTES, mb, col0, kb * PK, it.n, &full[stage]);
                tma_load_3d(sa + 2 * PA_BYTES + PCHUNK, mb, col0 + 64, kb * PK, it.n, &full[stage]);
              }
              __syncwarp();
            }
            stalled = true;
            ++filled;
            if (++stage == PSTAGES) { stage = 0; phase ^= 1u; }
          }
          it.kb = 0;
          ++it.n;
          if (r > 0 && it.left > 0)
            while (mask[it.n] == 0) ++it.n;
        }
      }
    }
    drain_loads(full, PSTAGES, stage, phase, filled, abort_flag, P.status);
  } else if (warp == 9) {
    // --------------------------------------------------------------------------- MMA issuer
    const bool leader = elect_one();
    constexpr uint32_t idesc = make_idesc(PBN, true, true);
    // 64-column chunks PCHUNK apart, 8 k-rows 1 KB apart, 128-byte swizzle
    constexpr uint64_t mn_major = ((uint64_t)(PCHUNK >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
    constexpr uint32_t k_step = UMMA_K * 128 >> 4;
    const int last16 = (P.T - (P.kT - 1) * PK + UMMA_K - 1) / UMMA_K;      // steps of 16 rows in the last step of a datum
    int stage = 0; uint32_t phase = 0, acc_phase = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
      const ProbeUnit w = probe_unit(P, u);
      for (int r = 0; r < rounds && ok; ++r) {
        const uint8_t* mask = s_mask + (w.g * rounds + r) * n_pad;
        RoundSteps it = round_steps(mask, s_kept[w.g * rounds + r], P.N, P.kT, r, P.S, w.slice);
        ok = __all_sync(0xffffffffu, mbar_wait(acc_empty, acc_phase ^ 1u, abort_flag, P.status));
        if (!ok) break;
        tc_fence_after();
        uint32_t begun = 0;
        int taken = 0;
        auto hand_over = [&]() {                 // the accumulators, complete when the products so far are
          if (leader) {
            *(volatile uint32_t*)&s_begun = begun;
            mbar_arrive(acc_full);
            umma_commit(acc_full);
          }
          __syncwarp();
          acc_phase ^= 1u;
        };
        while (it.left > 0 && ok) {
          const uint32_t m = __reduce_or_sync(0xffffffffu, (uint32_t)mask[it.n]), todo = m << 1 | (r == 0 ? 1u : 0u);
          const int end = min(P.kT, it.kb + it.left);
          it.left -= end - it.kb;
          for (int kb = it.kb; kb < end; ++kb) {
            if (taken == FLUSH) {
              hand_over();
              ok = __all_sync(0xffffffffu, mbar_wait(acc_empty, acc_phase ^ 1u, abort_flag, P.status));
              begun = 0;
              taken = 0;
            }
            ++taken;
            ok = ok && __all_sync(0xffffffffu, mbar_wait(&full[stage], phase, abort_flag, P.status));
            if (!ok) break;
            tc_fence_after();
            const uint32_t sa = smem_u32(base + stage * PSTAGE) >> 4;
            const uint64_t de = mn_major | (sa + (PA_BYTES >> 4)), db = mn_major | (sa + (2 * PA_BYTES >> 4));
            const int k16 = kb == P.kT - 1 ? last16 : PK / UMMA_K;
#pragma unroll
            for (int a = 0; a < 1 + PD; ++a) {
              if ((todo >> a & 1u) == 0u) continue;
              const uint64_t dop = a == 0 ? mn_major | sa : de;
              const uint32_t d = tmem_base + (uint32_t)(a * PBN);
#pragma unroll
              for (int k = 0; k < PK / UMMA_K; ++k)        // only the steps of 16 rows that hold any
                if (leader && k < k16)
                  umma_bf16(d, dop + (uint64_t)(k * k_step), db + (uint64_t)(k * k_step), idesc, k > 0 ? 1u : begun >> a & 1u);
            }
            if (leader) umma_commit(&empty[stage]);
            begun |= todo;
            if (++stage == PSTAGES) { stage = 0; phase ^= 1u; }
          }
          it.kb = 0;
          ++it.n;
          if (r > 0 && it.left > 0)
            while (mask[it.n] == 0) ++it.n;
        }
        if (!ok) break;
        hand_over();
      }
    }
    if (leader) drain_products(done, abort_flag, P.status);
    __syncwarp();
  }
  } else {
    // --------------------------------------------------------------------------------- the sums
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    const int eq = warp & 3, eg = warp >> 2;       // TMEM lane quarter, half of the columns
    constexpr int CW = PBN / 2;
    const uint32_t taddr = tmem_base + ((uint32_t)(eq * 32) << 16) + (uint32_t)(eg * CW);
    const int row = eq * 32 + lane;
    uint32_t acc_phase = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
      const ProbeUnit w = probe_unit(P, u);
      const int r0 = w.tile / P.ntiles * BM, col0 = w.tile % P.ntiles * PBN + eg * CW;
      float sum[1 + PD][CW];                       // G_s and the draws of a round
      double act = 0.0;
#pragma unroll
      for (int e = 0; e < CW; ++e) sum[0][e] = 0.f;
      for (int r = 0; r < rounds; ++r) {
#pragma unroll
        for (int a = 1; a <= PD; ++a)
#pragma unroll
          for (int e = 0; e < CW; ++e) sum[a][e] = 0.f;
        int parts = (round_steps(s_mask + (w.g * rounds + r) * n_pad, s_kept[w.g * rounds + r], P.N, P.kT, r, P.S, w.slice).left + FLUSH - 1) / FLUSH;
        do {
          // The lanes of a warp leave together.  No call here: it would put the sums into local memory.
          ok = __all_sync(0xffffffffu, mbar_wait_spin(acc_full, acc_phase, abort_flag, P.status));
          if (!ok) break;
          acc_phase ^= 1u;
          tc_fence_after();
          const uint32_t begun = *(volatile uint32_t*)&s_begun;
#pragma unroll
          for (int a = 0; a <= PD; ++a) {
            if (!__any_sync(0xffffffffu, (begun >> a & 1u) != 0u)) continue;      // the same for the whole warp: no predicates
#pragma unroll
            for (int h = 0; h < CW / 16; ++h) {
              uint32_t v[16];
              tmem_ld16(taddr + (uint32_t)(a * PBN + h * 16), v);
#pragma unroll
              for (int e = 0; e < 16; ++e) sum[a][h * 16 + e] += __uint_as_float(v[e]);
            }
          }
          // one arrival per warp: the arrivals of all threads at one barrier are served one after the other
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty);
        } while (--parts > 0);
        if (!ok) break;
        const int draws = round_draws(r, P.M);
        if (P.S > 1) {
#pragma unroll
          for (int a = 0; a <= PD; ++a) {
            if (a == 0 ? r > 0 : a > draws) continue;
            float* part = P.partial + ((size_t)u * (1 + P.M) + (a == 0 ? 0 : PD * r + a)) * BM * PBN + scratch_at(eg * (CW / 4), BM, row);
#pragma unroll
            for (int e = 0; e < CW; e += 4)
              *reinterpret_cast<float4*>(part + scratch_at(e / 4, BM, 0)) = make_float4(sum[a][e], sum[a][e + 1], sum[a][e + 2], sum[a][e + 3]);
          }
        } else {
#pragma unroll
          for (int a = 1; a <= PD; ++a) {
            if (a > draws) break;
            float t = 0.f;
#pragma unroll
            for (int e = 0; e < CW; ++e) {
              const float x = sum[a][e] - sum[0][e];
              t = fmaf(x, x, t);
            }
            act += (double)t;
          }
          if (r == 0 && r0 + row < P.d_out) {
            const int rows = gs_rows(P, r0);
            float* out = P.gs + w.g * P.gs_stride + gs_at(P, r0, rows, row, col0);
#pragma unroll
            for (int e = 0; e < CW; e += 4, out += rows * 4)
              if (col0 + e < P.d_in) *reinterpret_cast<float4*>(out) = make_float4(sum[0][e], sum[0][e + 1], sum[0][e + 2], sum[0][e + 3]);
          }
        }
      }
      if (!ok) break;
      if (P.S == 1) {      // a sum per warp: at a barrier of the eight those that gave up would be missed for good
        act = warp_sum(act);
        if (lane == 0) P.pact[(w.g * P.tiles + w.tile) * (ACC_THREADS / 32) + warp] = act;
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  // Not before all warps are here: the first thread to say so speaks for the CTA, and the CTAs of the next kernel would wait on
  // the SMs left to Eq. 3, whose CTAs need half of an SM's registers (20 us at the end of a probe).
  pdl_trigger();
  if (warp == 9) { tc_fence_after(); tmem_dealloc(tmem_base, 512); }
}

// Sliced tiles: sixteen CTAs per tile and batch add the slices in order and finish as the product's epilogue does.
constexpr int ADD_PARTS = 16, ADD_THREADS = 256;
__global__ void __launch_bounds__(ADD_THREADS) probe_add_kernel(ProbeParams P) {
  constexpr int BN = PBN;
  __shared__ double s_sum[ADD_THREADS / 32];
  pdl_wait();
  pdl_trigger();
  const int t = blockIdx.x / ADD_PARTS, rows = BM / ADD_PARTS, first = blockIdx.x % ADD_PARTS * rows;
  const int g = t / P.tiles, tile = t - g * P.tiles, r0 = tile / P.ntiles * BM;
  double act = 0.0;
  for (int i = threadIdx.x; i < rows * BN / 4; i += ADD_THREADS) {
    const int row = first + i % rows, q = i / rows, col = tile % P.ntiles * BN + q * 4;
    if (r0 + row >= P.d_out || col >= P.d_in) continue;
    float4 gs = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int ph = 0; ph <= P.M; ++ph) {
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int s = 0; s < P.S; ++s) {
        const float* part = P.partial + ((size_t)(t * P.S + s) * (1 + P.M) + ph) * BM * BN + scratch_at(q, BM, row);
        const float4 v = __ldcg(reinterpret_cast<const float4*>(part));
        x.x += v.x; x.y += v.y; x.z += v.z; x.w += v.w;
      }
      if (ph == 0) {
        gs = x;
        *reinterpret_cast<float4*>(P.gs + g * P.gs_stride + gs_at(P, r0, gs_rows(P, r0), row, col)) = x;
      } else {
        const float dx = x.x - gs.x, dy = x.y - gs.y, dz = x.z - gs.z, dw = x.w - gs.w;
        act += (double)((dx * dx + dy * dy) + (dz * dz + dw * dw));
      }
    }
  }
  block_act<ADD_THREADS>(P.pact + blockIdx.x, act, s_sum);
}

// The G_s of a group's batches into the running moments, four elements a thread: HBM / L2 bound.  m2 of the first batch is 0 and
// not stored, neither is anything of the last, whose squared deviations are summed per CTA in a fixed order.
constexpr int MOMENT_THREADS = 256;
__global__ void __launch_bounds__(MOMENT_THREADS) probe_moments_kernel(const float* gs, size_t gs_stride, float* mean, float* m2, long n4,
                                                                       int first, int batches, int M, double* ps) {
  __shared__ double s_sum[MOMENT_THREADS / 32];
  pdl_wait();
  const bool last = first + batches == M;
  double sq = 0.0;
  for (long i = (long)blockIdx.x * MOMENT_THREADS + threadIdx.x; i < n4; i += (long)gridDim.x * MOMENT_THREADS) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a, x[PG];
#pragma unroll
    for (int g = 0; g < PG; ++g)
      if (g < batches) x[g] = reinterpret_cast<const float4*>(gs + g * gs_stride)[i];
    if (first > 0) a = reinterpret_cast<float4*>(mean)[i];
    if (first > 1) b = reinterpret_cast<float4*>(m2)[i];
#pragma unroll
    for (int g = 0; g < PG; ++g)
      if (g < batches)
        sq += (double)((welford(x[g].x, first + g, M, a.x, b.x) + welford(x[g].y, first + g, M, a.y, b.y)) +
                       (welford(x[g].z, first + g, M, a.z, b.z) + welford(x[g].w, first + g, M, a.w, b.w)));
    if (!last) {
      reinterpret_cast<float4*>(mean)[i] = a;
      reinterpret_cast<float4*>(m2)[i] = b;
    }
  }
  if (last) block_act<MOMENT_THREADS>(ps + blockIdx.x, sq, s_sum);
}

// Alg. 1's averages from the tiles' and draws' sums, in a fixed order.
__global__ void __launch_bounds__(1024) probe_final_kernel(const double* __restrict__ pact, int np, const double* __restrict__ ps, int ns,
                                                           const double* __restrict__ vw, const double* __restrict__ sparsity, int M,
                                                           double scale, float* V_s, float* V_act, float* V_w, float* p_lo,
                                                           float* p_hi) {
  __shared__ double sh[3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double t[3] = {0.0, 0.0, 0.0};
  for (int i = threadIdx.x; i < np; i += 1024) t[0] += pact[i];
  for (int i = threadIdx.x; i < ns; i += 1024) t[1] += ps[i];
  for (int i = threadIdx.x; i < M * M; i += 1024) t[2] += vw[i];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    t[k] = warp_sum(t[k]);
    if (lane == 0) sh[k][warp] = t[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < 3; ++k) {
      t[k] = 0.0;
      for (int w = 0; w < 32; ++w) t[k] += sh[k][w];
    }
    const double mm = (double)M * (double)M;
    if (V_s) *V_s = (float)(scale * t[1] / (double)(M - 1));
    if (V_act) *V_act = (float)(scale * t[0] / mm);
    if (V_w) *V_w = (float)(t[2] / mm);
    double lo = 0.0, hi = 0.0;
    for (int i = 0; i < M; ++i) { lo += sparsity[i]; hi += sparsity[M + i]; }
    if (p_lo) *p_lo = (float)(lo / (double)M);
    if (p_hi) *p_hi = (float)(hi / (double)M);
  }
}

// [N][T][d] bf16, box of 64 columns x PK rows of one datum
bool datum_map(CUtensorMap* m, const void* p, int d, int T, int N) {
  const uint64_t dims[3] = {(uint64_t)d, (uint64_t)T, (uint64_t)N};
  const uint64_t strides[2] = {(uint64_t)d * 2, (uint64_t)T * d * 2};
  const uint32_t box[3] = {64, PK, 1};
  return make_map(m, p, 3, dims, strides, box);
}

cudaError_t run_probe(Handle* h, const ProbeMaps& maps, const ProbeParams& P, int ctas, cudaStream_t st) {
  static std::atomic<bool> attr_set[64];
  if (!attr_set[h->device].load(std::memory_order_acquire)) {
    const cudaError_t e = cudaFuncSetAttribute(probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PSMEM);
    if (e != cudaSuccess) return e;
    attr_set[h->device].store(true, std::memory_order_release);
  }
  cudaError_t e = launch_after(probe_kernel, dim3((unsigned)(P.units < ctas ? P.units : ctas)), dim3(PROBE_THREADS), PSMEM,
                               st, maps, P);
  h->launches += 1;
  if (e == cudaSuccess && P.S > 1) {
    e = launch_after(probe_add_kernel, dim3((unsigned)(P.units / P.S * ADD_PARTS)), dim3(ADD_THREADS), 0, st, P);
    h->launches += 1;
  }
  return e;
}

}  // namespace

// Shorter data leave the steps of 64 rows partly empty.  4096 rows, 768 -> 3072, M = 4, here and draw by draw: 251 and 709 us
// with T = 128, 276 and 690 with 64, 438 and 653 with 32, 794 and 687 with 16; 512 rows, 256 -> 256, M = 2: 37 and 119 with
// 32, 39 and 121 with 16.  The line at whole steps is on the safe side.  The scores of Eq. 3 must fit a CTA's shared memory.
bool probe_fused_ok(const Handle* h, int M) {
  return h->tensor_path && h->desc.T >= PROBE_MIN_T && (long)h->desc.N * h->desc.T <= SAMPLE_W_SMEM_ROWS && M * (M + 2) <= PARTIAL_SLOTS;
}

cudaError_t launch_probe_fused(Handle* h, int M, const void* const* X, const void* const* dY, float rho, float nu, double s_lo,
                               double s_hi, uint64_t seed, double scale, float* V_s, float* V_act, float* V_w, float* p_lo,
                               float* p_hi, cudaStream_t st) {
  static std::atomic<bool> attr_set[64];
#define PROBE_CUDA(...) do { const cudaError_t e_ = (__VA_ARGS__); if (e_ != cudaSuccess) return e_; } while (0)
  const vcas_layer_desc& d = h->desc;
  const int R = d.N * d.T, sub = h->sub_k, d_out = sub > 0 ? sub : d.d_out;
  const size_t vw_smem = (size_t)R * sizeof(float);
  if (h->device < 0 || h->device >= 64) return cudaErrorInvalidDevice;
  if (vw_smem > 32 * 1024 && !attr_set[h->device].load(std::memory_order_acquire)) {
    PROBE_CUDA(cudaFuncSetAttribute(probe_vw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    SAMPLE_W_SMEM_ROWS * (int)sizeof(float)));
    attr_set[h->device].store(true, std::memory_order_release);
  }
  ProbeGroup G = {};
  const int cols = d_out;
  auto up = [](size_t bytes) { return (bytes + 255) / 256 * 256; };
  G.b_at = up((size_t)R * sizeof(float));
  G.p_at = G.b_at + up((size_t)R * sizeof(float));
  G.keep_at = G.p_at + up((size_t)d.N * sizeof(float));
  G.scaled_at = G.keep_at + up((size_t)M * d.N);
  const size_t block = G.scaled_at + up((size_t)R * cols * 2);
  G.sub = reinterpret_cast<__nv_bfloat16*>(h->sub_dY);

  ProbeParams P = {};
  P.N = d.N; P.T = d.T; P.d_in = d.d_in; P.d_out = d_out;
  P.M = M;
  P.kT = (d.T + PK - 1) / PK;
  const int ctas = h->num_sms > 8 ? h->num_sms - 4 : h->num_sms;          // Eq. 3's CTAs run beside the product
  P.ntiles = (d.d_in + PBN - 1) / PBN;
  P.tiles = (d_out + BM - 1) / BM * P.ntiles;
  // slices of the contraction: as many as fill the CTAs once, of eight steps at least, and as the workspace holds
  auto slices = [&](int batches) {
    const int units = P.tiles * batches;
    long S = ctas / units;
    if (S > (long)d.N * P.kT / 8) S = (long)d.N * P.kT / 8;
    const long room = 3l * h->max_units * (BM * 256) / ((long)(1 + M) * BM * PBN * units);
    if (S > room) S = room;
    return (int)(S < 1 ? 1 : S);
  };
  // A group's blocks and its G_s lie where this probe needs nothing else.  The blocks: the compact operands of the two
  // workspace sets (each packG and packX, neighbours: R rows of d_out + d_in bf16, which hold one at least) and, if no
  // contraction is cut, the partial tiles.  G_s: Gs and Gact and, if one group is all there is, the moments behind them.
  const size_t elems = (size_t)d_out * d.d_in;
  P.gs = h->ws.Gs; P.gs_stride = (size_t)(h->ws.Gact - h->ws.Gs);
  P.pact = reinterpret_cast<double*>(h->ws2.Gact);
  P.partial = h->ws.partial_tiles;
  int most = 0;
  auto place = [&](void* region, size_t bytes, int limit) {
    for (size_t at = 0; at + block <= bytes && most < limit; at += block) G.block[most++] = reinterpret_cast<uint8_t*>(region) + at;
  };
  const size_t arena = (size_t)h->R_pad * (d.d_out + d.d_in) * 2;
  const int limit = sub > 0 && SUB_MAX / sub < PG ? SUB_MAX / sub : PG;
  place(h->ws.packG, arena, limit);
  place(h->ws2.packG, arena, limit);
  if (M <= limit && most < M && slices(M) == 1) place(h->ws.partial_tiles, 3 * (size_t)h->max_units * BM * 256 * sizeof(float), M);
  if (most < 1) return cudaErrorInvalidValue;
  if (most > M) most = M;
  while (most > 1 && most * rounds_of(M) * ((d.N + 3) & ~3) > PMASKS) --most;      // M < 64, N < 897: one batch fits
  if (most < M && most > 2) most = 2;                // the moments keep their place
  int sums = 0;                                      // entries of pact so far
  double* ps = h->ws2.partial;
  const int moment_ctas = (int)(elems / 4 / MOMENT_THREADS + 1 < 592 ? elems / 4 / MOMENT_THREADS + 1 : 592);
  P.status = h->ws.status; P.wait_limit_ns = h->wait_limit_ns; P.stall_once = h->stall_once;

  DrawParams Q = {};
  Q.vw = h->ws.partial; Q.sparsity = h->ws.partial + M * M; Q.status = h->ws.status;
  Q.N = d.N; Q.T = d.T; Q.M = M; Q.rho = rho; Q.nu = nu; Q.s_lo = s_lo; Q.s_hi = s_hi; Q.seed = seed;

  cudaStream_t side = h->side_stream;
  for (int i0 = 0; i0 < M; i0 += most) {
    const int batches = M - i0 < most ? M - i0 : most;
    ProbeMaps maps;
    for (int g = 0; g < batches; ++g) {
      G.dY[g] = (const __nv_bfloat16*)dY[i0 + g]; G.X[g] = (const __nv_bfloat16*)X[i0 + g];
      if (!datum_map(&maps.a[g], sub > 0 ? (const void*)(G.sub + (size_t)g * R * sub) : dY[i0 + g], d_out, d.T, d.N) ||
          !datum_map(&maps.e[g], G.scaled(g), d_out, d.T, d.N) || !datum_map(&maps.b[g], X[i0 + g], d.d_in, d.T, d.N))
        return cudaErrorInvalidValue;
    }
    if (i0 > 0) PROBE_CUDA(cudaStreamWaitEvent(st, h->ev_join, 0));       // Eq. 3 of the group before reads its scratch
    long blocks = (2l * R * batches + 7) / 8;
    if (blocks > (1l << 20)) blocks = 1l << 20;
    if (sub > 0) probe_norms_kernel<true><<<(unsigned)blocks, 256, 0, st>>>(G, batches, R, d.d_out, d.d_in, h->sub_rows, sub);
    else probe_norms_kernel<false><<<(unsigned)blocks, 256, 0, st>>>(G, batches, R, d.d_out, d.d_in, nullptr, 0);
    PROBE_CUDA(cudaGetLastError());
    Q.first_batch = i0;
    const dim3 draw_grid((unsigned)(M + 1), (unsigned)batches);
    const dim3 threads(DRAW_THREADS);
    PROBE_CUDA(d.N <= 32    ? launch_after(probe_draw_kernel<1>, draw_grid, threads, 0, st, G, Q)
               : d.N <= 64  ? launch_after(probe_draw_kernel<2>, draw_grid, threads, 0, st, G, Q)
               : d.N <= 128 ? launch_after(probe_draw_kernel<4>, draw_grid, threads, 0, st, G, Q)
               : d.N <= 256 ? launch_after(probe_draw_kernel<8>, draw_grid, threads, 0, st, G, Q)
                            : launch_after(probe_draw_kernel<32>, draw_grid, threads, 0, st, G, Q));
    PROBE_CUDA(cudaEventRecord(h->ev_fork, st));
    PROBE_CUDA(cudaStreamWaitEvent(side, h->ev_fork, 0));
    PROBE_CUDA(launch_maybe_after(false, probe_vw_kernel, dim3((unsigned)M, (unsigned)batches), dim3(SAMPLER_THREADS), vw_smem, side, G, Q));
    PROBE_CUDA(cudaEventRecord(h->ev_join, side));
    const long pieces = (long)R * (cols / 8);
    long scale_blocks = (pieces + 4 * SCALE_THREADS - 1) / (4 * SCALE_THREADS);
    if (scale_blocks > 8l * h->num_sms / batches) scale_blocks = 8l * h->num_sms / batches;
    const dim3 scale_grid((unsigned)scale_blocks, (unsigned)batches);
    const size_t scale_smem = (size_t)d.N * sizeof(float);
    PROBE_CUDA(sub > 0 ? launch_after(probe_scale_kernel<true>, scale_grid, dim3(SCALE_THREADS), scale_smem, st, G, d.N, d.T, M, cols)
                       : launch_after(probe_scale_kernel<false>, scale_grid, dim3(SCALE_THREADS), scale_smem, st, G, d.N, d.T, M, cols));
    h->launches += 4;
    P.batches = batches;
    P.S = slices(batches);
    P.units = P.tiles * batches * P.S;
    for (int g = 0; g < batches; ++g) P.keep[g] = G.block[g] + G.keep_at;
    PROBE_CUDA(run_probe(h, maps, P, ctas, st));
    const int parts = P.tiles * batches * (P.S > 1 ? ADD_PARTS : ACC_THREADS / 32);
    sums += parts;
    P.pact += parts;
    PROBE_CUDA(launch_after(probe_moments_kernel, dim3((unsigned)moment_ctas), dim3(MOMENT_THREADS), 0, st, (const float*)P.gs,
                            P.gs_stride, h->ws.mean, h->ws.m2, (long)(elems / 4), i0, batches, M, ps));
    h->launches += 1;
  }
  PROBE_CUDA(cudaStreamWaitEvent(st, h->ev_join, 0));
  probe_final_kernel<<<1, 1024, 0, st>>>(reinterpret_cast<const double*>(h->ws2.Gact), sums, ps, moment_ctas, Q.vw, Q.sparsity, M, scale, V_s, V_act, V_w, p_lo, p_hi);
  h->launches += 1;
#undef PROBE_CUDA
  return cudaGetLastError();
}

}  // namespace vcas
