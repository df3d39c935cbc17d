// The variance probe of a tensor-path layer (Alg. 1, App. D) with one product per batch.
//
// The gradient of a batch is a sum over its data, G_s = sum_n D_n with D_n = dY_n^T X_n, and a draw of SampleA only
// weights the terms: G_act,j = sum_n (keep_jn / p_jn) D_n.  The product kernel therefore forms every D_n once, in a
// fresh TMEM accumulator, and the epilogue warps add it to G_s and, weighted with w_jn = keep_jn / p_jn where that is not 0, to
// G_act,j of up to four draws in fp32 registers; V_act needs nothing but the squares of G_act,j - G_s, and G_s goes straight
// into the running mean and squared deviation of V_s.  (Draws past the first four, whose pass does not form G_s, add up the
// differences with keep_jn / p_jn - 1.)  (Running sums in TMEM with summation by parts save the
// registers of G_s, but lose the small data, whose weights 1 / p are large, in the rounding of the large ones.)
// No draw packs rows or has a product of its own:
// M batches of M draws cost M products instead of M + rho M^2, and the results carry no rounding of rescaled rows.
//
// Four launches serve up to four batches: norms of the rows of dY and X (which also gathers the sampled columns of dY), one
// CTA per draw for p, mask and w, one CTA per draw for Eq. 3 (beside the product, on the side stream), the product.
// Measured on B200: 4096 rows, 768 -> 3072, M = 4: 664 -> 179 us; 16384 rows, 4096 -> 128 of 11008, M = 2: 521 -> 241 us.
#include <atomic>

#include "rows.cuh"
#include "umma.cuh"
#include "water.cuh"

namespace vcas {
namespace {

constexpr int PD = 4;                        // most draws a product pass serves
constexpr int PG = 4;                        // most batches a launch serves
constexpr int PROBE_THREADS = 12 * 32;       // warps 0-7 accumulate, 8 loads, 9 issues, 10 and 11 fill the warpgroup
constexpr int ACC_THREADS = 256;
constexpr int PBUFS = 8;                     // TMEM accumulators of data in flight: all 512 columns
constexpr int PK = 128;                      // rows of a step
constexpr int PCHUNK = 64 * PK * 2;          // 64 columns of a step
constexpr int PBN = 64;                      // tile columns: 32 per accumulating thread and (1 + D) sums of each
constexpr int PSTAGE = (BM + PBN) / 64 * PCHUNK;
constexpr int PSTAGES = 4;
constexpr int PSMEM = PSTAGES * PSTAGE + 1024 /*alignment slack*/ + 256 /*barriers*/;

// What a group of batches leaves for its product
struct ProbeGroup {
  const __nv_bfloat16* dY[PG]; const __nv_bfloat16* X[PG];
  float* a; float* b;              // [batch][R] row square-norms of dY and X
  float* p;                        // [batch][M][N] keep probabilities
  float* w;                        // [batch][pass][N][PD] keep / p (1 past the last draw)
  __nv_bfloat16* sub;              // [batch][R][k] sampled columns of dY
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
    if (lane == 0) (y ? G.a : G.b)[(size_t)g * R + r] = s;
  }
}

// ------------------------------------------------------------------------------------ the draws
struct DrawParams {
  const float* a; const float* b;  // [batch][R]
  float* p; float* w;              // as in ProbeGroup
  double* sparsity;                // [2][batch of the probe] p_lo, p_hi
  double* vw;                      // [batch of the probe][M] Eq. 3
  int32_t* status;
  int N, T, M, passes, first_batch;
  float rho, nu;
  double s_lo, s_hi;
  uint64_t seed;
};

// Where w of (batch g, draw j, datum n) is.
__device__ __forceinline__ size_t w_index(const DrawParams& P, int g, int j, int n) {
  return (((size_t)g * P.passes + j / PD) * P.N + n) * PD + j % PD;
}

// CTA (j, batch), j < M: SampleA of draw j (Sec. 4.1), as in the sampled backward.  CTA (PD passes, batch): Eq. 4's sparsity.
constexpr int DRAW_THREADS = 512;
template <int SLOTS>
__global__ void __launch_bounds__(DRAW_THREADS) probe_draw_kernel(DrawParams P) {
  __shared__ float s_g[32 * SLOTS], s_sorted[32 * SLOTS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = blockIdx.x, g = blockIdx.y;
  for (int n = threadIdx.x; n < 32 * SLOTS; n += DRAW_THREADS) s_g[n] = 0.f;
  pdl_wait();
  pdl_trigger();
  if (j >= P.M && j < PD * P.passes) {
    for (int n = threadIdx.x; n < P.N; n += DRAW_THREADS) P.w[w_index(P, g, j, n)] = 1.f;
    return;
  }
  __syncthreads();
  for (int n = warp; n < P.N; n += DRAW_THREADS / 32) {
    const float s = datum_sqnorm_warp(P.a + ((size_t)g * P.N + n) * P.T, P.T, lane);
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
    const size_t o = ((size_t)g * P.M + j) * P.N;
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
      const int n = lane + 32 * i;
      if (n < P.N) {
        P.p[o + n] = v[i];
        P.w[w_index(P, g, j, n)] = bernoulli_keep(v[i], seed, 0u, (uint64_t)n) ? 1.0f / v[i] : 0.f;
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
__global__ void __launch_bounds__(SAMPLER_THREADS) probe_vw_kernel(DrawParams P) {
  extern __shared__ __align__(16) float s_w[];
  __shared__ WShared sh;
  const int tid = threadIdx.x, j = blockIdx.x, g = blockIdx.y, n = P.N * P.T;
  const size_t o = ((size_t)g * P.M + j) * P.N;
  const float* a = P.a + (size_t)g * n;
  const float* b = P.b + (size_t)g * n;
  for (int i = tid; i < n; i += SAMPLER_THREADS) {
    const int d = i / P.T;
    s_w[i] = P.w[w_index(P, g, j, d)] > 0.f ? sqrtf(a[i]) * sqrtf(b[i]) / P.p[o + d] : 0.f;
  }
  float dummy = 0.f;
  int kept = 0;
  for (int i = tid; i < P.N; i += SAMPLER_THREADS) kept += P.w[w_index(P, g, j, i)] > 0.f ? 1 : 0;
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

// ----------------------------------------------------------------------------------- the product
struct ProbeMaps { CUtensorMap a[PG], b[PG]; };      // per batch: dY (or its sampled columns) and X
struct ProbeParams {
  const float4* w;                 // [batch][pass][N] of PD draws
  float* mean; float* m2;          // d_out x d_in, by tiles: running mean and squared deviation of G_s
  double* pact; double* ps;        // [tiles] sum of squares of the differences so far; sum of m2 (last batch)
  float* partial;                  // [batch][unit][1 + D][128 x 64] when a tile's data are cut into slices
  int N, T, d_in, d_out, kT, steps, S, per, ntiles, units;    // kT: steps of a datum
  int first_batch, batches, M;
  int pass, passes;                // the draws of this pass are pass * PD ...
  int fresh;                       // pact starts here
  int32_t* status;
  unsigned long long wait_limit_ns;
  int stall_once;
};

// Welford's update of one element of batch `i` of M: returns its final squared deviation in the last batch, else 0.
__device__ __forceinline__ float welford(float x, int i, int M, float& mean, float& m2) {
  if (i == 0) { mean = x; m2 = 0.f; return 0.f; }
  const float d = x - mean;
  mean = fmaf(d, 1.0f / (float)(i + 1), mean);
  m2 = fmaf(d, x - mean, m2);
  return i == M - 1 ? m2 : 0.f;
}
// Where a tile's columns 4 q .. 4 q + 3 of `row` are in a scratch tile of `rows` rows.  The threads of a warp have consecutive
// rows, so they take 512 consecutive bytes: in rows of 64 columns an instruction met 32 cache lines, and the moments of a tile
// and batch took 4 us in which the products could run eight data ahead at most (189 -> 176 us for 768 -> 3072, M = 4).
__device__ __forceinline__ size_t scratch_at(int q, int rows, int row) { return ((size_t)q * rows + row) * 4; }
// G_s of batch i at W columns from 4 q0 on into the running moments, all loads before the first store.  m2 of the first batch
// is 0 and not stored, neither is anything of the last.  The moments of a tile have its rows below d_out.
template <int W>
__device__ __forceinline__ float welford_row(const ProbeParams& P, int i, int tile, int row, int q0, const float (&x)[W]) {
  float4 mean[W / 4], m2[W / 4];
  const int r0 = tile / P.ntiles * BM, rows = min(BM, P.d_out - r0);
  const size_t o = (size_t)r0 * P.d_in + (size_t)(tile % P.ntiles) * rows * PBN + scratch_at(q0, rows, row);
  const size_t step = (size_t)rows * 4;
#pragma unroll
  for (int e = 0; e < W / 4; ++e) {
    mean[e] = i > 0 ? *reinterpret_cast<const float4*>(P.mean + o + e * step) : make_float4(0.f, 0.f, 0.f, 0.f);
    m2[e] = i > 1 ? *reinterpret_cast<const float4*>(P.m2 + o + e * step) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float r = 0.f;
#pragma unroll
  for (int e = 0; e < W / 4; ++e) {
    r += (welford(x[4 * e], i, P.M, mean[e].x, m2[e].x) + welford(x[4 * e + 1], i, P.M, mean[e].y, m2[e].y)) +
         (welford(x[4 * e + 2], i, P.M, mean[e].z, m2[e].z) + welford(x[4 * e + 3], i, P.M, mean[e].w, m2[e].w));
    if (i < P.M - 1) {
      *reinterpret_cast<float4*>(P.mean + o + e * step) = mean[e];
      if (i > 0) *reinterpret_cast<float4*>(P.m2 + o + e * step) = m2[e];
    }
  }
  return r;
}
// The sums of THREADS threads over a tile, added in a fixed order by thread 0.
template <int THREADS>
__device__ __forceinline__ void tile_sums(const ProbeParams& P, bool exact, int tile, double act, double sq, double (*sh)[2]) {
  act = warp_sum(act);
  sq = warp_sum(sq);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { sh[warp][0] = act; sh[warp][1] = sq; }
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
  if (threadIdx.x == 0) {
    double t0 = 0.0, t1 = 0.0;
    for (int w = 0; w < THREADS / 32; ++w) { t0 += sh[w][0]; t1 += sh[w][1]; }
    P.pact[tile] = P.fresh ? t0 : P.pact[tile] + t0;
    if (exact && P.first_batch + P.batches == P.M) P.ps[tile] = t1;
  }
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// A unit is a tile of the gradient and a contiguous range of a batch's steps, worked off batch by batch; a step is up to
// 128 rows of one datum.  EXACT: this pass makes G_s.
template <int D, bool EXACT>
__global__ void __launch_bounds__(PROBE_THREADS, 1)
probe_kernel(const __grid_constant__ ProbeMaps maps, ProbeParams P) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ double s_sum[ACC_THREADS / 32][2];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(base + PSTAGES * PSTAGE);
  uint64_t* empty = full + PSTAGES;
  uint64_t* acc_full = empty + PSTAGES;      // [PBUFS] a datum's product is complete
  uint64_t* acc_empty = acc_full + PBUFS;      // [PBUFS] ... has been read
  uint32_t* tmem_holder = (uint32_t*)(acc_empty + PBUFS);
  volatile int* abort_flag = (int*)(tmem_holder + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < PSTAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < PBUFS; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], ACC_THREADS / 32); }
    *abort_flag = 0;
    *reinterpret_cast<volatile unsigned long long*>(abort_flag + 5) = P.wait_limit_ns;     // read by mbar_wait
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 9) tmem_alloc(tmem_holder, PBUFS * PBN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *(volatile uint32_t*)tmem_holder;
  pdl_wait();

  // The launch gives every thread 168 registers, 64512 in all.  The sums of four draws need more: the accumulating warpgroups
  // take 2 x 128 x 224 = 57344, the third keeps 128 x 56 = 7168.
  if (warp >= 8) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
  if (warp == 8) {
    // ------------------------------------------------------------------------- TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      bool ok = true, stalled = false;
      for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
        const int tile = u / P.S, s0 = (u - tile * P.S) * P.per, s1 = min(P.steps, s0 + P.per);
        const int row0 = tile / P.ntiles * BM, col0 = tile % P.ntiles * PBN;
        for (int g = 0; g < P.batches && ok; ++g) {
          int n = s0 / P.kT, kb = s0 - n * P.kT;
          for (int s = s0; s < s1; ++s) {
            ok = mbar_wait(&empty[stage], phase ^ 1u, abort_flag, P.status);
            if (!ok) break;
            uint8_t* sa = base + stage * PSTAGE;
            if (P.stall_once != 0 && blockIdx.x == 0 && !stalled) {
              stalled = true;                  // nothing will ever arrive for this stage: a wait runs out
            } else {
              mbar_expect_tx(&full[stage], PSTAGE);
              tma_load_3d(sa, &maps.a[g], row0, kb * PK, n, &full[stage]);           // rows past T are zero-filled
              tma_load_3d(sa + PCHUNK, &maps.a[g], row0 + 64, kb * PK, n, &full[stage]);
#pragma unroll
              for (int j = 0; j < PBN / 64; ++j)
                tma_load_3d(sa + (2 + j) * PCHUNK, &maps.b[g], col0 + j * 64, kb * PK, n, &full[stage]);
            }
            if (++stage == PSTAGES) { stage = 0; phase ^= 1u; }
            if (++kb == P.kT) { kb = 0; ++n; }
          }
        }
      }
    }
  } else if (warp == 9) {
    // --------------------------------------------------------------------------- MMA issuer
    const bool leader = elect_one();
    constexpr uint32_t idesc = make_idesc(PBN, true, true);
    // 64-column chunks PCHUNK apart, 8 k-rows 1 KB apart, 128-byte swizzle
    constexpr uint64_t mn_major = ((uint64_t)(PCHUNK >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
    constexpr uint32_t k_step = UMMA_K * 128 >> 4;
    const int last_rows = P.T - (P.kT - 1) * PK;
    int stage = 0; uint32_t phase = 0, buf = 0, buf_phase = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
      const int s0 = (u % P.S) * P.per, s1 = min(P.steps, s0 + P.per);
      for (int g = 0; g < P.batches && ok; ++g) {
        int kb = s0 % P.kT;
        bool fresh = true;
        for (int s = s0; s < s1 && ok; ++s) {
          if (fresh) ok = __all_sync(0xffffffffu, mbar_wait(&acc_empty[buf], buf_phase ^ 1u, abort_flag, P.status));
          ok = ok && __all_sync(0xffffffffu, mbar_wait(&full[stage], phase, abort_flag, P.status));
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(base + stage * PSTAGE);
          const uint64_t da = mn_major | (sa >> 4), db = mn_major | ((sa + 2 * PCHUNK) >> 4);
          const uint32_t d = tmem_base + buf * (uint32_t)PBN;
          auto product = [&](int k, uint32_t accumulate) {
            umma_bf16(d, da + (uint64_t)(k * k_step), db + (uint64_t)(k * k_step), idesc, accumulate);
          };
          const bool ends = kb == P.kT - 1;
          const int rows = ends ? last_rows : PK;
          const bool done = ends || s == s1 - 1;
          if (leader) {
            product(0, fresh ? 0u : 1u);
            if (rows == PK) {
#pragma unroll
              for (int k = 1; k < PK / UMMA_K; ++k) product(k, 1u);
            } else {                           // the steps of 16 rows that hold any
              for (int k = 1; k * UMMA_K < rows; ++k) product(k, 1u);
            }
            umma_commit(&empty[stage]);
            if (done) umma_commit(&acc_full[buf]);
          }
          if (done && ++buf == PBUFS) { buf = 0; buf_phase ^= 1u; }
          fresh = ends;
          kb = ends ? 0 : kb + 1;
          if (++stage == PSTAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
  }
  } else {
    // ------------------------------------------------------------------ accumulation and output
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    const int eq = warp & 3, eg = warp >> 2;       // TMEM lane quarter, half of the columns
    constexpr int CW = PBN / 2;
    const uint32_t tlane = ((uint32_t)(eq * 32) << 16) + (uint32_t)(eg * CW);
    uint32_t buf = 0, buf_phase = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < P.units && ok; u += gridDim.x) {
      const int tile = u / P.S, s0 = (u - tile * P.S) * P.per, s1 = min(P.steps, s0 + P.per);
      const int n0 = s0 / P.kT, n1 = (s1 - 1) / P.kT + 1;
      const int row = eq * 32 + lane, r0 = tile / P.ntiles * BM + row;
      double act = 0.0, sq = 0.0;
      for (int g = 0; g < P.batches; ++g) {
        uint64_t gs2[CW / 2], df2[D][CW / 2];      // two columns per register pair and instruction
#pragma unroll
        for (int e = 0; e < CW / 2; ++e) {
          gs2[e] = 0ull;
#pragma unroll
          for (int j = 0; j < D; ++j) df2[j][e] = 0ull;
        }
        const float4* wg = P.w + ((size_t)g * P.passes + P.pass) * P.N;
        float4 next = __ldg(wg + n0);
        for (int n = n0; n < n1; ++n) {
          const float w[4] = {next.x, next.y, next.z, next.w};
          next = __ldg(wg + min(n + 1, n1 - 1));   // on its way while this datum is added
          // The lanes of a warp leave together.  No call here: it would put the sums held in registers into local memory.
          ok = __all_sync(0xffffffffu, mbar_wait_spin(&acc_full[buf], buf_phase, abort_flag, P.status));
          if (!ok) break;
          tc_fence_after();
          static_assert(CW == 32, "one load");
          uint32_t v[CW];
          tmem_ld32(tmem_base + tlane + buf * (uint32_t)PBN, v);
          uint64_t x[CW / 2];
#pragma unroll
          for (int e = 0; e < CW / 2; ++e) x[e] = pack2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
          // fp32-bound: 0.35 us a datum with an FMA per draw and element, of 0.62 in all; dropped data cost a draw nothing
          if (EXACT) {
#pragma unroll
            for (int e = 0; e < CW / 2; ++e) gs2[e] = add2(gs2[e], x[e]);
          }
#pragma unroll
          for (int j = 0; j < D; ++j) {
            if (EXACT && !__any_sync(0xffffffffu, w[j] != 0.f)) continue;      // the same for the whole warp: no predicates
            const float c = EXACT ? w[j] : w[j] - 1.0f;
            const uint64_t cc = pack2(c, c);
#pragma unroll
            for (int e = 0; e < CW / 2; ++e) df2[j][e] = fma2(cc, x[e], df2[j][e]);
          }
          // one arrival per warp: the arrivals of all threads at one barrier are served one after the other
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[buf]);
          if (++buf == PBUFS) { buf = 0; buf_phase ^= 1u; }
        }
        if (!ok) break;
        float gs[CW], df[D][CW];
#pragma unroll
        for (int e = 0; e < CW / 2; ++e) {
          unpack2(gs2[e], gs[2 * e], gs[2 * e + 1]);
#pragma unroll
          for (int j = 0; j < D; ++j) {
            unpack2(df2[j][e], df[j][2 * e], df[j][2 * e + 1]);
            if (EXACT) { df[j][2 * e] -= gs[2 * e]; df[j][2 * e + 1] -= gs[2 * e + 1]; }
          }
        }
        float* part = P.partial + ((size_t)g * P.units + u) * (1 + D) * BM * PBN + scratch_at(eg * (CW / 4), BM, row);
        if (P.S > 1) {
#pragma unroll
          for (int e = 0; e < CW; e += 4) {
            if (EXACT) *reinterpret_cast<float4*>(part + scratch_at(e / 4, BM, 0)) = make_float4(gs[e], gs[e + 1], gs[e + 2], gs[e + 3]);
#pragma unroll
            for (int j = 0; j < D; ++j)
              *reinterpret_cast<float4*>(part + (size_t)(1 + j) * BM * PBN + scratch_at(e / 4, BM, 0)) = make_float4(df[j][e], df[j][e + 1], df[j][e + 2], df[j][e + 3]);
          }
        } else if (r0 < P.d_out) {
#pragma unroll
          for (int j = 0; j < D; ++j) {
            float t = 0.f;
#pragma unroll
            for (int e = 0; e < CW; ++e) t = fmaf(df[j][e], df[j][e], t);
            act += (double)t;
          }
          if (EXACT) sq += (double)welford_row<CW>(P, P.first_batch + g, tile, row, eg * (CW / 4), gs);
        }
      }
      if (!ok) break;
      if (P.S == 1) tile_sums<ACC_THREADS>(P, EXACT, tile, act, sq, s_sum);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  // Not before all warps are here: the first thread to say so speaks for the CTA, and the CTAs of the kernel that adds slices
  // would wait on the SMs left to Eq. 3, whose CTAs need all of an SM's registers (20 us at the end of a probe).
  pdl_trigger();
  if (warp == 9) { tc_fence_after(); tmem_dealloc(tmem_base, PBUFS * PBN); }
}

// Sliced tiles: four CTAs per tile add the slices in order and finish as the product's epilogue does; a CTA's sums are
// kept like those of a tile.
constexpr int ADD_PARTS = 4, ADD_THREADS = 256;
template <int D, bool EXACT>
__global__ void __launch_bounds__(ADD_THREADS) probe_add_kernel(ProbeParams P) {
  constexpr int BN = PBN;
  __shared__ double s_sum[ADD_THREADS / 32][2];
  pdl_wait();
  const int tile = blockIdx.x / ADD_PARTS, rows = BM / ADD_PARTS, first = blockIdx.x % ADD_PARTS * rows;
  double act = 0.0, sq = 0.0;
  for (int i = threadIdx.x; i < rows * BN / 4; i += ADD_THREADS) {
    const int row = first + i % rows, q0 = i / rows;
    if (tile / P.ntiles * BM + row >= P.d_out) continue;
    for (int g = 0; g < P.batches; ++g) {
      float x[1 + D][4] = {};
#pragma unroll 4
      for (int s = 0; s < P.S; ++s) {
        const float* part = P.partial + ((size_t)g * P.units + tile * P.S + s) * (1 + D) * BM * BN + scratch_at(q0, BM, row);
#pragma unroll
        for (int q = EXACT ? 0 : 1; q <= D; ++q) {
          const float4 v = __ldcg(reinterpret_cast<const float4*>(part + (size_t)q * BM * BN));
          x[q][0] += v.x; x[q][1] += v.y; x[q][2] += v.z; x[q][3] += v.w;
        }
      }
#pragma unroll
      for (int q = 1; q <= D; ++q) act += (double)((x[q][0] * x[q][0] + x[q][1] * x[q][1]) + (x[q][2] * x[q][2] + x[q][3] * x[q][3]));
      if (EXACT) sq += (double)welford_row<4>(P, P.first_batch + g, tile, row, q0, x[0]);
    }
  }
  tile_sums<ADD_THREADS>(P, EXACT, blockIdx.x, act, sq, s_sum);
}

// Alg. 1's averages from the tiles' and draws' sums, in a fixed order.
__global__ void __launch_bounds__(1024) probe_final_kernel(const double* __restrict__ pact, const double* __restrict__ ps, int tiles,
                                                           const double* __restrict__ vw, const double* __restrict__ sparsity, int M,
                                                           double scale, float* V_s, float* V_act, float* V_w, float* p_lo,
                                                           float* p_hi) {
  __shared__ double sh[3][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double t[3] = {0.0, 0.0, 0.0};
  for (int i = threadIdx.x; i < tiles; i += 1024) { t[0] += pact[i]; t[1] += ps[i]; }
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

// Tiles of a pass and the slices of their data: as many as fill the CTAs once.
void probe_tiling(ProbeParams& P, int ctas) {
  P.ntiles = (P.d_in + PBN - 1) / PBN;
  const int tiles = (P.d_out + BM - 1) / BM * P.ntiles;
  P.S = ctas / tiles;
  if (P.S > P.steps / 4) P.S = P.steps / 4;
  if (P.S < 1) P.S = 1;
  P.per = (P.steps + P.S - 1) / P.S;
  P.S = (P.steps + P.per - 1) / P.per;                                    // no empty slice
  P.units = tiles * P.S;
}
// entries of pact and ps that a pass writes
int probe_sums(const ProbeParams& P) { return P.S > 1 ? P.units / P.S * ADD_PARTS : P.units; }

template <int D, bool EXACT>
cudaError_t run_probe(Handle* h, const ProbeMaps& maps, const ProbeParams& P, int ctas, cudaStream_t st) {
  static std::atomic<bool> attr_set[64];
  if (!attr_set[h->device].load(std::memory_order_acquire)) {
    const cudaError_t e = cudaFuncSetAttribute(probe_kernel<D, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize, PSMEM);
    if (e != cudaSuccess) return e;
    attr_set[h->device].store(true, std::memory_order_release);
  }
  cudaError_t e = launch_after(probe_kernel<D, EXACT>, dim3((unsigned)(P.units < ctas ? P.units : ctas)), dim3(PROBE_THREADS),
                               PSMEM, st, maps, P);
  h->launches += 1;
  if (e == cudaSuccess && P.S > 1) {
    e = launch_after(probe_add_kernel<D, EXACT>, dim3((unsigned)(P.units / P.S * ADD_PARTS)), dim3(ADD_THREADS), 0, st, P);
    h->launches += 1;
  }
  return e;
}

}  // namespace

// Shorter data would leave the steps of 128 rows mostly empty, and every datum costs a pass of the epilogue over its tile;
// the scores of Eq. 3 must fit a CTA's shared memory.
bool probe_fused_ok(const Handle* h, int M) {
  return h->tensor_path && h->desc.T >= 64 && (long)h->desc.N * h->desc.T <= SAMPLE_W_SMEM_ROWS && M * (M + 2) <= PARTIAL_SLOTS;
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
  // What a group's batches leave for its product lies in packG and packX, which are neighbours and which this probe does not
  // need otherwise (R rows of d_out + d_in bf16: at least one batch fits, since the sampled rows are fewer than d_out).
  const int passes = (M + PD - 1) / PD;
  const size_t scratch = (size_t)h->R_pad * (d.d_out + d.d_in) * 2;
  const size_t per_batch = (size_t)R * (2 * sizeof(float) + 2 * (size_t)sub) + (size_t)(M + passes * PD) * d.N * sizeof(float) + 1280;
  int most = (int)(scratch / per_batch);
  if (most < 1) return cudaErrorInvalidValue;
  if (most > PG) most = PG;
  if (most > M) most = M;
  ProbeGroup G = {};
  uint8_t* cur = reinterpret_cast<uint8_t*>(h->ws.packG);
  auto take = [&](size_t bytes) { uint8_t* q = cur; cur += (bytes + 255) / 256 * 256; return q; };
  G.sub = reinterpret_cast<__nv_bfloat16*>(take((size_t)most * R * sub * 2));
  G.a = reinterpret_cast<float*>(take((size_t)most * R * sizeof(float)));
  G.b = reinterpret_cast<float*>(take((size_t)most * R * sizeof(float)));
  G.p = reinterpret_cast<float*>(take((size_t)most * M * d.N * sizeof(float)));
  G.w = reinterpret_cast<float*>(take((size_t)most * passes * PD * d.N * sizeof(float)));

  ProbeParams P = {};
  P.N = d.N; P.T = d.T; P.d_in = d.d_in; P.d_out = d_out;
  P.kT = (d.T + PK - 1) / PK;
  P.steps = d.N * P.kT;
  const int ctas = h->num_sms > 2 * PD ? h->num_sms - PD : h->num_sms;    // Eq. 3's CTAs run beside the product
  // all passes have the same tiles, so that their sums add up entry by entry
  probe_tiling(P, ctas);
  const int sums = probe_sums(P);
  P.mean = h->ws.mean; P.m2 = h->ws.m2;
  P.pact = reinterpret_cast<double*>(h->ws.Gact);                         // this probe keeps no gradient
  P.ps = P.pact + sums;
  P.partial = h->ws.partial_tiles;
  P.M = M; P.w = reinterpret_cast<const float4*>(G.w); P.passes = passes;
  P.status = h->ws.status; P.wait_limit_ns = h->wait_limit_ns; P.stall_once = h->stall_once;

  DrawParams Q = {};
  Q.a = G.a; Q.b = G.b; Q.p = G.p; Q.w = G.w;
  Q.vw = h->ws.partial; Q.sparsity = h->ws.partial + M * M; Q.status = h->ws.status;
  Q.N = d.N; Q.T = d.T; Q.M = M; Q.passes = passes; Q.rho = rho; Q.nu = nu; Q.s_lo = s_lo; Q.s_hi = s_hi; Q.seed = seed;

  cudaStream_t side = h->side_stream;
  for (int i0 = 0; i0 < M; i0 += most) {
    const int batches = M - i0 < most ? M - i0 : most;
    ProbeMaps maps;
    for (int g = 0; g < batches; ++g) {
      G.dY[g] = (const __nv_bfloat16*)dY[i0 + g]; G.X[g] = (const __nv_bfloat16*)X[i0 + g];
      if (!datum_map(&maps.a[g], sub > 0 ? (const void*)(G.sub + (size_t)g * R * sub) : dY[i0 + g], d_out, d.T, d.N) ||
          !datum_map(&maps.b[g], X[i0 + g], d.d_in, d.T, d.N))
        return cudaErrorInvalidValue;
    }
    if (i0 > 0) PROBE_CUDA(cudaStreamWaitEvent(st, h->ev_join, 0));       // Eq. 3 of the group before reads its scratch
    long blocks = (2l * R * batches + 7) / 8;
    if (blocks > (1l << 20)) blocks = 1l << 20;
    if (sub > 0) probe_norms_kernel<true><<<(unsigned)blocks, 256, 0, st>>>(G, batches, R, d.d_out, d.d_in, h->sub_rows, sub);
    else probe_norms_kernel<false><<<(unsigned)blocks, 256, 0, st>>>(G, batches, R, d.d_out, d.d_in, nullptr, 0);
    PROBE_CUDA(cudaGetLastError());
    Q.first_batch = i0;
    const dim3 draw_grid((unsigned)(PD * passes + 1), (unsigned)batches);
    const dim3 threads(DRAW_THREADS);
    PROBE_CUDA(d.N <= 32    ? launch_after(probe_draw_kernel<1>, draw_grid, threads, 0, st, Q)
               : d.N <= 64  ? launch_after(probe_draw_kernel<2>, draw_grid, threads, 0, st, Q)
               : d.N <= 128 ? launch_after(probe_draw_kernel<4>, draw_grid, threads, 0, st, Q)
               : d.N <= 256 ? launch_after(probe_draw_kernel<8>, draw_grid, threads, 0, st, Q)
                            : launch_after(probe_draw_kernel<32>, draw_grid, threads, 0, st, Q));
    PROBE_CUDA(cudaEventRecord(h->ev_fork, st));
    PROBE_CUDA(cudaStreamWaitEvent(side, h->ev_fork, 0));
    PROBE_CUDA(launch_maybe_after(false, probe_vw_kernel, dim3((unsigned)M, (unsigned)batches), dim3(SAMPLER_THREADS), vw_smem, side, Q));
    PROBE_CUDA(cudaEventRecord(h->ev_join, side));
    h->launches += 3;
    P.first_batch = i0; P.batches = batches;
    for (P.pass = 0; P.pass < passes; ++P.pass) {
      P.fresh = i0 == 0 && P.pass == 0;
      PROBE_CUDA(M == 2         ? run_probe<2, true>(h, maps, P, ctas, st)
                 : P.pass == 0 ? run_probe<PD, true>(h, maps, P, ctas, st)
                                : run_probe<PD, false>(h, maps, P, ctas, st));
    }
  }
  PROBE_CUDA(cudaStreamWaitEvent(st, h->ev_join, 0));
  probe_final_kernel<<<1, 1024, 0, st>>>(P.pact, P.ps, sums, Q.vw, Q.sparsity, M, scale, V_s, V_act, V_w, p_lo, p_hi);
  h->launches += 1;
#undef PROBE_CUDA
  return cudaGetLastError();
}

}  // namespace vcas
