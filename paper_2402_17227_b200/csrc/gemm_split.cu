// The two products of the sampled backward on the tensor cores with the precision of fp32 arithmetic, for fp32
// layers and for bf16 layers whose widths are not multiples of 64:
//   dX[rows of kept data] = (1/p_n) dY[rows] W                   (App. E; zero rows for dropped data)
//   dW = G_tilde^T X over the kept rows                           (Sec. 4.2)
// An fp32 operand is cut into three bf16 parts, x = x1 + x2 + x3 (split.cuh), once, by a pass of its own; the
// product is the sum of the part products down to 2^-18: x1y1, x1y2, x2y1, x2y2, x1y3, x3y1 (what is left out is below
// 2^-26 of |x||y|).  A bf16 operand is its own single part; the rescaled rows of dY that enter a sampled dW product are
// formed in fp32 and cut into three.
// tcgen05 accumulates with truncation: over a contraction of 3072 its sum was measured to drift by 3e-6, against 5e-7
// for a chain of fp32 FMAs.  Every stage of 32 (a single part: 64) terms therefore starts a fresh TMEM accumulator, takes
// the lower products first, while the sum is small, and the leading x1y1 last; the epilogue warps add the stages up in
// fp32 registers (round to nearest) while the next one runs: measured below 1e-7 at every length.
//
// Persistent CTAs, 128 x 256 tiles, possibly a slice of the contraction: warps 0-7 accumulate and write, warp 8 loads
// by TMA (every part of both operands is one stage), warp 9 issues the products.
#include <atomic>

#include "split.cuh"
#include "umma.cuh"

namespace vcas {
namespace {

constexpr int MODE_DX = 0, MODE_DW = 1;
constexpr int SPLIT_THREADS = 10 * 32;
constexpr int ACC_WARPS = 8;
constexpr int BN = 256;                      // tile columns
constexpr int MAX_SPLIT = 16;

// derivative of the erf-form GELU: Phi(x) + x phi(x)
__device__ __forceinline__ float gelu_prime_erf(float x) {
  const float Phi = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
  const float phi = 0.39894228040143268f * expf(-0.5f * x * x);
  return fmaf(x, phi, Phi);
}

template <int PA, int PB> struct SplitCfg {
  static constexpr int KS = PA + PB > 2 ? 32 : 64;             // terms of the contraction in a stage
  static constexpr int CHUNK = 64 * KS * 2;                    // 64 columns of an MN-major operand
  static constexpr int A_PART = BM * KS * 2, B_PART = BN * KS * 2;
  static constexpr int STAGE_BYTES = PA * A_PART + PB * B_PART;
  static constexpr int STAGES = 221184 / STAGE_BYTES;          // 3, 5 or 4 stages of 72, 40 or 48 KB
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*alignment slack*/ + 256 /*barriers*/;
};

struct SplitParams {
  const void* H;             // dX: optional GELU pre-activation [R, d_in]
  void* out;                 // dX [R, d_in] in the layer dtype; dW [d_out, d_in] fp32
  // dX: kept data and 1/p_n (nullptr: every datum is kept with scale 1)
  const int32_t* idxA; const int32_t* counts; const float* scaleA;
  const int32_t* cnt;        // dW: length of the contraction
  float* partial;            // [tile][slice][128][256] fp32 partial tiles when the contraction is cut into slices
  int slices, max_units;
  int32_t* status;
  unsigned long long wait_limit_ns;
  int stall_once;
  int N, T, d_in, d_out;
};

// Output tiles and slices, from the device-resident counts.  dX rows are those of the kept data in compact order (row c =
// token c % T of the (c / T)-th kept datum), so a tile may span several data.
struct Work { int rows, stages, ntiles, S, per, units; };
template <int MODE, int KS> __device__ __forceinline__ Work work_of(const SplitParams& P) {
  Work w;
  const int K = MODE == MODE_DX ? P.d_out : *P.cnt;
  w.rows = MODE == MODE_DX ? (P.idxA != nullptr ? P.counts[0] : P.N) * P.T : P.d_out;
  w.stages = (K + KS - 1) / KS;
  w.ntiles = (P.d_in + BN - 1) / BN;
  const int tiles = (w.rows + BM - 1) / BM * w.ntiles;
  w.S = P.slices;
  if ((long)tiles * w.S > P.max_units) w.S = P.max_units / tiles;      // more kept than expected: fewer slices
  if (w.S > w.stages) w.S = w.stages;
  if (w.S < 1) w.S = 1;
  w.per = (w.stages + w.S - 1) / w.S;
  w.units = tiles * w.S;
  return w;
}
__device__ __forceinline__ size_t dx_row(const SplitParams& P, int c, float& sc) {
  const int k = c / P.T;
  const int n = P.idxA != nullptr ? P.idxA[k] : k;
  sc = P.scaleA != nullptr ? P.scaleA[n] : 1.0f;
  return (size_t)n * P.T + (c - k * P.T);
}
// Eight consecutive columns of one output row: rescaled, times GELU' (GELU: there may be one), stored.
template <typename T, int MODE, bool GELU>
__device__ __forceinline__ void finish8(const SplitParams& P, size_t row, float sc, int col, float (&v)[8]) {
  const size_t o = row * (size_t)P.d_in + col;
  if (MODE == MODE_DW) { store8(reinterpret_cast<float*>(P.out) + o, v); return; }
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] *= sc;
  if (GELU && P.H != nullptr) {
    Vec8<T> h;
    h.load(reinterpret_cast<const T*>(P.H) + o);
    float x[8];
    h.get(x);
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] *= gelu_prime_erf(x[e]);
  }
  store8(reinterpret_cast<T*>(P.out) + o, v);
}

// Four columns of an fp32 output row.
template <int MODE, bool GELU>
__device__ __forceinline__ void finish4(const SplitParams& P, int row, float sc, int col, float (&v)[4]) {
  const size_t o = (size_t)row * P.d_in + col;
  if (MODE == MODE_DX) {
#pragma unroll
    for (int e = 0; e < 4; ++e) v[e] *= sc;
    if (GELU && P.H != nullptr) {
      const float4 h = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(P.H) + o));
      const float x[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] *= gelu_prime_erf(x[e]);
    }
  }
  *reinterpret_cast<float4*>(reinterpret_cast<float*>(P.out) + o) = make_float4(v[0], v[1], v[2], v[3]);
}

// Where columns 4 q .. 4 q + 3 of `row` are in a slice of a tile: eight rows of four columns fill a cache line.  The product's
// warps (32 rows, the same columns) and the adding ones (8 rows x 32 columns) both work on whole lines; in rows of 256 columns
// every store of the product met 32 (fp32 layer of 4096 rows, 768 -> 3072: 98 -> 88 us; bf16, 4950 rows, 776 -> 1000: 65 -> 58).
__device__ __forceinline__ size_t partial_at(int row, int q) { return (((size_t)(row / 8) * (BN / 4) + q) * 8 + row % 8) * 4; }

// GELU: an instance of its own.  The factor's code stands in the unrolled output loop 128 times, and jumping over it cost a
// tile more in instruction fetches than its products took: the output of a first 128 x 256 tile of fp32 was 17000 to 34000
// cycles, of a later one 12000, and is 7200 (fp32: 15834 rows, 368 -> 856 at ratio 0.3, 107.4 -> 101.9 us the call; dense, 9728 rows,
// 64 -> 944, 83.1 -> 79.5; bf16, 4950 rows, 776 -> 1000, 58.5 -> 57.8).
template <typename T, int MODE, int PA, int PB, bool GELU>
__global__ void __launch_bounds__(SPLIT_THREADS, 1)
split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, SplitParams P) {
  using C = SplitCfg<PA, PB>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(base + C::STAGES * C::STAGE_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* acc_full = empty + C::STAGES;      // [2] the accumulator of a stage is complete
  uint64_t* acc_empty = acc_full + 2;          // [2] ... has been read
  uint64_t* done = acc_empty + 2;              // see drain_products
  uint32_t* tmem_holder = (uint32_t*)(done + 1);
  volatile int* abort_flag = (int*)(tmem_holder + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < C::STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], ACC_WARPS); }
    mbar_init(done, 1);
    *abort_flag = 0;
    *reinterpret_cast<volatile unsigned long long*>(abort_flag + 5) = P.wait_limit_ns;     // read by mbar_wait
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
  }
  if (warp == 9) tmem_alloc(tmem_holder, 2 * BN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *(volatile uint32_t*)tmem_holder;
  pdl_wait();
  const Work W = work_of<MODE, C::KS>(P);

  if (warp == 8) {
    // ------------------------------------------------------------------------- TMA producer
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0, filled = 0;
      bool ok = true, stalled = false;
      for (int u = blockIdx.x; u < W.units && ok; u += gridDim.x) {
        const int tile = u / W.S, slice = u - tile * W.S;
        const int row0 = tile / W.ntiles * BM, col0 = tile % W.ntiles * BN;
        const int k1 = min(W.stages, (slice + 1) * W.per);
        for (int k = slice * W.per; k < k1; ++k) {
          ok = mbar_wait(&empty[stage], phase ^ 1u, abort_flag, P.status);
          if (!ok) break;
          uint8_t* sa = base + stage * C::STAGE_BYTES;
          uint8_t* sb = sa + PA * C::A_PART;
          if (P.stall_once != 0 && blockIdx.x == 0 && !stalled) {
            stalled = true;                    // nothing will ever arrive for this stage: a wait runs out
          } else {
            mbar_expect_tx(&full[stage], C::STAGE_BYTES);
            if (MODE == MODE_DX) {
#pragma unroll
              for (int p = 0; p < PA; ++p) tma_load_3d(sa + p * C::A_PART, &tmA, k * C::KS, row0, p, &full[stage]);
            } else {
#pragma unroll
              for (int j = 0; j < 2 * PA; ++j)
                tma_load_3d(sa + j * C::CHUNK, &tmA, row0 + (j & 1) * 64, k * C::KS, j >> 1, &full[stage]);
            }
#pragma unroll
            for (int j = 0; j < 4 * PB; ++j)
              tma_load_3d(sb + j * C::CHUNK, &tmB, col0 + (j & 3) * 64, k * C::KS, j >> 2, &full[stage]);
          }
          ++filled;
          if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      drain_loads(full, C::STAGES, stage, phase, filled, abort_flag, P.status);
    }
  } else if (warp == 9) {
    // --------------------------------------------------------------------------- MMA issuer
    if (elect_one()) {
      constexpr uint32_t idesc = make_idesc(BN, MODE == MODE_DW, true);
      // MN-major: 64-column chunks CHUNK apart, 8 k-rows 1 KB apart, 128-byte swizzle; K-major A: 128 rows of KS terms, 8
      // rows 16 KS bytes apart, 128-byte swizzle for KS = 64 and 64-byte swizzle for KS = 32
      constexpr uint64_t mn_major = ((uint64_t)(C::CHUNK >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
      constexpr uint64_t k_major = (1ull << 16) | ((uint64_t)(16 * C::KS >> 4) << 32) | (1ull << 46) | ((C::KS == 64 ? 2ull : 4ull) << 61);
      constexpr uint64_t a_bits = MODE == MODE_DW ? mn_major : k_major;
      constexpr uint32_t a_step = MODE == MODE_DW ? (UMMA_K * 128 >> 4) : (UMMA_K * 2 >> 4);
      constexpr uint32_t b_step = UMMA_K * 128 >> 4;
      int stage = 0; uint32_t phase = 0; uint32_t it = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < W.units && ok; u += gridDim.x) {
        const int slice = u % W.S;
        const int n = min(W.stages, (slice + 1) * W.per) - slice * W.per;
        for (int j = 0; j < n; ++j, ++it) {
          const uint32_t buf = it & 1u;
          ok = mbar_wait(&acc_empty[buf], ((it >> 1) & 1u) ^ 1u, abort_flag, P.status) &&
               mbar_wait(&full[stage], phase, abort_flag, P.status);
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(base + stage * C::STAGE_BYTES), sb = sa + PA * C::A_PART;
          const uint32_t d = tmem_base + buf * (uint32_t)BN;
          auto product = [&](int pa, int pb, bool fresh) {
            const uint64_t da = a_bits | ((sa + pa * C::A_PART) >> 4), db = mn_major | ((sb + pb * C::B_PART) >> 4);
#pragma unroll
            for (int k4 = 0; k4 < C::KS / UMMA_K; ++k4)
              umma_bf16(d, da + (uint64_t)(k4 * a_step), db + (uint64_t)(k4 * b_step), idesc, fresh && k4 == 0 ? 0u : 1u);
          };
          if constexpr (PA == 3) product(2, 0, true);
          if constexpr (PB == 3) { product(0, 2, false); product(1, 1, false); }
          if constexpr (PA == 3) product(1, 0, false);
          if constexpr (PB == 3) product(0, 1, false);
          product(0, 0, PA == 1);
          umma_commit(&empty[stage]);
          umma_commit(&acc_full[buf]);
          if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
        }
      }
      drain_products(done, abort_flag, P.status);
    }
  } else {
    // ----------------------------------------------------------- fp32 accumulation and output
    const int eq = warp & 3, eg = warp >> 2;       // TMEM lane quarter, half of the columns
    constexpr int CW = BN / 2;
    const uint32_t taddr = tmem_base + ((uint32_t)(eq * 32) << 16) + (uint32_t)(eg * CW);
    uint32_t it = 0;
    bool ok = true;
    for (int u = blockIdx.x; u < W.units && ok; u += gridDim.x) {
      const int tile = u / W.S, slice = u - tile * W.S;
      const int n = min(W.stages, (slice + 1) * W.per) - slice * W.per;
      float acc[CW];
#pragma unroll
      for (int e = 0; e < CW; ++e) acc[e] = 0.f;
      for (int j = 0; j < n; ++j, ++it) {
        const uint32_t buf = it & 1u;
        // The lanes of a warp leave together.  No call here: it would put the sums held in registers into local memory.
        ok = __all_sync(0xffffffffu, mbar_wait_spin(&acc_full[buf], (it >> 1) & 1u, abort_flag, P.status));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int h = 0; h < CW / 32; ++h) {
          uint32_t v[32];
          tmem_ld32(taddr + buf * (uint32_t)BN + h * 32, v);
#pragma unroll
          for (int e = 0; e < 32; ++e) acc[h * 32 + e] += __uint_as_float(v[e]);
        }
        // one arrival per warp: the arrivals of all threads at one barrier are served one after the other
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[buf]);
      }
      const int row = eq * 32 + lane, r0 = tile / W.ntiles * BM + row;
      const int col0 = tile % W.ntiles * BN + eg * CW;
      constexpr bool EXCHANGE = sizeof(T) == 4;      // lanes of rows past the last take part
      if (!ok || (!EXCHANGE && r0 >= W.rows)) continue;
      if (W.S > 1) {
        if (EXCHANGE && r0 >= W.rows) continue;
        float* part = P.partial + (size_t)u * BM * BN + partial_at(row, eg * (CW / 4));
#pragma unroll
        for (int e = 0; e < CW; e += 4)
          *reinterpret_cast<float4*>(part + partial_at(0, e / 4)) = make_float4(acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
      } else if constexpr (!EXCHANGE) {
        float sc = 1.0f;
        const size_t r = MODE == MODE_DX ? dx_row(P, r0, sc) : (size_t)r0;
#pragma unroll
        for (int e = 0; e < CW; e += 8) {
          if (col0 + e >= P.d_in) break;
          float v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) v[i] = acc[e + i];
          finish8<T, MODE, GELU>(P, r, sc, col0 + e, v);
        }
      } else {
        // Every eight lanes exchange their rows' pieces of four columns, so that they store 128 bytes of one row at a time (a
        // row per lane met 32 cache lines a store: 4 x 64 rows, 256 -> 256, 35.4 -> 32.0 us).  Not in bf16 layers: rows
        // half as long, and the exchange cost more than the lines (4950 rows, 776 -> 1000: 61 -> 67 us).
        float sc = 1.0f;
        int target = -1;
        if (r0 < W.rows) target = MODE == MODE_DX ? (int)dx_row(P, r0, sc) : r0;
#pragma unroll
        for (int c = 0; c < CW; c += 32) {
          if (col0 + c >= P.d_in) break;
          float x[8][4];
#pragma unroll
          for (int i = 0; i < 32; ++i) x[i / 4][i % 4] = acc[c + i];
#pragma unroll
          for (int bit = 1; bit < 8; bit *= 2) {
            const bool up = (lane & bit) != 0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              if (i & bit) continue;
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float got = __shfl_xor_sync(0xffffffffu, up ? x[i][e] : x[i | bit][e], bit);
                if (up) x[i][e] = got; else x[i | bit][e] = got;
              }
            }
          }
          const int col = col0 + c + (lane & 7) * 4;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = __shfl_sync(0xffffffffu, target, (lane & 24) + i);
            const float f = __shfl_sync(0xffffffffu, sc, (lane & 24) + i);
            if (r >= 0 && col < P.d_in) finish4<MODE, GELU>(P, r, f, col, x[i]);
          }
        }
      }
    }
  }
  __syncwarp();
  pdl_trigger();       // by each warp as it leaves its loop; the loading warp, the first to be done, speaks for the CTA
  tc_fence_before();
  __syncthreads();
  if (warp == 9) { tc_fence_after(); tmem_dealloc(tmem_base, 2 * BN); }
}

// Adds the slices of every tile in order and writes the output: a warp takes 8 rows x 32 columns, eight columns a thread.
constexpr int ADD_THREADS = 256, ADD_ROWS = 8, ADD_COLS = 32;
template <typename T, int MODE, int KS>
__global__ void __launch_bounds__(ADD_THREADS) split_add_kernel(SplitParams P) {
  pdl_wait();
  pdl_trigger();
  const Work W = work_of<MODE, KS>(P);
  if (W.S == 1) return;                        // the product has written the output itself
  const int cblocks = (P.d_in + ADD_COLS - 1) / ADD_COLS;
  const int total = (W.rows + ADD_ROWS - 1) / ADD_ROWS * cblocks;
  const int lane = threadIdx.x & 31;
  for (int it = blockIdx.x * (ADD_THREADS / 32) + (threadIdx.x >> 5); it < total; it += gridDim.x * (ADD_THREADS / 32)) {
    const int rb = it / cblocks, row = rb * ADD_ROWS + lane % ADD_ROWS, col = (it - rb * cblocks) * ADD_COLS + lane / ADD_ROWS * 8;
    if (row >= W.rows || col >= P.d_in) continue;
    const int tile = row / BM * W.ntiles + col / BN;
    const float* part = P.partial + (size_t)tile * W.S * BM * BN + partial_at(row % BM, col % BN / 4);
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int s = 0; s < W.S; ++s) {
      const float4 x = __ldcg(reinterpret_cast<const float4*>(part + (size_t)s * BM * BN));
      const float4 y = __ldcg(reinterpret_cast<const float4*>(part + (size_t)s * BM * BN + partial_at(0, 1)));
      v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
      v[4] += y.x; v[5] += y.y; v[6] += y.z; v[7] += y.w;
    }
    float sc = 1.0f;
    const size_t r = MODE == MODE_DX ? dx_row(P, row, sc) : (size_t)row;
    finish8<T, MODE, true>(P, r, sc, col, v);
  }
}

// ------------------------------------------------------------------------------ operand parts
// One launch for what a product needs beforehand: the rows of dY of kept data, compact (all rows without a list), the
// whole of a second matrix, and zeros in the rows of dX that belong to dropped data.  HBM / L2 bound: a warp takes
// 256 elements of a row at a time, up to four such pieces in flight.
struct PrepParams {
  const void* Y; __nv_bfloat16* Yp; size_t y_stride;        // rows of dY, their parts (nullptr: not wanted)
  const void* M; __nv_bfloat16* Mp; size_t m_stride;        // whole matrix of m_rows x m_d, its parts (nullptr: none)
  void* dX;                                                 // zero rows (nullptr: none)
  const int32_t* idxA; const int32_t* dropA; const int32_t* counts;
  int N, T, d_in, d_out, m_rows, m_d;
};
constexpr int PREP_THREADS = 256, PREP_PIECES = 4, PREP_ELEMS = 256 * PREP_PIECES;
template <typename T, bool CUT>
__device__ __forceinline__ void prep_row(const T* src, __nv_bfloat16* dst, size_t stride, int d, int first, int lane) {
  Vec8<T> v[PREP_PIECES];
#pragma unroll
  for (int q = 0; q < PREP_PIECES; ++q) {
    const int c = first + q * 256 + lane * 8;
    if (c < d) v[q].load(src + c);
  }
#pragma unroll
  for (int q = 0; q < PREP_PIECES; ++q) {
    const int c = first + q * 256 + lane * 8;
    if (c >= d) break;
    if constexpr (CUT) {
      float f[8];
      v[q].get(f);
      store_parts3<true>(f, dst + c, stride);
    } else {
      *reinterpret_cast<uint4*>(dst + c) = v[q].v;
    }
  }
}
// EARLY: the matrix is cut before the wait for the kernel before, in an instance of its own: the others, whose code is short
// enough that more of it costs them 0.5 us, take it behind the rows, which the product needs first.
template <typename T, bool EARLY>
__global__ void __launch_bounds__(PREP_THREADS) prep_kernel(PrepParams P) {
  constexpr bool CUT = sizeof(T) == 4;
  const int lane = threadIdx.x & 31;
  const int yseg = (P.d_out + PREP_ELEMS - 1) / PREP_ELEMS, mseg = (P.m_d + PREP_ELEMS - 1) / PREP_ELEMS,
            zseg = (P.d_in + PREP_ELEMS - 1) / PREP_ELEMS;
  const int warps = gridDim.x * (PREP_THREADS / 32);
  const int all_m = P.M != nullptr ? P.m_rows * mseg : 0, n_m = EARLY ? 0 : all_m;
  int i = blockIdx.x * (PREP_THREADS / 32) + (threadIdx.x >> 5);
  auto cut_m = [&](int item) {
    const int r = item / mseg, first = (item - r * mseg) * PREP_ELEMS;
    prep_row<T, CUT>(reinterpret_cast<const T*>(P.M) + (size_t)r * P.m_d, P.Mp + (size_t)r * P.m_d, P.m_stride, P.m_d, first, lane);
  };
  if constexpr (EARLY) {
    pdl_trigger();
    for (; i < all_m; i += warps) cut_m(i);
    i -= all_m;
    pdl_wait();
  } else {
    pdl_wait();
    pdl_trigger();
  }
  const int cntA = P.idxA != nullptr ? P.counts[0] : P.N;
  const int n_y = P.Y != nullptr ? cntA * P.T * yseg : 0, n_z = P.dX != nullptr ? (P.N - cntA) * P.T * zseg : 0;
  for (; i < n_y + n_m + n_z; i += warps) {
    if (i < n_y) {
      const int c = i / yseg, first = (i - c * yseg) * PREP_ELEMS;
      const int k = c / P.T;
      const size_t r = (size_t)(P.idxA != nullptr ? P.idxA[k] : k) * P.T + (c - k * P.T);
      prep_row<T, CUT>(reinterpret_cast<const T*>(P.Y) + r * P.d_out, P.Yp + (size_t)c * P.d_out, P.y_stride, P.d_out, first, lane);
    } else if (!EARLY && i < n_y + n_m) {
      cut_m(i - n_y);
    } else {
      const int c = (i - n_y - n_m) / zseg, first = (i - n_y - n_m - c * zseg) * PREP_ELEMS;
      const int k = c / P.T;
      T* row = reinterpret_cast<T*>(P.dX) + ((size_t)P.dropA[k] * P.T + (c - k * P.T)) * P.d_in;
      const float z[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int e = first + lane * 8; e < min(first + PREP_ELEMS, P.d_in); e += 256) store8(row + e, z);
    }
  }
}

// ------------------------------------------------------------------------------------ host side
// Slices of the contraction from the expected number of tiles and k-blocks: the fewest microseconds of waves x
// (k-blocks per slice x cost + set-up) under the measured cost of a k-block.
int split_slices(const Handle* h, int sms, long tiles, int k, double kblock_us) {
  const int kb = k > BK ? (k + BK - 1) / BK : 1;
  int best = 1;
  double best_t = 1e30;
  for (int s = 1; s <= MAX_SPLIT && (s == 1 || kb / s >= 2); ++s) {
    if (tiles * s > h->max_units) break;
    const double waves = (double)((tiles * s + sms - 1) / sms);
    const double t = waves * ((double)((kb + s - 1) / s) * kblock_us + 1.5) + (s > 1 ? 3.5 + 0.3 * s : 0.0);
    if (t < best_t - 1e-9) { best_t = t; best = s; }
  }
  return best;
}

template <typename T, int MODE, int PA, int PB, bool GELU = false>
cudaError_t run_split(Handle* h, const CUtensorMap& a, const CUtensorMap& b, SplitParams& P, long exp_tiles, long max_tiles,
                      int k, long max_rows, bool programmatic, cudaStream_t st) {
  static std::atomic<bool> attr_set[64];
  using C = SplitCfg<PA, PB>;
  if (h->device < 0 || h->device >= 64) return cudaErrorInvalidDevice;
  if (!attr_set[h->device].load(std::memory_order_acquire)) {
    const cudaError_t e = cudaFuncSetAttribute(split_kernel<T, MODE, PA, PB, GELU>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    attr_set[h->device].store(true, std::memory_order_release);
  }
  // A sampled dX leaves one SM to SampleW, whose CTA does not fit beside one of these and would wait for a product to end
  // (fp32, 8192 rows, 512 -> 512: 67.5 and 66.8 us the call; 8192, 256 -> 1024: 54.6 and 54.1; 2048, 768 -> 3072: 78.2 and 77.7).  Also
  // where that makes a wave more: of 4700 rows, 148 tiles, dX alone takes 52 us on all SMs and 81 on one less (fp32, 1024 -> 1024;
  // bf16, 1000 -> 3000: 50 and 78), but the call 116 and 105 (145 and 136), as the dW branch is not held up.  With stage
  // profiling, where nothing runs beside it, too: the stages timed are the call's, bit for bit.
  const int sms = MODE == MODE_DX && P.counts != nullptr && h->num_sms > 1 ? h->num_sms - 1 : h->num_sms;
  P.slices = split_slices(h, sms, exp_tiles, k, PA * PB == 9 ? 1.7 : (PA * PB == 3 ? 0.9 : 0.55));
  long grid = max_tiles * P.slices;
  if (grid > sms) grid = sms;
  cudaError_t e = launch_maybe_after(programmatic, split_kernel<T, MODE, PA, PB, GELU>, dim3((unsigned)grid), dim3(SPLIT_THREADS),
                                     C::SMEM_BYTES, st, a, b, P);
  h->launches += 1;
  if (e == cudaSuccess && P.slices > 1) {
    const long pieces = (max_rows + ADD_ROWS - 1) / ADD_ROWS * ((P.d_in + ADD_COLS - 1) / ADD_COLS);
    long nb = (pieces + ADD_THREADS / 32 - 1) / (ADD_THREADS / 32);
    const long cap = (long)h->num_sms * 8;
    if (nb > cap) nb = cap;
    e = launch_after(split_add_kernel<T, MODE, C::KS>, dim3((unsigned)nb), dim3(ADD_THREADS), 0, st, P);
    h->launches += 1;
  }
  return e != cudaSuccess ? e : cudaGetLastError();
}

// [parts][rows][d] bf16, box of box_cols x box_rows of one part
bool part_map(CUtensorMap* m, const void* p, int d, long rows, int parts, size_t stride, uint32_t box_cols, uint32_t box_rows) {
  const uint64_t dims[3] = {(uint64_t)d, (uint64_t)rows, (uint64_t)parts};
  const uint64_t strides[2] = {(uint64_t)d * 2, (uint64_t)stride * 2};
  const uint32_t box[3] = {box_cols, box_rows, 1};
  return make_map(m, p, 3, dims, strides, box, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16,
                  box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B);
}

SplitParams split_params(Handle* h, int which) {
  SplitParams P = {};
  P.partial = h->ws.partial_tiles + (size_t)which * h->max_units * (BM * BN);
  P.max_units = h->max_units;
  P.status = h->ws.status;
  P.wait_limit_ns = h->wait_limit_ns;
  P.stall_once = h->stall_once;
  P.N = h->desc.N; P.T = h->desc.T; P.d_in = h->desc.d_in; P.d_out = h->desc.d_out;
  return P;
}

}  // namespace

int split_max_units(const vcas_layer_desc& d, int num_sms) {
  const long nt = (d.d_in + BN - 1) / BN;
  const long dx = ((long)d.N * d.T + BM - 1) / BM * nt, dw = (d.d_out + BM - 1) / BM * nt;
  const long most = (dx > dw ? dx : dw) * MAX_SPLIT;
  return (int)(most < num_sms ? most : num_sms);      // a cut contraction fills the SMs once
}

cudaError_t launch_split_prep(Handle* h, const void* dY, bool dense, const void* M, __nv_bfloat16* Mp, int m_rows, int m_d,
                              void* dX_zero, bool programmatic, bool early, cudaStream_t st) {
  const vcas_layer_desc& d = h->desc;
  PrepParams P = {};
  P.Y = dY; P.Yp = h->ws.packY; P.y_stride = (size_t)h->R_pad * d.d_out;
  P.M = M; P.Mp = Mp; P.m_rows = m_rows; P.m_d = M != nullptr ? m_d : 8; P.m_stride = (size_t)((m_rows + 63) / 64 * 64) * m_d;
  P.dX = dX_zero;
  if (!dense) { P.idxA = h->ws.idxA; P.dropA = h->ws.dropA; P.counts = h->ws.counts; }
  P.N = d.N; P.T = d.T; P.d_in = d.d_in; P.d_out = d.d_out;
  const long R = (long)d.N * d.T;
  auto pieces = [](int w) { return (long)(w + PREP_ELEMS - 1) / PREP_ELEMS; };
  long items = M != nullptr ? m_rows * pieces(m_d) : 0;
  if (dY != nullptr || dX_zero != nullptr) items += R * (dX_zero == nullptr || d.d_out > d.d_in ? pieces(d.d_out) : pieces(d.d_in));
  long blocks = (items + PREP_THREADS / 32 - 1) / (PREP_THREADS / 32);
  const long cap = (long)h->num_sms * 16;
  if (blocks > cap) blocks = cap;
  const dim3 grid((unsigned)blocks), threads(PREP_THREADS);
  const cudaError_t e = d.dtype != VCAS_DTYPE_F32 ? launch_maybe_after(programmatic, prep_kernel<__nv_bfloat16, false>, grid, threads, 0, st, P)
      : early                                     ? launch_maybe_after(programmatic, prep_kernel<float, true>, grid, threads, 0, st, P)
                                                  : launch_maybe_after(programmatic, prep_kernel<float, false>, grid, threads, 0, st, P);
  h->launches += 1;
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_split_dx(Handle* h, const void* dY, const void* W, bool dense, float rho_hint, const void* Hpre,
                            void* dX, cudaStream_t st) {
  const vcas_layer_desc& d = h->desc;
  const bool fp32 = d.dtype == VCAS_DTYPE_F32;
  SplitParams P = split_params(h, 0);
  P.H = Hpre; P.out = dX;
  if (!dense) { P.idxA = h->ws.idxA; P.counts = h->ws.counts; P.scaleA = h->ws.scaleA; }
  const long R = (long)d.N * d.T, nt = (d.d_in + BN - 1) / BN;
  const int parts = fp32 ? 3 : 1;
  const uint32_t ks = fp32 ? 32 : 64;
  CUtensorMap a, b;
  // a bf16 product of all rows reads dY where it is
  const void* A = fp32 || !dense ? (const void*)h->ws.packY : dY;
  if (!part_map(&a, A, d.d_out, dense ? R : h->R_pad, parts, (size_t)h->R_pad * d.d_out, ks, BM)) return cudaErrorInvalidValue;
  if (!part_map(&b, fp32 ? (const void*)h->ws.packW : W, d.d_in, d.d_out, parts, (size_t)((d.d_out + 63) / 64 * 64) * d.d_in, 64, ks))
    return cudaErrorInvalidValue;
  const long max_tiles = (R + BM - 1) / BM * nt;
  const long exp_rows = dense ? R : (long)((double)rho_hint * (double)R) + 1;
  const long exp_tiles = (exp_rows + BM - 1) / BM * nt;
  if (Hpre != nullptr) {
    if (fp32) return run_split<float, MODE_DX, 3, 3, true>(h, a, b, P, exp_tiles, max_tiles, d.d_out, R, true, st);
    return run_split<__nv_bfloat16, MODE_DX, 1, 1, true>(h, a, b, P, exp_tiles, max_tiles, d.d_out, R, !dense, st);
  }
  if (fp32) return run_split<float, MODE_DX, 3, 3>(h, a, b, P, exp_tiles, max_tiles, d.d_out, R, true, st);
  return run_split<__nv_bfloat16, MODE_DX, 1, 1>(h, a, b, P, exp_tiles, max_tiles, d.d_out, R, !dense, st);
}

cudaError_t launch_split_dw(Handle* h, const void* dY, const void* X, bool dense, int cnt_hint, float* dW, bool programmatic,
                            cudaStream_t st) {
  const vcas_layer_desc& d = h->desc;
  const bool fp32 = d.dtype == VCAS_DTYPE_F32;
  SplitParams P = split_params(h, 1);
  P.out = dW;
  P.cnt = dense ? h->ws.counts + 2 : h->ws.counts + 1;
  const long rows = dense ? (long)d.N * d.T : h->R_pad;     // rows of a dense operand past the last are zero-filled
  const void* A = !dense ? h->ws.packG : (fp32 ? (const void*)h->ws.packY : dY);
  const void* B = !dense || fp32 ? (const void*)h->ws.packX : X;
  const uint32_t ks = !dense || fp32 ? 32 : 64;
  CUtensorMap a, b;
  if (!part_map(&a, A, d.d_out, rows, !dense || fp32 ? 3 : 1, (size_t)h->R_pad * d.d_out, 64, ks)) return cudaErrorInvalidValue;
  if (!part_map(&b, B, d.d_in, rows, fp32 ? 3 : 1, (size_t)h->R_pad * d.d_in, 64, ks)) return cudaErrorInvalidValue;
  const long tiles = (long)((d.d_out + BM - 1) / BM) * ((d.d_in + BN - 1) / BN);
  if (fp32) return run_split<float, MODE_DW, 3, 3>(h, a, b, P, tiles, tiles, cnt_hint, d.d_out, programmatic, st);
  if (dense) return run_split<__nv_bfloat16, MODE_DW, 1, 1>(h, a, b, P, tiles, tiles, cnt_hint, d.d_out, programmatic, st);
  return run_split<__nv_bfloat16, MODE_DW, 3, 1>(h, a, b, P, tiles, tiles, cnt_hint, d.d_out, programmatic, st);
}

}  // namespace vcas
