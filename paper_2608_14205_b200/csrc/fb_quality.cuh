// Prediction-quality metrics of the evaluation (not part of the per-layer hot path):
// the mean over tokens of the cosine similarity between two row-major matrices (hidden
// states before / after the residual update, or the two router invocations' logits), and
// the number of final top-k assignments the early pass recovered (hit rate numerator).
// Sums are formed in a fixed order, in double precision, so results are reproducible.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/freebalance.h"
#include "fb_ptx.cuh"

namespace fb {

constexpr int kCosineWarpsPerBlock = 2;      // small blocks: a finished row's place is taken at once
constexpr int kMeanThreads = 1024;
constexpr int kCosineSteps = 4;              // steps of a bf16 row whose loads are in flight
constexpr int kCosineBlocksPerSm = 12;       // for 80 registers a thread, which the four steps need

__device__ __forceinline__ double load_as_double(const __nv_bfloat16* p, long long i) {
  return static_cast<double>(__bfloat162float(p[i]));
}
__device__ __forceinline__ double load_as_double(const float* p, long long i) { return static_cast<double>(p[i]); }

// A bf16 value (the upper half of a 32-bit word with a zero lower half) times 2^-896 as a double, by moving its
// bits: 8 exponent bits under a double's 11-bit exponent.  Exact, zeros and subnormals included (a double's
// subnormals lie 896 binades below).  Infinities and NaNs become finite values: the caller looks for them itself.
__device__ __forceinline__ double bf16_scaled(uint32_t u) {
  return __hiloint2double(static_cast<int>(static_cast<uint32_t>(static_cast<int32_t>(u) >> 3) & 0x8fffffffu), 0);
}

// A lane's part of the sums a.b, a.a and b.b of two rows.  Rows whose start and length allow it are read 16 bytes per
// lane and step (kVec elements); otherwise lane l takes elements l, l + 32, ...  Either way a lane adds its elements
// in ascending order, exact products into doubles.
struct CosineSums {
  double dot = 0.0, na = 0.0, nb = 0.0;
  __device__ __forceinline__ void add(double x, double y) { dot += x * y; na += x * x; nb += y * y; }
};
template <class Tin>
__device__ __forceinline__ CosineSums row_sums(const Tin* __restrict__ a, const Tin* __restrict__ b, long long row, int n, int lane) {
  constexpr int kVec = 16 / static_cast<int>(sizeof(Tin)), kStep = 32 * kVec;
  const long long base = row * n;
  CosineSums s;
  const bool wide = n % kVec == 0 && reinterpret_cast<uintptr_t>(a) % 16 == 0 && reinterpret_cast<uintptr_t>(b) % 16 == 0;
  if constexpr (sizeof(Tin) == 2) {
    if (wide) {
      // Four steps' loads in flight (the latency of the loads is what a row waits for).  Conversions to double run
      // at a quarter of the rate of double arithmetic, and two per element kept their unit busy for half of the
      // time: a's elements are scaled by bit moves instead, which makes the sums dot 2^126, na 2^-770 and nb,
      // scaled back exactly below - the same bits as with two conversions.
      __nv_bfloat162 special = __float2bfloat162_rn(0.0f);      // NaN once a has an infinity or a NaN (times 0)
      for (int j0 = 0; j0 < n; j0 += kCosineSteps * kStep) {
        uint4 qa[kCosineSteps], qb[kCosineSteps];
#pragma unroll
        for (int q = 0; q < kCosineSteps; ++q) {
          const int j = j0 + q * kStep + lane * kVec;
          qa[q] = j < n ? *reinterpret_cast<const uint4*>(a + base + j) : make_uint4(0, 0, 0, 0);
          qb[q] = j < n ? *reinterpret_cast<const uint4*>(b + base + j) : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int q = 0; q < kCosineSteps; ++q) {
          if (j0 + q * kStep >= n) break;
          const uint32_t wa[4] = {qa[q].x, qa[q].y, qa[q].z, qa[q].w}, wb[4] = {qb[q].x, qb[q].y, qb[q].z, qb[q].w};
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            special = __hfma2(*reinterpret_cast<const __nv_bfloat162*>(&wa[t]), __float2bfloat162_rn(0.0f), special);
#pragma unroll
            for (int h = 0; h < 2; ++h) {                       // low half = the earlier element
              const double x = bf16_scaled(h ? wa[t] & 0xffff0000u : wa[t] << 16), up = x * 0x1p1022;
              const double y = static_cast<double>(__uint_as_float(h ? wb[t] & 0xffff0000u : wb[t] << 16));
              s.dot += up * y; s.na += x * up; s.nb += y * y;
            }
          }
        }
      }
      if (!__any_sync(0xffffffffu, __hisnan(special.x) || __hisnan(special.y))) {
        s.dot *= 0x1p-126; s.na *= 0x1p770;
        return s;
      }
      s = CosineSums();                                         // once more, with conversions
    }
  } else if (wide) {
    for (int j = lane * kVec; j < n; j += kStep) {
      const float4 x = *reinterpret_cast<const float4*>(a + base + j), y = *reinterpret_cast<const float4*>(b + base + j);
      s.add(x.x, y.x); s.add(x.y, y.y); s.add(x.z, y.z); s.add(x.w, y.w);
    }
    return s;
  }
  const int per = wide ? kVec : 1;
  for (int j = lane * per; j < n; j += 32 * per)
    for (int t = 0; t < per; ++t) s.add(load_as_double(a, base + j + t), load_as_double(b, base + j + t));
  return s;
}

// The three partial sums are combined by a butterfly, which gives every lane the same total.
__device__ __forceinline__ double cosine_of(double dot, double na, double nb) {
  return (na > 0.0 && nb > 0.0) ? dot / (sqrt(na) * sqrt(nb)) : 0.0;
}
__device__ __forceinline__ double row_cosine(CosineSums s) {
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    s.dot += __shfl_xor_sync(0xffffffffu, s.dot, off);
    s.na += __shfl_xor_sync(0xffffffffu, s.na, off);
    s.nb += __shfl_xor_sync(0xffffffffu, s.nb, off);
  }
  return cosine_of(s.dot, s.na, s.nb);
}
// Two rows' cosines at once, with the same additions: where a butterfly step would form a value twice, half of the
// lanes go on with another sum instead (10 exchanges instead of 30, one square root and division sequence instead
// of two).  Lane 0 returns the first row's, lane 16 the second's.
__device__ __forceinline__ double exchange_add(double keep_low, double keep_high, int lane, int off) {
  const bool high = (lane & off) != 0;
  return (high ? keep_high : keep_low) + __shfl_xor_sync(0xffffffffu, high ? keep_low : keep_high, off);
}
__device__ __forceinline__ double row_cosines(const CosineSums& s, const CosineSums& t, int lane) {
  const double dot = exchange_add(s.dot, t.dot, lane, 16), na = exchange_add(s.na, t.na, lane, 16);
  double nb = exchange_add(s.nb, t.nb, lane, 16);
  const double dot_na = exchange_add(dot, na, lane, 8);         // lanes with bit 3: na
  nb += __shfl_xor_sync(0xffffffffu, nb, 8);
  double v = exchange_add(dot_na, nb, lane, 4);                 // lanes with bit 2: nb
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  const double n1 = __shfl_sync(0xffffffffu, v, (lane & 16) | 8), n2 = __shfl_sync(0xffffffffu, v, (lane & 16) | 4);
  return cosine_of(v, n1, n2);
}

// One warp per row.
template <class Tin>
__global__ void __launch_bounds__(32 * kCosineWarpsPerBlock, kCosineBlocksPerSm)
fb_row_cosine_kernel(const Tin* __restrict__ a, const Tin* __restrict__ b, long long rows, int n,
                     double* __restrict__ row_cos) {
  const long long row = static_cast<long long>(blockIdx.x) * kCosineWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  pdl_launch_dependents();
  pdl_wait();
  if (row >= rows) return;
  const double c = row_cosine(row_sums(a, b, row, n, lane));
  if (lane == 0) row_cos[row] = c;
}

// The three quality figures of a step, row by row, in one launch: the hidden-state cosine, the logit cosine
// and the number of recovered assignments into rows[0 .. T), [T .. 2 T), [2 T .. 3 T).  Bound by the reads of the
// hidden states and, for short rows, by a warp's chain of loads and exchanges.  With the sums kernel behind it,
// [T, d, E] = 8192 x 2048 x 128: 20.4 -> 18.0 us; 4096 x 4096 x 8: 25.2 -> 16.7; 1733 x 7168 x 256: 32.9 -> 19.0;
// 16384 x 7168 x 256: 93.2 -> 83.8 (5.8 TB/s), against eight warps per block, one step's loads in flight, two
// conversions per element and a reduction per sum.  Two steps in flight: 18.1, 17.8, 23.0 and 87.1 us.
struct QualityParams {
  const __nv_bfloat16 *h_prev, *h;       // [T][d]
  const float *z_early, *z;              // [T][E]
  const int32_t *ids_early, *ids;        // [T][k]
  long long T;
  int32_t d, E, k;
  double* rows;                          // [3][T]
  double* out;                           // [3]: mean, mean, sum
};
__global__ void __launch_bounds__(32 * kCosineWarpsPerBlock, kCosineBlocksPerSm)
fb_quality_rows_kernel(const __grid_constant__ QualityParams p) {
  const long long row = static_cast<long long>(blockIdx.x) * kCosineWarpsPerBlock + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  pdl_launch_dependents();
  pdl_wait();
  if (row >= p.T) return;
  const int32_t mine = lane < p.k ? p.ids[row * p.k + lane] : INT32_MAX;
  const int32_t early = lane < p.k ? p.ids_early[row * p.k + lane] : INT32_MIN;
  uint32_t hits = 0;
#pragma unroll
  for (int y = 0; y < FB_MAX_TOPK; ++y) hits += __popc(__ballot_sync(0xffffffffu, mine == __shfl_sync(0xffffffffu, early, y)));
  const CosineSums logits = row_sums(p.z_early, p.z, row, p.E, lane);
  const double c = row_cosines(row_sums(p.h_prev, p.h, row, p.d, lane), logits, lane);
  if ((lane & 15) == 0) p.rows[lane == 0 ? row : p.T + row] = c;
  if (lane == 1) p.rows[2 * p.T + row] = static_cast<double>(hits);
}
// Sums of the three columns by one cluster, in a fixed order.
constexpr int kQualityBlocks = 8;
__global__ void __cluster_dims__(kQualityBlocks, 1, 1) __launch_bounds__(kMeanThreads)
fb_quality_sums_kernel(const __grid_constant__ QualityParams p) {
  __shared__ double part[3][kMeanThreads / 32];
  __shared__ double sums[3];
  const int t = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  double s[3] = {0.0, 0.0, 0.0};
#pragma unroll 4
  for (long long i = static_cast<long long>(cluster_ctarank()) * kMeanThreads + t; i < p.T; i += kQualityBlocks * kMeanThreads) {
#pragma unroll
    for (int c = 0; c < 3; ++c) s[c] += __ldcg(p.rows + c * p.T + i);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], off);
    if ((t & 31) == 0) part[c][t >> 5] = s[c];
  }
  __syncthreads();
  if (t < 96) {
    const int c = t >> 5;
    double v = part[c][t & 31];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    if ((t & 31) == 0) sums[c] = v;
  }
  cluster_arrive();
  cluster_wait();
  if (cluster_ctarank() == 0 && t < 3) {
    double v = 0.0;
    for (uint32_t r = 0; r < kQualityBlocks; ++r) v += ld_cluster_double(map_to_cta(smem_u32(&sums[t]), r));
    p.out[t] = p.T > 0 && t < 2 ? v / static_cast<double>(p.T) : v;
  }
  cluster_arrive();
  cluster_wait();
}

// Mean of v[0 .. count) by one block: strided partial sums with eight loads in flight, then warp
// butterflies; the order of the additions is fixed.
__global__ void __launch_bounds__(kMeanThreads)
fb_mean_kernel(const double* __restrict__ v, long long count, double* __restrict__ out) {
  __shared__ double part[kMeanThreads / 32];
  static_assert(kMeanThreads == 1024, "one warp adds the warps' sums");
  pdl_launch_dependents();
  pdl_wait();
  double s = 0.0;
#pragma unroll 8
  for (long long i = threadIdx.x; i < count; i += kMeanThreads) s += __ldcg(v + i);
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = part[threadIdx.x];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (threadIdx.x == 0) *out = count > 0 ? s / static_cast<double>(count) : 0.0;
  }
}

// hits = sum over tokens i of |ids_a[i, :] intersect ids_b[i, :]| (ids within a token are distinct).
// One cluster: its blocks' sums meet in the first one's shared memory, so nothing has to be cleared
// before (a memset between the kernels keeps them from overlapping).
constexpr int kHitsBlocks = 8;
constexpr int kHitsThreads = 1024;
__global__ void __cluster_dims__(kHitsBlocks, 1, 1) __launch_bounds__(kHitsThreads)
fb_topk_hits_kernel(const int32_t* __restrict__ ids_a, const int32_t* __restrict__ ids_b, int T, int k,
                    uint32_t* __restrict__ hits) {
  __shared__ uint32_t block_sum, cluster_sum;
  if (threadIdx.x == 0) { block_sum = 0; cluster_sum = 0; }
  __syncthreads();
  cluster_arrive();
  pdl_launch_dependents();
  pdl_wait();
  uint32_t mine = 0;
  for (long long i = static_cast<long long>(blockIdx.x) * kHitsThreads + threadIdx.x; i < T; i += kHitsBlocks * kHitsThreads) {
    int32_t a[FB_MAX_TOPK];
#pragma unroll
    for (int y = 0; y < FB_MAX_TOPK; ++y) a[y] = y < k ? ids_a[i * k + y] : INT32_MIN;
#pragma unroll
    for (int x = 0; x < FB_MAX_TOPK; ++x) {
      const int32_t e = x < k ? ids_b[i * k + x] : INT32_MAX;
#pragma unroll
      for (int y = 0; y < FB_MAX_TOPK; ++y) mine += a[y] == e ? 1u : 0u;
    }
  }
  mine = __reduce_add_sync(0xffffffffu, mine);
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&block_sum, mine);
  __syncthreads();
  cluster_wait();
  if (threadIdx.x == 0) red_add_cluster(map_to_cta(smem_u32(&cluster_sum), 0u), block_sum);
  cluster_arrive();
  cluster_wait();
  if (cluster_ctarank() == 0 && threadIdx.x == 0) *hits = cluster_sum;
}

// SM clock probe: one thread records (global nanosecond timer, SM cycle counter) pairs, `n` of
// them about `period_ns` apart, and ends by itself.  The ratio of the differences between two
// samples is the clock the SMs actually ran at in between - what a kernel sees under load,
// which the driver's clock query (a few samples per second) cannot resolve.
__global__ void __launch_bounds__(32, 1)
fb_clock_probe_kernel(unsigned long long* __restrict__ samples, int n, unsigned period_ns) {
  if (threadIdx.x != 0) return;
  for (int i = 0; i < n; ++i) {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    samples[2 * i] = t;
    samples[2 * i + 1] = static_cast<unsigned long long>(clock64());
    if (period_ns) __nanosleep(period_ns);
  }
}

// Stand-in for an attention kernel in overlap experiments: compute-bound (register FMAs only,
// no memory traffic but one store per thread at the end), one block per SM by its shared-memory
// footprint, on exactly as many SMs as the grid has blocks.  Other streams' kernels share the
// remaining SMs, and memory-bound blocks with a small footprint can sit beside a stand-in block.
constexpr int kStandinThreads = 1024;
constexpr int kStandinSmemBytes = 120 * 1024;          // two such blocks do not fit one SM
__global__ void __launch_bounds__(kStandinThreads, 1)
fb_standin_attention_kernel(float* __restrict__ out, int iters) {
  extern __shared__ float standin_smem[];
  float a0 = threadIdx.x * 1e-3f, a1 = a0 + 1.0f, a2 = a0 + 2.0f, a3 = a0 + 3.0f;
  const float m = 1.0000001f, c = 1e-7f;
  for (int i = 0; i < iters; ++i) {
#pragma unroll 8
    for (int u = 0; u < 8; ++u) {
      a0 = fmaf(a0, m, c); a1 = fmaf(a1, m, c); a2 = fmaf(a2, m, c); a3 = fmaf(a3, m, c);
    }
  }
  if (threadIdx.x == 0) standin_smem[0] = a0;          // touches the allocation so that it is kept
  out[static_cast<size_t>(blockIdx.x) * kStandinThreads + threadIdx.x] = a0 + a1 + a2 + a3;
}

}  // namespace fb
