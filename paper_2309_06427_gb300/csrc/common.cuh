// Shared device-side definitions of the sspcg CUDA library (sm_103a).
#pragma once

#include <atomic>
#include <cstdint>
#include <cuda_runtime.h>

namespace sspcg {

constexpr int kMaxNx = 28;

// Per-problem solve outcome codes (same values as the SSPCG_SOLVE_* enum of sspcg.h).
enum SolveCode : int { kOk = 0, kMaxIter = 1, kBreakdown = 2, kNotSpd = 3, kNonFinite = 4 };

// Packed-batch descriptor of one problem: shape and float offsets into each
// packed array kind (see SSPCG_ARRAY_* in sspcg.h).
struct ProbDesc {
  int32_t N, nx, nu, id;  // id: index of the problem in the caller's per-problem output arrays
  int64_t oA, oB, oq, orr, odiag, ooff, ovec;
};

// Problem set of a launch: either a device descriptor array (batched) or a
// single descriptor passed by value (single-problem calls; no device memory).
struct ProbSet {
  const ProbDesc *desc;  // device array of nprob descriptors, or nullptr
  ProbDesc single;       // used when desc == nullptr (problem 0)
  int32_t nprob;
  __device__ __forceinline__ ProbDesc get(int p) const { return desc ? desc[p] : single; }
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// Double-float ("float-float") arithmetic: a value is hi + lo with |lo| <=
// ulp(hi)/2.  Error-free transformations after Knuth (TwoSum) and Dekker
// (Fast2Sum); the exact product uses one fused multiply-add.  About 48
// significant bits from FP32 units, which on this GPU run at 64x the FP64
// rate.
// ---------------------------------------------------------------------------
struct df {
  float hi, lo;
};

__device__ __forceinline__ df two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}

__device__ __forceinline__ df fast_two_sum(float a, float b) {  // requires |a| >= |b| or a == 0
  float s = __fadd_rn(a, b);
  float e = __fsub_rn(b, __fsub_rn(s, a));
  return {s, e};
}

__device__ __forceinline__ df df_add(df a, df b) {
  df s = two_sum(a.hi, b.hi);
  float e = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  return fast_two_sum(s.hi, e);
}

// acc += a * b with the product formed exactly.
__device__ __forceinline__ df df_fma(df acc, float a, float b) {
  float p = __fmul_rn(a, b);
  float pe = __fmaf_rn(a, b, -p);
  df s = two_sum(acc.hi, p);
  float e = __fadd_rn(s.lo, __fadd_rn(acc.lo, pe));
  return fast_two_sum(s.hi, e);
}

__device__ __forceinline__ df df_shfl_xor(df v, int o) {
  return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

__device__ __forceinline__ df warp_sum(df v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = df_add(v, df_shfl_xor(v, o));
  return v;
}

__device__ __forceinline__ double df_to_double(df v) { return (double)v.hi + (double)v.lo; }

// Products of double-float values: the exact product of the high parts (one
// FMA gives its error) plus the cross terms; the lo * lo term is below the
// format's precision.
__device__ __forceinline__ df df_mul(df a, df b) {
  float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return fast_two_sum(p, e);
}

// c + a * b for double-float a, b, c.
__device__ __forceinline__ df df_fma3(df a, df b, df c) {
  float p = __fmul_rn(a.hi, b.hi);
  float pe = __fmaf_rn(a.hi, b.hi, -p);
  pe = __fmaf_rn(a.hi, b.lo, pe);
  pe = __fmaf_rn(a.lo, b.hi, pe);
  df s = two_sum(c.hi, p);
  float e = __fadd_rn(s.lo, __fadd_rn(c.lo, pe));
  return fast_two_sum(s.hi, e);
}

__device__ __forceinline__ df df_neg(df a) { return {-a.hi, -a.lo}; }

// 1 / x: the FP32 reciprocal and one Newton step y + y (1 - x y) with the
// residual formed in double-float (about 46 bits).
__device__ __forceinline__ df df_rcp(df x) {
  const float y = __frcp_rn(x.hi);
  const df r = df_fma3(df_neg(x), df{y, 0.0f}, df{1.0f, 0.0f});  // 1 - x y
  return fast_two_sum(y, __fmul_rn(y, r.hi));
}

// sqrt(x), x > 0: the FP32 square root and one Newton step s + (x - s^2) / (2 s).
__device__ __forceinline__ df df_sqrt(df x) {
  const float s = __fsqrt_rn(x.hi);
  const df r = df_fma3(df{-s, 0.0f}, df{s, 0.0f}, x);  // x - s^2
  return fast_two_sum(s, __fdiv_rn(r.hi, __fmul_rn(2.0f, s)));
}

// Ceil-div helpers.
__host__ __device__ __forceinline__ int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }
__host__ __device__ __forceinline__ int64_t round_up(int64_t a, int64_t b) { return cdiv(a, b) * b; }

// Chunks of consecutive block rows of one problem, for kernels that give a thread one column of a chunk's [A_k B_k]
// (or one row of it): as many block rows as make kChunkItems columns.  kChunkFloats holds a chunk's blocks with odd
// row strides for every nx, nu <= 28 (the most is 7616, at nx = 28, nu = 4).
constexpr int kChunkItems = 256;
constexpr int kChunkFloats = 7616;
__host__ __device__ __forceinline__ int chunk_rows(int nx, int nu) {
  const int c = kChunkItems / (nx + nu);
  return c > 64 ? 64 : c;
}

// Chunks of the true residual (residual.cu), which keeps nx + nu doubles per block row beside the blocks, in
// kResFloats, for batches with some nu > nx: as above, but at least 128 rows where they fit, so that the half that works
// row by row has a warp for every quarter of the SM (N 64 to 512 alone: nx 4, nu 28 1.9 times as fast, nx 1, nu 28 3
// times).
constexpr int kResFloats = kChunkFloats + 2 * (kChunkItems + kMaxNx);
__host__ __device__ __forceinline__ int residual_rows(int nx, int nu) {
  const int fit = kResFloats / (nx * (nx | 1) + nx * (nu | 1) + 2 * (nx + nu)), few = (128 + nx - 1) / nx;
  const int c = chunk_rows(nx, nu), w = few < fit ? few : fit;
  return c > w ? c : w > 64 ? 64 : w;
}

// CTAs of a launch over chunks: ``per`` for every problem, which is cut into ``share`` chunks at least.
struct ChunkSplit {
  int per, share;
};

// The split of nprob problems of at most ``rows`` block rows; full: rows of a full chunk of the largest blocks; least:
// rows that a CTA is worth.  A CTA costs as much as some ten rows of small blocks, so problems are cut into shorter
// chunks only while all CTAs run at once, three to an SM: a lone problem goes to many CTAs (nx = 14, N = 103, build and
// solve: 681 to 677 us), 304 problems of 64 rows to one each.  (Seven CTAs to an SM are slower at 64 problems of 64 rows,
// one or two on few long problems.  Cutting without regard to what runs at once made the 304 problems' Schur blocks of
// nx = 4 take 30 us for 6, the right-hand side of 512 problems of 20 rows 11 us for 5.)  Longer problems get a CTA per
// full chunk, up to 56 CTAs per SM in all: the largest of a mixed batch of 4096 end it (two CTAs each, primal steps: 133
// us for 158), and CTAs that find no chunk cost the more the more problems are small.
inline ChunkSplit chunk_split(int64_t nprob, int sms, int rows, int full, int least) {
  if (rows < 1 || nprob < 1) return {1, 1};
  int64_t share = 3 * (int64_t)sms / nprob;
  if (share > cdiv(rows, least)) share = cdiv(rows, least);
  if (share < 1) share = 1;
  int64_t per = 56 * (int64_t)sms / nprob;
  if (per > cdiv(rows, full)) per = cdiv(rows, full);
  if (per < share) per = share;
  return {(int)per, (int)share};
}

// Rows per chunk of a problem.
__host__ __device__ __forceinline__ int chunk_length(int full, int rows, int share) {
  if (share < 2) return full;  // no division: short kernels notice it
  const int c = (rows + share - 1) / share;
  return c < 1 ? 1 : c < full ? c : full;
}

// Quotients by a divisor d <= 64 known at run time, for e < 2^20: the high word of e times ceil(2^32 / d), whose
// excess over e / d is below e d / 2^32 < 1 / d.
struct Divisor {
  uint32_t mul;  // 0: d = 1
  __device__ __forceinline__ explicit Divisor(int d) : mul(d > 1 ? 0xffffffffu / (uint32_t)d + 1u : 0u) {}
  __device__ __forceinline__ int quotient(int e) const { return mul ? (int)__umulhi((uint32_t)e, mul) : e; }
};

// f(e, src[e]) for e < n, consecutive threads on consecutive values, eight loads of a thread in flight at a time
// (chunks are short: with the loads one after the other, waiting for them is most of the time).
template <typename F>
__device__ __forceinline__ void for_values(const float *src, int n, int tid, int nthr, F &&f) {
  constexpr int U = 8;
  for (int e0 = tid; e0 < n; e0 += U * nthr) {
    float v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = e0 + u * nthr < n ? __ldg(src + e0 + u * nthr) : 0.0f;
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (e0 + u * nthr < n) f(e0 + u * nthr, v[u]);
  }
}

// ``rows`` dense rows of width w (global) into rows of stride ld (shared memory).
__device__ __forceinline__ void stage_chunk(float *dst, const float *src, int rows, int w, int ld, int tid, int nthr) {
  const Divisor by_w(w);
  for_values(src, rows * w, tid, nthr, [&](int e, float v) { dst[e + by_w.quotient(e) * (ld - w)] = v; });
}

// Find the problem owning global knot g: knot_start is an exclusive prefix
// of (N_i + 1) with nprob + 1 entries.
__device__ __forceinline__ int find_problem(const int64_t *knot_start, int nprob, int64_t g) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (knot_start[mid] <= g) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Host: set a kernel's largest dynamic shared memory once per device.  Bit d
// of ``done`` records device d; devices beyond 63 set it on every call.
template <typename Kern>
inline cudaError_t smem_attr_once(std::atomic<uint64_t> &done, Kern kernel, int bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev >= 0 && dev < 64 ? (uint64_t{1} << dev) : 0;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_acq_rel);
  return e;
}

}  // namespace sspcg
