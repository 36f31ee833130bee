// FP32 Schur blocks and off-diagonal preconditioner blocks: the products of
// build.cu, entry by entry in the same order of sums (bit-identical), by CTAs
// that take chunks of consecutive blocks of one problem.
//
// The arithmetic is small (0.05 ms of FP32 on a batch of 4096 problems), as are
// the bytes (0.2 ms of HBM); a warp per knot spent its time on waiting for its
// own loads, on index divisions, and on five 32-bit shared-memory loads per four
// multiply-adds.  Here a chunk's blocks come to shared memory with coalesced
// loads from many threads at once, each thread forms a 4 x 4 tile of a result
// from two 128-bit loads per term, every thread of a CTA has a tile whatever nx
// is, and results leave through shared memory in consecutive order.  4096
// problems of N 16-128 and nx 4, 12, 14, 21: Schur blocks 0.72 to 0.43 ms, off-
// diagonal blocks 0.53 to 0.39 ms, the whole build 2.33 to 1.92 ms.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace sspcg {
namespace {

__host__ __device__ __forceinline__ int tiles4(int x) { return (x + 3) >> 2; }

// acc[r][s] += u[r] v[s] for the four entries at u and v (16-byte aligned)
__device__ __forceinline__ void outer(float (&acc)[4][4], const float *u, const float *v) {
  const float4 a = *reinterpret_cast<const float4 *>(u), b = *reinterpret_cast<const float4 *>(v);
  const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int s = 0; s < 4; ++s) acc[r][s] = fmaf(av[r], bv[s], acc[r][s]);
}

// ---------------------------------------------------------------------------
// D_{b+1} = A_b Q_b^-1 A_b^T + B_b R_b^-1 B_b^T + Q_{b+1}^-1, E_b = -A_b Q_b^-1
// (D_0 = Q_0^-1).  In shared memory, term by term: u_l = column l of A_b Q_b^-1
// (then of B_b R_b^-1), v_l = column l of A_b (then of B_b).  Tiles of the upper
// triangle only, mirrored, so D is exactly symmetric.
// ---------------------------------------------------------------------------
constexpr int kSchurThreads = 256;
constexpr int kSchurFloats = 10240;  // 40 KB: five CTAs per SM

__host__ __device__ __forceinline__ int schur_chunk(int nx, int nu) {
  const int t = tiles4(nx), by_tiles = kSchurThreads / (t * (t + 1) / 2);
  const int by_smem = kSchurFloats / (2 * (nx + nu) * 4 * t);
  return by_tiles < by_smem ? by_tiles : by_smem;
}

__global__ void __launch_bounds__(kSchurThreads) schur_f32_kernel(ProbSet ps, ChunkSplit split,
                                                                  const float *__restrict__ A,
                                                                  const float *__restrict__ B,
                                                                  const float *__restrict__ qd,
                                                                  const float *__restrict__ rd, float *__restrict__ D,
                                                                  float *__restrict__ E) {
  __shared__ __align__(16) float sm[kSchurFloats];
  const int tid = threadIdx.x;
  const ProbDesc d = ps.get(blockIdx.x / split.per);
  const int N = d.N, nx = d.nx, nu = d.nu, nn = nx * nx, m = nx + nu, nt = tiles4(nx), ld = 4 * nt;
  const int ntl = nt * (nt + 1) / 2, per = split.per, C = chunk_length(schur_chunk(nx, nu), N, split.share);
  const Divisor by_nx(nx), by_nu(nu), by_ntl(ntl);
  const int part = blockIdx.x % per;
  if (part == 0) {
    float *D0 = D + d.odiag;
    for (int e = tid; e < nn; e += kSchurThreads) {
      const int i = by_nx.quotient(e);
      D0[e] = i == e - i * nx ? 1.0f / qd[d.oq + i] : 0.0f;
    }
  }
  for (int b0 = part * C; b0 < N; b0 += per * C) {
    const int nb = min(C, N - b0);
    float *su = sm, *sv = sm + nb * m * ld;
    const float *Ab = A + d.oA + (int64_t)b0 * nn, *Bb = B + d.oB + (int64_t)b0 * nx * nu;
    const float *qb = qd + d.oq + (int64_t)b0 * nx, *rb = rd + d.orr + (int64_t)b0 * nu;
    float *Eb = E + d.ooff + (int64_t)b0 * nn;
    for_values(Ab, nb * nn, tid, kSchurThreads, [&](int e, float a) {
      const int r = by_nx.quotient(e), l = e - r * nx, kk = by_nx.quotient(r), i = r - kk * nx;
      const float aq = a / __ldg(qb + kk * nx + l);
      const int o = (kk * m + l) * ld + i;
      su[o] = aq;
      sv[o] = a;
      Eb[e] = -aq;
    });
    for_values(Bb, nb * nx * nu, tid, kSchurThreads, [&](int e, float x) {
      const int r = by_nu.quotient(e), l = e - r * nu, kk = by_nx.quotient(r), i = r - kk * nx;
      const int o = (kk * m + nx + l) * ld + i;
      su[o] = x / __ldg(rb + kk * nu + l);
      sv[o] = x;
    });
    __syncthreads();
    // one tile per thread: nb * ntl <= kSchurThreads
    const int kk = by_ntl.quotient(tid);
    int ti = 0, tj = tid - kk * ntl;
    while (tj >= nt - ti) tj -= nt - ti, ++ti;
    tj += ti;
    float acc[4][4] = {};
    const bool in = kk < nb;
    if (in) {
      const float *u = su + kk * m * ld + 4 * ti, *v = sv + kk * m * ld + 4 * tj;
#pragma unroll 4
      for (int l = 0; l < m; ++l) outer(acc, u + l * ld, v + l * ld);
    }
    __syncthreads();  // u and v no longer read: the results take their place
    if (in) {
      float *o = sm + kk * nn;
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int i = 4 * ti + r, j = 4 * tj + s;
          if (i > j || j >= nx) continue;
          float x = acc[r][s];
          if (i == j) x += 1.0f / qb[(kk + 1) * nx + i];
          o[i * nx + j] = x;
          o[j * nx + i] = x;
        }
    }
    __syncthreads();
    float *Db = D + d.odiag + (int64_t)(b0 + 1) * nn;
    for (int e = tid; e < nb * nn; e += kSchurThreads) Db[e] = sm[e];
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// PE_b = -c PD_{b+1} E_b PD_b.  PD is exactly symmetric, so its rows serve as the
// columns that the first product needs; T = PD_{b+1} E_b is kept transposed for
// the second.
// ---------------------------------------------------------------------------
constexpr int kOffThreads = 256;
constexpr int kOffFloats = 11520;  // 45 KB: four to five CTAs per SM

__host__ __device__ __forceinline__ int off_chunk(int nx) {
  const int t = tiles4(nx), by_tiles = kOffThreads / (t * t), blk = nx * 4 * t;
  const int by_smem = (kOffFloats - blk) / (3 * blk);  // PD: one block more than there are products
  return by_tiles < by_smem ? by_tiles : by_smem;
}

__global__ void __launch_bounds__(kOffThreads, 4) precond_off_f32_kernel(ProbSet ps, ChunkSplit split, float c,
                                                                      const float *__restrict__ E,
                                                                      const float *__restrict__ PD,
                                                                      float *__restrict__ PE) {
  __shared__ __align__(16) float sm[kOffFloats];
  const int tid = threadIdx.x;
  const ProbDesc d = ps.get(blockIdx.x / split.per);
  const int N = d.N, nx = d.nx, nn = nx * nx, nt = tiles4(nx), ld = 4 * nt, blk = nx * ld, ntl = nt * nt;
  const int per = split.per, C = chunk_length(off_chunk(nx), N, split.share);
  const Divisor by_ntl(ntl), by_nt(nt);
  for (int b0 = (int)(blockIdx.x % per) * C; b0 < N; b0 += per * C) {
    const int nb = min(C, N - b0);
    float *sP = sm, *sE = sP + (nb + 1) * blk, *sT = sE + nb * blk;
    const float *Pb = PD + d.odiag + (int64_t)b0 * nn, *Eb = E + d.ooff + (int64_t)b0 * nn;
    stage_chunk(sP, Pb, (nb + 1) * nx, nx, ld, tid, kOffThreads);
    stage_chunk(sE, Eb, nb * nx, nx, ld, tid, kOffThreads);
    __syncthreads();
    // one tile per thread: nb * ntl <= kOffThreads
    const int kk = by_ntl.quotient(tid), tl = tid - kk * ntl, ti = by_nt.quotient(tl), tj = tl - ti * nt;
    const bool in = kk < nb;
    float acc[4][4] = {};
    if (in) {
      const float *u = sP + (kk + 1) * blk + 4 * ti, *v = sE + kk * blk + 4 * tj;
#pragma unroll 4
      for (int l = 0; l < nx; ++l) outer(acc, u + l * ld, v + l * ld);
      float *t = sT + kk * blk + 4 * ti;
#pragma unroll
      for (int s = 0; s < 4; ++s)
        if (4 * tj + s < nx)
          *reinterpret_cast<float4 *>(t + (4 * tj + s) * ld) = make_float4(acc[0][s], acc[1][s], acc[2][s], acc[3][s]);
    }
    __syncthreads();
    if (in) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s) acc[r][s] = 0.0f;
      const float *u = sT + kk * blk + 4 * ti, *v = sP + kk * blk + 4 * tj;
#pragma unroll 4
      for (int l = 0; l < nx; ++l) outer(acc, u + l * ld, v + l * ld);
      float *o = sE + kk * nn;  // E is no longer read
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int s = 0; s < 4; ++s)
          if (4 * ti + r < nx && 4 * tj + s < nx) o[(4 * ti + r) * nx + 4 * tj + s] = -c * acc[r][s];
    }
    __syncthreads();
    float *Ob = PE + d.ooff + (int64_t)b0 * nn;
    for (int e = tid; e < nb * nn; e += kOffThreads) Ob[e] = sE[e];
    __syncthreads();
  }
}

}  // namespace

// A CTA's barriers and index arithmetic take a microsecond that a few small blocks don't have: they stay with the warp
// per knot of build.cu.  Schur blocks up to 4,500 knots: 3.1 us for 3.7 (nx 2, N 8 alone) and 4.3 for 4.8 (nx 2, 64
// problems of N 64), but 128 of N 40, nx 4 5.2 by chunks for 6.2, one of N 8, nx 12 4.8 for 6.2.  Off-diagonal blocks up
// to 8,000, us with the inverses: nx 2, N 64 alone 8.4 for 10.4, nx 3, 128 of N 40 12.5 for 13.9, 512 of N 20 14.5 either
// way.
bool few_small_knots(int64_t total, int max_nx, int max_nu) { return total <= 4500 && max_nx <= 8 && max_nu <= 8; }
bool few_small_offs(int64_t total, int max_nx) { return total <= 8000 && max_nx <= 8; }

cudaError_t launch_schur_f32(const ProbSet &ps, const int2 *refs, int64_t total_knots, int max_N, int max_nx, int max_nu,
                             const float *A, const float *B, const float *qd, const float *rd, float *D, float *E,
                             cudaStream_t st, int sms) {
  if (ps.nprob == 0) return cudaSuccess;
  if (few_small_knots(total_knots, max_nx, max_nu))
    return launch_schur_build<float>(ps, refs, total_knots, A, B, qd, rd, D, E, st, sms, std::max(max_nx, max_nu));
  const ChunkSplit split = chunk_split(ps.nprob, sms, max_N, schur_chunk(max_nx, max_nu), 3);
  schur_f32_kernel<<<(unsigned)ps.nprob * split.per, kSchurThreads, 0, st>>>(ps, split, A, B, qd, rd, D, E);
  return cudaGetLastError();
}

cudaError_t launch_precond_off_f32(const ProbSet &ps, const int2 *refs, int64_t total_off, int max_N, int max_nx,
                                   int kind, const float *E, const float *PD, float *PE, cudaStream_t st, int sms,
                                   int64_t off_elems) {
  if (off_elems == 0 || max_N == 0) return cudaSuccess;
  if (kind == 2 || kind == 3)  // block-Jacobi, Jacobi: no off-diagonal blocks
    return cudaMemsetAsync(PE, 0, sizeof(float) * off_elems, st);
  if (few_small_offs(total_off, max_nx))
    return launch_precond_off<float>(ps, refs, total_off, kind, E, PD, PE, st, sms, off_elems, max_nx);
  const ChunkSplit split = chunk_split(ps.nprob, sms, max_N, off_chunk(max_nx), 3);
  precond_off_f32_kernel<<<(unsigned)ps.nprob * split.per, kOffThreads, 0, st>>>(ps, split, kind == 0 ? 1.0f : 0.5f, E,
                                                                                 PD, PE);
  return cudaGetLastError();
}

}  // namespace sspcg
