// The two outer steps of the Schur-complement method around the PCG solve
// (Eq. schur, Sec. II-A): the right-hand side gamma = c - C G^-1 g from the
// constraint values c and the cost gradient g = (q_0, r_0, ..., q_N), and
// the primal step delta z = G^-1 (g - C^T lambda*) = G^-1 (g + C^T mu) from
// the library's solution mu = -lambda*.  With the constraint rows -x_0 and
// A_k x_k + B_k u_k - x_{k+1} and G = blockdiag(diag qd_k, diag rd_k):
//   gamma_0     = c_0 + q_0 / qd_0
//   gamma_{k+1} = c_{k+1} - A_k (q_k / qd_k) - B_k (r_k / rd_k) + q_{k+1} / qd_{k+1}
//   dx_k = (q_k - mu_k + A_k^T mu_{k+1}) / qd_k   (no A term at k = N)
//   du_k = (r_k + B_k^T mu_{k+1}) / rd_k
// A CTA takes chunks of consecutive block rows of one problem (common.cuh).
// Both kernels are bound by reading A and B once; a row of a block is read by
// one thread, so form_gamma brings the blocks to shared memory with coalesced
// loads first (a warp per knot with a row per lane touched 32 lines per load and
// left lanes past nx idle), and recover_step, which reads columns, reads them
// where they are.  Both steps with the true residual of residual.cu, 4096
// problems of N 20-100 and nx 4, 12, 14, 21: 2.47 ms before, 1.26 ms now.
#include <algorithm>

#include "../../include/sspcg.h"
#include "common.cuh"
#include "host.h"

namespace sspcg {
namespace {

constexpr int kKktThreads = 256;

// With ``per`` CTAs for each problem, CTA b takes chunks b % per, b % per + per, ... of problem b / per.
__global__ void __launch_bounds__(kKktThreads, 7)  // what the shared memory holds; five CTAs take a quarter longer
    form_gamma_kernel(ProbSet ps, ChunkSplit split, const float *__restrict__ A, const float *__restrict__ B,
                      const float *__restrict__ qd, const float *__restrict__ rd, const float *__restrict__ c,
                      const float *__restrict__ q, const float *__restrict__ r, float *__restrict__ gamma) {
  __shared__ float sm[kChunkFloats];
  __shared__ float sg[kChunkItems + kMaxNx];  // scaled gradients q_k / qd_k, r_k / rd_k, nx + nu per block
  const int tid = threadIdx.x;
  const ProbDesc d = ps.get(blockIdx.x / split.per);
  const int N = d.N, nx = d.nx, nu = d.nu, m = nx + nu, per = split.per,
            C = chunk_length(chunk_rows(nx, nu), N + 1, split.share);
  const int lda = nx | 1, ldb = nu | 1;
  const Divisor by_m(m), by_nx(nx);
  float *sA = sm, *sB = sm + C * nx * lda;
  for (int k0 = (int)(blockIdx.x % per) * C; k0 <= N; k0 += per * C) {
    const int k1 = min(N + 1, k0 + C), kb = k0 > 0 ? k0 - 1 : 0, nb = k1 - 1 - kb;  // rows [k0, k1), blocks [kb, k1 - 1)
    stage_chunk(sA, A + d.oA + (int64_t)kb * nx * nx, nb * nx, nx, lda, tid, kKktThreads);
    if (nu > 0) stage_chunk(sB, B + d.oB + (int64_t)kb * nx * nu, nb * nx, nu, ldb, tid, kKktThreads);
    for (int e = tid; e < nb * m; e += kKktThreads) {
      const int kk = by_m.quotient(e), j = e - kk * m, k = kb + kk;
      sg[e] = j < nx ? q[d.ovec + k * nx + j] / qd[d.oq + k * nx + j]
                     : r[d.orr + k * nu + j - nx] / rd[d.orr + k * nu + j - nx];
    }
    __syncthreads();
    for (int e = tid; e < (k1 - k0) * nx; e += kKktThreads) {
      const int kk = by_nx.quotient(e), i = e - kk * nx, k = k0 + kk;
      const int64_t o = d.ovec + (int64_t)k * nx + i;
      const float own = q[o] / qd[d.oq + (int64_t)k * nx + i];
      float acc = 0.f;
      if (k > 0) {
        const int b = k - 1 - kb;
        const float *a = sA + (b * nx + i) * lda, *s = sg + b * m;
        for (int j = 0; j < nx; ++j) acc = fmaf(a[j], s[j], acc);
        const float *bb = sB + (b * nx + i) * ldb;
        for (int j = 0; j < nu; ++j) acc = fmaf(bb[j], s[nx + j], acc);
      }
      gamma[o] = k == 0 ? c[o] + own : c[o] - acc + own;
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kKktThreads)
    recover_step_kernel(ProbSet ps, ChunkSplit split, const float *__restrict__ A, const float *__restrict__ B,
                        const float *__restrict__ qd, const float *__restrict__ rd, const float *__restrict__ q,
                        const float *__restrict__ r, const float *__restrict__ mu, float *__restrict__ dx,
                        float *__restrict__ du) {
  __shared__ float sm[kChunkItems + kMaxNx];  // mu_{k+1} of the chunk's block rows
  const int tid = threadIdx.x;
  const ProbDesc d = ps.get(blockIdx.x / split.per);
  const int N = d.N, nx = d.nx, nu = d.nu, m = nx + nu, per = split.per,
            C = chunk_length(chunk_rows(nx, nu), N + 1, split.share);
  const Divisor by_m(m);
  for (int k0 = (int)(blockIdx.x % per) * C; k0 <= N; k0 += per * C) {
    const int k1 = min(N + 1, k0 + C), nb = min(k1, N) - k0;
    for (int e = tid; e < nb * nx; e += kKktThreads) sm[e] = mu[d.ovec + (int64_t)(k0 + 1) * nx + e];
    __syncthreads();
    for (int e = tid; e < (k1 - k0) * m; e += kKktThreads) {
      const int kk = by_m.quotient(e), j = e - kk * m, k = k0 + kk;
      const bool state = j < nx;
      if (!state && k == N) continue;
      float acc = 0.f;
      if (k < N) {
        // column j of A_k, or column j - nx of B_k
        const float *col = state ? A + d.oA + (int64_t)k * nx * nx + j : B + d.oB + (int64_t)k * nx * nu + (j - nx);
        const int w = state ? nx : nu;
        const float *s = sm + kk * nx;
        for (int l0 = 0; l0 < nx; l0 += 8) {  // eight loads in flight
          float v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = l0 + u < nx ? __ldg(col + (l0 + u) * w) : 0.0f;
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (l0 + u < nx) acc = fmaf(v[u], s[l0 + u], acc);
        }
      }
      if (state) {
        const int64_t o = d.ovec + (int64_t)k * nx + j;
        dx[o] = (q[o] - mu[o] + acc) / qd[d.oq + (int64_t)k * nx + j];
      } else {
        const int64_t o = d.orr + (int64_t)k * nu + (j - nx);
        du[o] = (r[o] + acc) / rd[o];
      }
    }
    __syncthreads();
  }
}

ChunkSplit kkt_split(int64_t nprob, int max_N, int nx, int nu) {
  return chunk_split(nprob, host::sms(), max_N + 1, chunk_rows(nx, nu), 4);
}

bool shape_ok(int N, int nx, int nu) {
  return N >= 0 && N <= SSPCG_MAX_N && nx >= 1 && nx <= SSPCG_MAX_NX && nu >= 0 && nu <= SSPCG_MAX_NX;
}

ProbDesc single(int N, int nx, int nu) {
  ProbDesc d{};
  d.N = N; d.nx = nx; d.nu = nu;
  return d;
}

}  // namespace
}  // namespace sspcg

using namespace sspcg;

#define KKT_CUDA(call)                                          \
  do {                                                          \
    cudaError_t e_ = (call);                                    \
    if (e_ != cudaSuccess) return sspcg::host::cuda_error(e_);  \
  } while (0)

extern "C" {

sspcg_status sspcg_form_gamma(int32_t N, int32_t nx, int32_t nu, const float *A, const float *B, const float *qd,
                              const float *rd, const float *c, const float *q, const float *r, float *gamma,
                              sspcg_stream stream) {
  if (!shape_ok(N, nx, nu)) return SSPCG_ERR_INVALID_ARG;
  if (!qd || !c || !q || !gamma || (N > 0 && (!A || (nu > 0 && (!B || !rd || !r))))) return SSPCG_ERR_INVALID_ARG;
  const ChunkSplit split = kkt_split(1, N, nx, nu);
  form_gamma_kernel<<<split.per, kKktThreads, 0, (cudaStream_t)stream>>>(ProbSet{nullptr, single(N, nx, nu), 1}, split, A, B, qd,
                                                                   rd, c, q, r, gamma);
  KKT_CUDA(cudaGetLastError());
  return SSPCG_OK;
}

sspcg_status sspcg_recover_step(int32_t N, int32_t nx, int32_t nu, const float *A, const float *B, const float *qd,
                                const float *rd, const float *q, const float *r, const float *mu, float *dx,
                                float *du, sspcg_stream stream) {
  if (!shape_ok(N, nx, nu)) return SSPCG_ERR_INVALID_ARG;
  if (!qd || !q || !mu || !dx || (N > 0 && (!A || (nu > 0 && (!B || !rd || !r || !du)))))
    return SSPCG_ERR_INVALID_ARG;
  const ChunkSplit split = kkt_split(1, N, nx, nu);
  recover_step_kernel<<<split.per, kKktThreads, 0, (cudaStream_t)stream>>>(ProbSet{nullptr, single(N, nx, nu), 1}, split, A, B,
                                                                     qd, rd, q, r, mu, dx, du);
  KKT_CUDA(cudaGetLastError());
  return SSPCG_OK;
}

sspcg_status sspcg_form_gamma_batched(sspcg_plan *plan, const float *A, const float *B, const float *qd,
                                      const float *rd, const float *c, const float *q, const float *r, float *gamma,
                                      sspcg_stream stream) {
  if (!plan) return SSPCG_ERR_INVALID_ARG;
  const host::PlanView v = host::plan_view(plan);
  if (v.nprob == 0) return SSPCG_OK;
  if (!qd || !c || !q || !gamma || (v.total_off > 0 && (!A || !B || !rd || !r))) return SSPCG_ERR_INVALID_ARG;
  const ChunkSplit split = kkt_split(v.nprob, v.max_N, v.max_nx, v.max_nu);
  form_gamma_kernel<<<(unsigned)v.nprob * split.per, kKktThreads, 0, (cudaStream_t)stream>>>(v.ps, split, A, B, qd, rd, c, q, r,
                                                                                       gamma);
  KKT_CUDA(cudaGetLastError());
  return SSPCG_OK;
}

sspcg_status sspcg_recover_step_batched(sspcg_plan *plan, const float *A, const float *B, const float *qd,
                                        const float *rd, const float *q, const float *r, const float *mu, float *dx,
                                        float *du, sspcg_stream stream) {
  if (!plan) return SSPCG_ERR_INVALID_ARG;
  const host::PlanView v = host::plan_view(plan);
  if (v.nprob == 0) return SSPCG_OK;
  if (!qd || !q || !mu || !dx || (v.total_off > 0 && (!A || !B || !rd || !r || !du))) return SSPCG_ERR_INVALID_ARG;
  const ChunkSplit split = kkt_split(v.nprob, v.max_N, v.max_nx, v.max_nu);
  recover_step_kernel<<<(unsigned)v.nprob * split.per, kKktThreads, 0, (cudaStream_t)stream>>>(v.ps, split, A, B, qd, rd, q, r,
                                                                                         mu, dx, du);
  KKT_CUDA(cudaGetLastError());
  return SSPCG_OK;
}

}  // extern "C"
