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
// Two kernels for each step, bit-identical: a CTA takes chunks of consecutive
// block rows of one problem (common.cuh), or a warp takes a knot with a row (for
// the primal step a column) per lane.  Both are bound by reading A and B once.  A
// warp per knot touches a line per lane and leaves lanes past nx idle, which costs
// 4.5 times the time with nx = 4 on many knots; a chunk's blocks come to shared
// memory for the right-hand side, whose rows are read by one thread each, which
// costs a trip through it and two barriers.  gamma_chunks and recover_chunks draw
// the lines.
#include "../../include/sspcg.h"
#include "common.cuh"
#include "host.h"

namespace sspcg {
namespace {

constexpr int kKktThreads = 256;

// With ``per`` CTAs for each problem, CTA b takes chunks b % per, b % per + per, ... of problem b / per.
__global__ void __launch_bounds__(kKktThreads, 7)  // what the shared memory holds; five CTAs take a quarter longer
    form_gamma_chunks(ProbSet ps, ChunkSplit split, const float *__restrict__ A, const float *__restrict__ B,
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
    recover_step_chunks(ProbSet ps, ChunkSplit split, const float *__restrict__ A, const float *__restrict__ B,
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

// A warp per knot: refs[g] = (problem, knot) of warp g (nullptr: one problem, knot g).
constexpr int kKktWarps = kKktThreads / 32;

__global__ void __launch_bounds__(kKktThreads)
    form_gamma_knots(ProbSet ps, const int2 *refs, int64_t knots, const float *__restrict__ A,
                     const float *__restrict__ B, const float *__restrict__ qd, const float *__restrict__ rd,
                     const float *__restrict__ c, const float *__restrict__ q, const float *__restrict__ r,
                     float *__restrict__ gamma) {
  const int lane = threadIdx.x & 31;
  const int64_t g = (int64_t)blockIdx.x * kKktWarps + (threadIdx.x >> 5);
  if (g >= knots) return;
  const int2 ref = refs ? refs[g] : make_int2(0, (int)g);
  const ProbDesc d = ps.get(ref.x);
  const int k = ref.y, m = d.nx, u = d.nu;
  // scaled gradient of knot k-1, one entry per lane (zero past the block)
  float sq = 0.f, sr = 0.f;
  if (k > 0) {
    if (lane < m) sq = q[d.ovec + (int64_t)(k - 1) * m + lane] / qd[d.oq + (int64_t)(k - 1) * m + lane];
    if (lane < u) sr = r[d.orr + (int64_t)(k - 1) * u + lane] / rd[d.orr + (int64_t)(k - 1) * u + lane];
  }
  float acc = 0.f;
  if (k > 0) {
    const float *Ar = A + d.oA + (int64_t)(k - 1) * m * m + (int64_t)(lane < m ? lane : 0) * m;
    for (int j = 0; j < m; ++j) {
      const float s = __shfl_sync(0xffffffffu, sq, j);
      if (lane < m) acc = fmaf(Ar[j], s, acc);
    }
    if (u > 0) {
      const float *Br = B + d.oB + (int64_t)(k - 1) * m * u + (int64_t)(lane < m ? lane : 0) * u;
      for (int j = 0; j < u; ++j) {
        const float s = __shfl_sync(0xffffffffu, sr, j);
        if (lane < m) acc = fmaf(Br[j], s, acc);
      }
    }
  }
  if (lane < m) {
    const int64_t e = d.ovec + (int64_t)k * m + lane;
    const float own = q[e] / qd[d.oq + (int64_t)k * m + lane];
    gamma[e] = k == 0 ? c[e] + own : c[e] - acc + own;
  }
}

__global__ void __launch_bounds__(kKktThreads)
    recover_step_knots(ProbSet ps, const int2 *refs, int64_t knots, const float *__restrict__ A,
                       const float *__restrict__ B, const float *__restrict__ qd, const float *__restrict__ rd,
                       const float *__restrict__ q, const float *__restrict__ r, const float *__restrict__ mu,
                       float *__restrict__ dx, float *__restrict__ du) {
  const int lane = threadIdx.x & 31;
  const int64_t g = (int64_t)blockIdx.x * kKktWarps + (threadIdx.x >> 5);
  if (g >= knots) return;
  const int2 ref = refs ? refs[g] : make_int2(0, (int)g);
  const ProbDesc d = ps.get(ref.x);
  const int k = ref.y, m = d.nx, u = d.nu, N = d.N;
  // mu_{k+1}, one entry per lane
  const float mn = (k < N && lane < m) ? mu[d.ovec + (int64_t)(k + 1) * m + lane] : 0.f;
  float ax = 0.f, bu = 0.f;
  if (k < N) {
    const float *Ac = A + d.oA + (int64_t)k * m * m + (lane < m ? lane : 0);                    // column lane of A_k
    const float *Bc = u > 0 ? B + d.oB + (int64_t)k * m * u + (lane < u ? lane : 0) : nullptr;  // of B_k
    for (int l = 0; l < m; ++l) {
      const float s = __shfl_sync(0xffffffffu, mn, l);
      if (lane < m) ax = fmaf(Ac[(int64_t)l * m], s, ax);
      if (lane < u) bu = fmaf(Bc[(int64_t)l * u], s, bu);
    }
  }
  if (lane < m) {
    const int64_t e = d.ovec + (int64_t)k * m + lane;
    dx[e] = (q[e] - mu[e] + ax) / qd[d.oq + (int64_t)k * m + lane];
  }
  if (k < N && lane < u) {
    const int64_t e = d.orr + (int64_t)k * u + lane;
    du[e] = (r[e] + bu) / rd[e];
  }
}

// What the launches take of a batch, or of one problem.
struct Set {
  ProbSet ps;
  const int2 *refs;
  int64_t knots, rows;  // of all problems
  int max_N, max_nx, max_nu;
  ChunkSplit split() const {
    return chunk_split(ps.nprob, host::sms(), max_N + 1, chunk_rows(max_nx, max_nu), 4);
  }
  unsigned knot_ctas() const { return (unsigned)cdiv(knots, kKktWarps); }
};

// Chunks for the right-hand side: of small blocks (nx 8 on average) from 10,000 knots on, 20,000 with more inputs than
// states, of medium ones (16) from 60,000, never of large ones nor with more than 8 inputs and fewer states.  Chunks
// against warps, us, with A and B in L2 unless said otherwise: nx 4, 64 problems of N 64 4.9 / 3.3, 512 of N 20 5.2 / 5.4,
// 8192 of N 20 33 / 51; nx 1, nu 2, 1024 of N 64 12 / 20; nx 14, 2048 of N 20 25 / 20, 1024 of N 64 40 / 40 (from HBM 53 /
// 56), 8192 of N 20 95 / 113; nx 21, 8192 of N 20 163 / 154; nx 4, nu 28, 1024 of N 64 38 / 34; N 16-128, nx 4, 12, 14, 21:
// 512 problems 26 / 19 (from HBM 38 / 36), 4096 171 / 195.
bool gamma_chunks(const Set &s) {
  if (s.max_nu > s.max_nx && s.max_nu > 8) return false;
  return (s.rows <= 8 * s.knots && s.knots >= (s.max_nu > s.max_nx ? 20000 : 10000)) ||
         (s.rows <= 16 * s.knots && s.knots >= 60000);
}
// Chunks for the primal step from 16,000 knots on, unless there are more than two inputs to a state, and of large blocks
// (12) up to 2,000: nx 14, N 64 alone 3.5 / 4.1; nx 4, 64 problems of N 64 3.7 / 3.3, 8192 of N 20 22 / 55; nx 21, 512 of N 20 10.5 / 9.9 (from HBM 20 / 24), 2048 40 / 63; nx 28, 512 of N 20
// 15 / 11; the mixed 4096 133 / 267; nx 4, nu 28, 2048 of N 20 22 / 16 (from HBM 33 / 38).
bool recover_chunks(const Set &s) {
  return (s.knots >= 16000 && s.max_nu <= 2 * s.max_nx) || (s.rows >= 12 * s.knots && s.knots <= 2000);
}

cudaError_t launch_form_gamma(const Set &s, const float *A, const float *B, const float *qd, const float *rd,
                              const float *c, const float *q, const float *r, float *gamma, cudaStream_t st) {
  if (gamma_chunks(s)) {
    const ChunkSplit split = s.split();
    form_gamma_chunks<<<(unsigned)s.ps.nprob * split.per, kKktThreads, 0, st>>>(s.ps, split, A, B, qd, rd, c, q, r,
                                                                                gamma);
  } else {
    form_gamma_knots<<<s.knot_ctas(), kKktThreads, 0, st>>>(s.ps, s.refs, s.knots, A, B, qd, rd, c, q, r, gamma);
  }
  return cudaGetLastError();
}

cudaError_t launch_recover_step(const Set &s, const float *A, const float *B, const float *qd, const float *rd,
                                const float *q, const float *r, const float *mu, float *dx, float *du,
                                cudaStream_t st) {
  if (recover_chunks(s)) {
    const ChunkSplit split = s.split();
    recover_step_chunks<<<(unsigned)s.ps.nprob * split.per, kKktThreads, 0, st>>>(s.ps, split, A, B, qd, rd, q, r, mu,
                                                                                  dx, du);
  } else {
    recover_step_knots<<<s.knot_ctas(), kKktThreads, 0, st>>>(s.ps, s.refs, s.knots, A, B, qd, rd, q, r, mu, dx, du);
  }
  return cudaGetLastError();
}

bool shape_ok(int N, int nx, int nu) {
  return N >= 0 && N <= SSPCG_MAX_N && nx >= 1 && nx <= SSPCG_MAX_NX && nu >= 0 && nu <= SSPCG_MAX_NX;
}

Set single(int N, int nx, int nu) {
  ProbDesc d{};
  d.N = N; d.nx = nx; d.nu = nu;
  return {ProbSet{nullptr, d, 1}, nullptr, N + 1, (int64_t)(N + 1) * nx, N, nx, nu};
}

Set batch(const host::PlanView &v) { return {v.ps, v.kref, v.knots, v.rows, v.max_N, v.max_nx, v.max_nu}; }

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
  KKT_CUDA(launch_form_gamma(single(N, nx, nu), A, B, qd, rd, c, q, r, gamma, (cudaStream_t)stream));
  return SSPCG_OK;
}

sspcg_status sspcg_recover_step(int32_t N, int32_t nx, int32_t nu, const float *A, const float *B, const float *qd,
                                const float *rd, const float *q, const float *r, const float *mu, float *dx,
                                float *du, sspcg_stream stream) {
  if (!shape_ok(N, nx, nu)) return SSPCG_ERR_INVALID_ARG;
  if (!qd || !q || !mu || !dx || (N > 0 && (!A || (nu > 0 && (!B || !rd || !r || !du)))))
    return SSPCG_ERR_INVALID_ARG;
  KKT_CUDA(launch_recover_step(single(N, nx, nu), A, B, qd, rd, q, r, mu, dx, du, (cudaStream_t)stream));
  return SSPCG_OK;
}

sspcg_status sspcg_form_gamma_batched(sspcg_plan *plan, const float *A, const float *B, const float *qd,
                                      const float *rd, const float *c, const float *q, const float *r, float *gamma,
                                      sspcg_stream stream) {
  if (!plan) return SSPCG_ERR_INVALID_ARG;
  const host::PlanView v = host::plan_view(plan);
  if (v.nprob == 0) return SSPCG_OK;
  if (!qd || !c || !q || !gamma || (v.total_off > 0 && (!A || !B || !rd || !r))) return SSPCG_ERR_INVALID_ARG;
  KKT_CUDA(launch_form_gamma(batch(v), A, B, qd, rd, c, q, r, gamma, (cudaStream_t)stream));
  return SSPCG_OK;
}

sspcg_status sspcg_recover_step_batched(sspcg_plan *plan, const float *A, const float *B, const float *qd,
                                        const float *rd, const float *q, const float *r, const float *mu, float *dx,
                                        float *du, sspcg_stream stream) {
  if (!plan) return SSPCG_ERR_INVALID_ARG;
  const host::PlanView v = host::plan_view(plan);
  if (v.nprob == 0) return SSPCG_OK;
  if (!qd || !q || !mu || !dx || (v.total_off > 0 && (!A || !B || !rd || !r || !du))) return SSPCG_ERR_INVALID_ARG;
  KKT_CUDA(launch_recover_step(batch(v), A, B, qd, rd, q, r, mu, dx, du, (cudaStream_t)stream));
  return SSPCG_OK;
}

}  // extern "C"
