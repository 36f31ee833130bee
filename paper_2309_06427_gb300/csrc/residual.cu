// True residual ||gamma - S lambda||_2 / ||gamma||_2 in FP64 with S applied in
// the factored form of Eq. (schur), S = C G^-1 C^T, from the QP data.
// Diagnostic: one CTA per problem, walking its block rows in chunks that give
// every thread one column of a chunk's [A_k B_k].
//
// Bound: the FP64 units, which take a warp instruction in 19 cycles per SM here
// whatever its active lanes.  So a chunk's blocks come to shared memory with
// coalesced loads, every FP32 value becomes a double by integer arithmetic on
// its bits, a division is seven FP64 instructions, and columns of A_k and B_k
// share one loop, so that a warp runs each FP64 instruction once for all its
// lanes.  Problems go to the CTAs largest first: an SM holds several at a time,
// and a large one begun late would outlast all others.  The call with the two
// steps of kkt.cu, 4096 problems of N 16-128 and nx 4, 12, 14, 21: 2.47 ms before,
// 1.49 ms in chunks in the order of the batch, 1.26 ms largest first (1.36 ms
// with CTAs of 128 threads), 1.20 ms with the two steps as they are cut now.
#include "common.cuh"
#include "kernels.h"

namespace sspcg {

constexpr int kResThreads = 256;

// (double)f without the FP64 pipe: exponent rebiased and mantissa shifted; zeros by selection, subnormals,
// infinities and NaN by the conversion.
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f), mag = u & 0x7fffffffu;
  if (mag - 0x00800000u >= 0x7f000000u && mag != 0u) {  // rare; volatile, so that it stays behind the branch
    double d;
    asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(f));
    return d;
  }
  const uint32_t hi = mag == 0u ? 0u : (mag >> 3) + 0x38000000u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(mag << 29));
}

// s / q for an FP32 q > 0: Newton's method on the FP32 reciprocal, then one correction of the quotient.
__device__ __forceinline__ double divide(double s, float q) {
  const float y0 = __frcp_rn(q);
  const double d = widen(q);
  if (!(y0 >= 1.17549435e-38f && y0 <= 3.402823466e38f)) return s / d;  // q outside the reciprocal's normal range
  double y = widen(y0);
  y = fma(y, fma(-d, y, 1.0), y);
  y = fma(y, fma(-d, y, 1.0), y);
  const double t = s * y;
  if ((__double2hiint(t) & 0x7ff00000) == 0x7ff00000) return t;  // infinite or NaN: no correction
  return fma(fma(-d, t, s), y, t);
}

// WIDE: chunks of residual_rows for problems with nu > nx, v_x and v_u before the blocks in one array.  Batches without
// such a problem run the other form: with v_x and v_u in an array of their own lone problems take up to 7 % less.  A
// problem's result does not depend on the others of its batch.
template <bool WIDE>
__global__ void __launch_bounds__(kResThreads) residual_qp_kernel(ProbSet ps, const int32_t *order,
                                                                  const float *__restrict__ A,
                                                                  const float *__restrict__ B,
                                                                  const float *__restrict__ qd,
                                                                  const float *__restrict__ rd,
                                                                  const float *__restrict__ gamma,
                                                                  const float *__restrict__ lambda, double *out) {
  __shared__ __align__(16) float sm[WIDE ? kResFloats : kChunkFloats];
  __shared__ double sx[kChunkItems + 2 * kMaxNx];  // lambda of the chunk's block rows and of the next one
  __shared__ double sv_[WIDE ? 1 : kChunkItems + kMaxNx];
  __shared__ double sy[kMaxNx];                    // A_{k-1} v_x(k-1) + B_{k-1} v_u(k-1) for the next chunk's first row
  __shared__ double red[2][kResThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int p = blockIdx.x; p < ps.nprob; p += gridDim.x) {
    const ProbDesc d = ps.get(order ? order[p] : p);
    const int N = d.N, nx = d.nx, nu = d.nu, m = nx + nu,
              C = WIDE && nu > nx ? residual_rows(nx, nu) : chunk_rows(nx, nu);
    const int lda = nx | 1, ldb = nu | 1;
    const float *Ap = A + d.oA, *Bp = B + d.oB, *q = qd + d.oq, *r = rd + d.orr;
    const float *g = gamma + d.ovec, *x = lambda + d.ovec;
    const Divisor by_m(m), by_nx(nx);
    double *sv = WIDE ? reinterpret_cast<double *>(sm) : sv_;  // v_x and v_u of the chunk, nx + nu per block row
    float *sA = WIDE ? sm + 2 * C * m : sm, *sB = sA + C * nx * lda;
    double res2 = 0.0, g2 = 0.0;
    if (tid < nx) sy[tid] = 0.0;
    for (int k0 = 0; k0 <= N; k0 += C) {
      const int k1 = min(N + 1, k0 + C), nb = min(k1, N) - k0;  // block rows [k0, k1), blocks [k0, k0 + nb)
      stage_chunk(sA, Ap + (int64_t)k0 * nx * nx, nb * nx, nx, lda, tid, kResThreads);
      if (nu > 0) stage_chunk(sB, Bp + (int64_t)k0 * nx * nu, nb * nx, nu, ldb, tid, kResThreads);
      for (int e = tid; e < (min(k1 + 1, N + 1) - k0) * nx; e += kResThreads) sx[e] = widen(x[k0 * nx + e]);
      __syncthreads();
      // v_x(k)[j] = (-x_k[j] + sum_l A_k[l][j] x_{k+1}[l]) / q_k[j];  v_u(k)[j] = sum_l B_k[l][j] x_{k+1}[l] / r_k[j]
      for (int e = tid; e < (k1 - k0) * m; e += kResThreads) {
        const int kk = by_m.quotient(e), c = e - kk * m, k = k0 + kk;
        const bool state = c < nx;
        if (!state && k == N) continue;
        // one loop for the columns of A_k and B_k: a warp holds both
        const double *xn = sx + (kk + 1) * nx;
        const float *col = state ? sA + kk * nx * lda + c : sB + kk * nx * ldb + (c - nx);
        const int ld = state ? lda : ldb;
        double s = state ? -sx[kk * nx + c] : 0.0;
        if (k < N)
          for (int l = 0; l < nx; ++l) s = fma(widen(col[l * ld]), xn[l], s);
        sv[e] = divide(s, state ? q[k * nx + c] : r[k * nu + c - nx]);
      }
      __syncthreads();
      // (S x)_k[i] = -v_x(k)[i] + y_k[i], y_k = A_{k-1} v_x(k-1) + B_{k-1} v_u(k-1); y of row k1 is for the next chunk
      double y_next = 0.0;
      for (int e = tid; e < (nb + 1) * nx; e += kResThreads) {
        const int kk = by_nx.quotient(e), i = e - kk * nx;
        double y = 0.0;
        if (kk == 0) {
          y = sy[i];
        } else {
          const float *a = sA + ((kk - 1) * nx + i) * lda, *b = sB + ((kk - 1) * nx + i) * ldb;
          const double *v = sv + (kk - 1) * m;
          for (int j = 0; j < nx; ++j) y = fma(widen(a[j]), v[j], y);
          for (int j = 0; j < nu; ++j) y = fma(widen(b[j]), v[nx + j], y);
        }
        const int k = k0 + kk;
        if (k < k1) {
          const double gi = widen(g[k * nx + i]);
          const double ri = gi - (y - sv[kk * m + i]);
          res2 = fma(ri, ri, res2);
          g2 = fma(gi, gi, g2);
        } else {
          y_next = y;
        }
      }
      __syncthreads();
      for (int e = tid; e < (nb + 1) * nx; e += kResThreads) {  // the thread that formed it stores it
        const int kk = by_nx.quotient(e);
        if (k0 + kk >= k1) sy[e - kk * nx] = y_next;
      }
      __syncthreads();
    }
    res2 = warp_sum(res2);
    g2 = warp_sum(g2);
    if (lane == 0) { red[0][wid] = res2; red[1][wid] = g2; }
    __syncthreads();
    if (tid == 0) {
      double a = 0.0, b = 0.0;
      for (int w = 0; w < kResThreads / 32; ++w) { a += red[0][w]; b += red[1][w]; }
      out[d.id] = b > 0.0 ? sqrt(a / b) : 0.0;
    }
    __syncthreads();
  }
}

cudaError_t launch_residual_qp(const ProbSet &ps, const int32_t *order, bool wide, const float *A, const float *B,
                               const float *qd, const float *rd, const float *gamma, const float *lambda, double *relres_true,
                               cudaStream_t st) {
  if (ps.nprob == 0) return cudaSuccess;
  if (wide)
    residual_qp_kernel<true><<<ps.nprob, kResThreads, 0, st>>>(ps, order, A, B, qd, rd, gamma, lambda, relres_true);
  else
    residual_qp_kernel<false><<<ps.nprob, kResThreads, 0, st>>>(ps, order, A, B, qd, rd, gamma, lambda, relres_true);
  return cudaGetLastError();
}

}  // namespace sspcg
