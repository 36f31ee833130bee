// Host-side declarations shared by the CUDA translation units of sspcg.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

namespace sspcg {

// Operator forms for S p.
enum OpForm : int { kOpBlock = 0, kOpQp = 1 };
// Precision of the dot-product reductions.
enum RedMode : int { kRedF32 = 0, kRedDf = 1, kRedF64 = 2 };

// Padded leading dimension of a matrix staged in shared memory: odd, so that
// 32 consecutive rows touch 32 distinct banks.
__host__ __device__ __forceinline__ int pad_ld(int x) { return x | 1; }

// Shared-memory carve-up of one PCG problem, in elements of the working
// precision; every region starts 16-byte aligned.  The first K block rows of
// the operator and preconditioner blocks are staged (K = N+1: fully
// resident; K = 0: everything read from L2/HBM each iteration).  The same
// function sizes launches on the host and carves on the device.
//
// Every vector has a zero segment before block row 0 and after block row N
// (the offsets below point at block row 0), so that a row's three block
// products read their neighbour segments without branches: the segment of
// the missing neighbour is zero.  A single-knot problem (N = 0) stages one
// zero off-diagonal slot, so that its clamped off-diagonal reads stay in
// bounds.
struct PcgLayout {
  int64_t p, r, w, x, e, u, s, v;   // vectors (e: the polynomial's residual; u, s: single-reduction CG)
  int64_t vu;                       // v_u block rows (QP form), after v_x
  int64_t iq, ir;                   // 1/q, 1/r (QP form)
  int64_t m0, m1, pd, pe;           // staged blocks
  int64_t total;
};

// Vectors are stored with a block-row stride of nx rounded up to 4 elements,
// so that every block row starts 16-byte aligned and a thread can load a
// whole block-row segment with 128-bit loads.
__host__ __device__ __forceinline__ int vec_stride(int x) { return (x + 3) & ~3; }

// Staged off-diagonal slots of a layout with K staged block rows: K (at most N), and one zero slot for N = 0.
__host__ __device__ __forceinline__ int64_t staged_off_slots(int K, int N) {
  const int64_t Ks = K < N ? K : N;
  return (N == 0 && K > 0) ? 1 : Ks;
}

__host__ __device__ inline PcgLayout pcg_layout(int op, int K, int N, int nx, int nu, int poly = 0, int cg = 0) {
  PcgLayout L{};
  const int64_t n = N + 1, NXP = vec_stride(nx), NUP = vec_stride(nu);
  const int64_t RVP = (n + 2) * NXP;  // a vector with its two zero segments
  const int64_t Ks = staged_off_slots(K, N);
  const int64_t ld = pad_ld(nx), ldb = pad_ld(nu > 0 ? nu : 1);
  int64_t o = 0;
  L.p = o + NXP; o += RVP;
  L.r = o + NXP; o += RVP;
  L.w = o + NXP; o += RVP;
  L.x = o + NXP; o += RVP;
  L.e = o + NXP;
  if (poly) o += RVP;
  L.u = o + NXP;
  if (cg) o += RVP;
  L.s = o + NXP;
  if (cg) o += RVP;
  L.v = o + NXP;  // the block form has no v (no region)
  L.vu = op == kOpQp ? L.v + (n + 1) * NXP + NUP : L.v;
  if (op == kOpQp) o += RVP + (int64_t)(N + 1) * NUP;   // v_x with its zero segments, then v_u after one
  L.iq = o;
  if (op == kOpQp) o += n * NXP;
  L.ir = o;
  if (op == kOpQp) o += (int64_t)N * NUP;
  if (op == kOpQp) {
    L.m0 = o; o += round_up(Ks * nx * ld, 4);    // A_k, row stride ld
    L.m1 = o; o += round_up(Ks * nx * ldb, 4);   // B_k, row stride ldb
  } else {
    L.m0 = o; o += round_up((int64_t)K * nx * ld, 4);  // D_k
    L.m1 = o; o += round_up(Ks * nx * ld, 4);          // E_k
  }
  L.pd = o; o += round_up((int64_t)K * nx * ld, 4);    // PD_k
  L.pe = o; o += round_up(Ks * nx * ld, 4);            // PE_k
  L.total = o;
  return L;
}

// Largest number of staged block rows whose layout fits in ``elems``; -1 when
// not even the vectors fit.
__host__ __device__ inline int pcg_max_resident(int op, int N, int nx, int nu, int64_t elems, int poly = 0,
                                                int cg = 0) {
  if (pcg_layout(op, N + 1, N, nx, nu, poly, cg).total <= elems) return N + 1;
  if (pcg_layout(op, 0, N, nx, nu, poly, cg).total > elems) return -1;
  int lo = 0, hi = N;  // invariant: layout(lo) fits, layout(hi + 1) does not
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (pcg_layout(op, mid, N, nx, nu, poly, cg).total <= elems) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// The kernel with a thread per row pair (pcg_one.cuh): FP32 textbook PCG with double-float sums and a degree-0
// preconditioner, for problems that fit in shared memory whole.
//
// Its blocks are staged as 2 x 2 tiles: tile (q, c) holds rows 2q, 2q+1 and columns 2c, 2c+1 as four consecutive
// values (m00, m01, m10, m11), zero past an odd last row or column.  A thread owns a pair of rows of the unknowns,
// so one 128-bit load feeds four multiply-adds whichever way the block is read: along tile row q for rows 2q, 2q+1
// of M v, or down tile column c for rows 2c, 2c+1 of M^T v.  Tile rows are an odd number of tiles long, so that
// eight threads on consecutive tile rows (one phase of a 128-bit shared-memory load) touch 32 distinct banks.
__host__ __device__ __forceinline__ int tile_half(int x) { return (x + 1) >> 1; }
__host__ __device__ __forceinline__ int tile_ld(int cols) { return tile_half(cols) | 1; }
__host__ __device__ __forceinline__ int tile_block(int rows, int cols) {  // values of a block
  return cols > 0 ? 4 * tile_half(rows) * tile_ld(cols) : 0;
}

// Its shared memory, in floats; regions and vectors as in PcgLayout, without w and x.  A single-knot problem
// (N = 0) has one zero off-diagonal slot of each kind.
struct OneLayout {
  int64_t p, r, v, vu, iq, ir, m0, m1, pd, pe, total;
};
__host__ __device__ inline OneLayout pcg_one_layout(int op, int N, int nx, int nu) {
  OneLayout L{};
  const int64_t n = N + 1, NXP = vec_stride(nx), NUP = vec_stride(nu), RVP = (n + 2) * NXP;
  const int64_t blk = tile_block(nx, nx), blkb = tile_block(nx, nu), slots = N > 0 ? N : 1;
  const bool qp = op == kOpQp;
  int64_t o = 0;
  L.p = o + NXP; o += RVP;
  L.r = o + NXP; o += RVP;
  L.v = o + NXP; o += qp ? RVP : 0;
  L.vu = o + NUP; o += qp ? n * NUP : 0;  // v_u(-1) is zero
  L.iq = o; o += qp ? n * NXP : 0;
  L.ir = o; o += qp ? N * NUP : 0;
  L.m0 = o; o += qp ? slots * blk : n * blk;  // A_k; D_k, transposed
  L.m1 = o; o += slots * (qp ? blkb : blk);   // B_k; E_k
  L.pd = o; o += n * blk;                     // PD_k, transposed
  L.pe = o; o += slots * blk;                 // PE_k
  L.total = o;
  return L;
}

// Arguments of a PCG launch (by value).
struct PcgArgs {
  ProbSet ps;
  const int32_t *work;   // problem indices in processing order (device), or nullptr: identity
  int32_t nwork;
  int32_t *counter;      // work-queue counter (device, zeroed before launch), or nullptr: static
  const float *A, *B, *qd, *rd;  // QP operator data (packed, FP32)
  const float *D, *E;            // block operator data (packed, FP32)
  const void *PD, *PE;           // preconditioner blocks in the working precision
  const float *gamma;
  void *lambda;                  // solution: float when lambda_f32, else the working precision
  int32_t lambda_f32;
  int32_t *iters;
  double *relres;
  int32_t *status;       // in: nonzero skips the problem; out: solve code
  float tol2;            // tol^2
  int32_t max_iter;      // <= 0: 10 (N+1) nx
  int32_t warm;          // 0, 1, 2 (see sspcg_options)
  int32_t poly;          // degree d of the polynomial preconditioner sum_{j<=d} (I - Phi^-1 S)^j Phi^-1
  int32_t cg;            // 1: single-reduction (Chronopoulos-Gear) PCG (QP form, FP32, double-float sums)
  int64_t smem_elems;    // dynamic shared memory of the launch, in elements of the working precision
  int32_t max_resident;  // cap on staged block rows (a schedule override); large = no cap
  void *gscratch;        // vectors in global memory: CTA b uses gscratch + b * gstride elements
  int64_t gstride;       //   (nullptr: vectors in shared memory)
  int32_t warp;          // 1: one problem per warp (smem_elems per warp), QP form, textbook PCG
  int32_t one;           // 1: the kernel with a thread per row pair (pcg_one_ok holds for every problem)
  const float *pad;      // padded copies of A, B, PE of the streamed problems (QP form, FP32), or nullptr
  const int64_t *pad_off;  // per problem id: offset of its copies in pad, or -1 (read the inputs)
};

// Floats of one padded region (rows of vec_stride(width) values), a multiple of 8 so that every region of a
// problem starts 32-byte aligned (the PCG reads padded rows of a multiple of 8 values with 256-bit loads).
__host__ __device__ __forceinline__ int64_t pad_region(int64_t rows, int width) {
  return round_up(rows * vec_stride(width), 8);
}

// Padded copies for the streamed block rows of the listed problems (desc indices): A_k and PE_k rows of
// vec_stride(nx) values, B_k rows of vec_stride(nu), zeros in the padding; problem p's copies start at
// pad_off[desc[p].id] (a multiple of 8 floats): A, then B at + pad_region(N nx, nx), then PE after B's
// pad_region(N nx, nu).  PE nullptr: no PE copy.
cudaError_t launch_pad_rows(const ProbDesc *desc, const int32_t *list, int32_t count, const float *A,
                            const float *B, const float *PE, const int64_t *pad_off, float *pad, int sms,
                            cudaStream_t st);

// PCG launch for one nx; dispatches to the instantiation for that nx.
// f64: the FP64 path (QP operator form only).  Each problem stages as many
// block rows as fit in ``smem`` bytes (at most a.max_resident).
cudaError_t launch_pcg(int nx, int op, int red, bool f64, const PcgArgs &a, int grid, int block, size_t smem,
                       cudaStream_t st);

int pcg_max_smem_bytes();
// CTAs of that PCG variant that fit on one SM at ``block`` threads and ``smem`` bytes of dynamic shared memory
// (registers, threads and shared memory; gv: vectors in a global workspace; cg: single-reduction PCG;
// warp: one problem per warp; one: a thread per row pair).
cudaError_t occupancy_pcg(int nx, int op, int red, bool f64, bool gv, bool cg, bool warp, bool one, int block,
                          size_t smem, int *ctas);

// Whether the kernel with a thread per row pair solves a problem of these options in a CTA of ``block`` threads
// with ``budget`` bytes of dynamic shared memory.
inline bool pcg_one_ok(int op, bool f64, int red, int poly, int cg, int block, int64_t budget, int64_t N, int nx,
                       int nu) {
  return !f64 && red == kRedDf && poly == 0 && !(cg && op == kOpQp) && (N + 1) * tile_half(nx) <= block &&
         pcg_one_layout(op, (int)N, nx, nu).total * (int64_t)sizeof(float) <= budget;
}

// Schur build and preconditioner assembly; Real = float (FP32 blocks; the Schur
// and the off-diagonal blocks of few small knots only) or double (the FP64
// path).  refs[i] = (problem, block row) of work item i
// (nullptr: one problem, item i is block row i, or i + 1 for off-diagonals).
// mx: the largest nx and nu of the launch (sizes the per-warp shared memory).
template <typename Real>
cudaError_t launch_schur_build(const ProbSet &ps, const int2 *refs, int64_t total_knots, const float *A,
                               const float *B, const float *qd, const float *rd, Real *D, Real *E,
                               cudaStream_t st, int sms, int mx);
// The same in FP32 (build_f32.cu), refs as above (read for few small knots only); max_N, max_nx, max_nu: the largest
// sizes of the set; off_elems: values of PE.
bool few_small_offs(int64_t total, int max_nx);
cudaError_t launch_schur_f32(const ProbSet &ps, const int2 *refs, int64_t total_knots, int max_N, int max_nx, int max_nu,
                             const float *A, const float *B, const float *qd, const float *rd, float *D, float *E, cudaStream_t st, int sms);
cudaError_t launch_precond_off_f32(const ProbSet &ps, const int2 *refs, int64_t total_off, int max_N, int max_nx,
                                   int kind, const float *E, const float *PD, float *PE, cudaStream_t st, int sms, int64_t off_elems);
// Schur blocks with full SPD cost blocks from their inverses: Qi laid out like
// D, R_{k-1}^-1 of problem p at roff[p] + (k-1) nu^2 (roff nullptr: offset 0).
cudaError_t launch_schur_full(const ProbSet &ps, const int2 *refs, int64_t total_knots, const int64_t *roff,
                              const float *A, const float *B, const float *Qi, const float *Ri, float *D, float *E,
                              cudaStream_t st, int mx);
// Diagonal blocks of Phi^-1 (FP64 inverses), one thread per knot: every
// knot of a launch must have the same nx.
template <typename Real>
cudaError_t launch_precond_inv(const ProbSet &ps, const int2 *refs, int64_t total_knots, int nx, int kind,
                               const Real *D, Real *PD, int32_t *status, cudaStream_t st);
// Off-diagonal blocks of Phi^-1 (any mix of nx).
template <typename Real>
cudaError_t launch_precond_off(const ProbSet &ps, const int2 *refs, int64_t total_off, int kind,
                               const Real *E, const Real *PD, Real *PE, cudaStream_t st, int sms, int64_t off_elems,
                               int mx);
// order: problem indices in the order in which they start (device), or nullptr: as numbered; wide: some nu > nx.
cudaError_t launch_residual_qp(const ProbSet &ps, const int32_t *order, bool wide, const float *A, const float *B,
                               const float *qd, const float *rd, const float *gamma, const float *lambda, double *relres_true,
                               cudaStream_t st);

}  // namespace sspcg
