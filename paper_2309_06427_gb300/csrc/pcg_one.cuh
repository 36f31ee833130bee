// PCG with a thread per row pair: the FP32 kernel for problems that fit in
// shared memory whole and have at most one row pair per thread (textbook PCG,
// double-float sums, degree-0 preconditioner; both operator forms).  The
// iteration is the one of pcg.cuh and every block product is formed in the same
// order; what differs is where the values live, and that the block sums group
// rows 2c and 2c + 1 of a thread where pcg.cuh groups rows t, t + T, ..., so that
// alpha and beta agree to a rounding of the double-float sum to FP32.
//
// pcg.cuh gives a thread single rows, takes one 32-bit shared-memory load per
// multiply-add and keeps every vector in shared memory.  With one problem of
// nx = 14, N = 64 on each SM that is 10,000 cycles per iteration at 42 % issue:
// 16,500 warp instructions, 41 % of them shared-memory or global accesses, and
// the latency of two block sums.  Here
//   - blocks are staged as 2 x 2 tiles (kernels.h) and a thread owns rows 2c,
//     2c + 1 of a block row: one 128-bit load brings four matrix entries,
//     whichever way the block is read, and a vector segment is read once for
//     two rows (a third of the load instructions);
//   - even and odd terms of a dot product are the two halves of a packed FP32
//     multiply-add where a tile holds them side by side (products by rows);
//   - the pair's entries of r, p, w, z, x and 1/q stay in registers; only r, p
//     and v pass through shared memory, and x and w have no vector there, so
//     that more problems fit whole (nx = 14, nu = 7: N <= 71 instead of 68).
// Measured (GB300; us per iteration with one problem on each SM, pcg.cuh
// before): nx = 14, N = 64: 4.74 -> 3.52; nx = 21, N = 30: 5.01 -> 3.56; nx = 4,
// N = 64: 2.20 -> 1.42, and 1520 of them at once 6.97 -> 4.41.  The sums are
// pcg.cuh's, renormalised after every addition: folding the low parts only at
// the end takes 5 % (nx = 14) to 15 % (nx = 4) less and leaves the sums 1.2
// times (terms of one sign) to 1.9 times as far from the exact ones.
// What bounds it: the shared-memory load pipe for the larger blocks (nx = 14, 512
// threads: 76 % busy; every matrix entry comes through it once per use, a quarter
// of the wavefronts are bank conflicts of tile loads by columns where a warp phase
// crosses a block row), the latency of five barriers and two block sums for the
// smaller ones (nx = 4: a third of the issue slots and 28 % of L1 busy).
#pragma once

#include "pcg.cuh"

namespace sspcg {

// Two values of adjacent rows (or columns).
struct Pair {
  float a, b;
  __device__ __forceinline__ static Pair load(const float *p) {  // p: an even index of a vector (8-byte aligned)
    const float2 v = *reinterpret_cast<const float2 *>(p);
    return {v.x, v.y};
  }
  __device__ __forceinline__ void store(float *p) const { *reinterpret_cast<float2 *>(p) = make_float2(a, b); }
};

// a.a b.a + a.b b.b
__device__ __forceinline__ df dot(Pair a, Pair b) {
  const float p = __fmul_rn(a.a, b.a);
  return df_fma(df{p, __fmaf_rn(a.a, b.a, -p)}, a.b, b.b);
}

// (a.x b.x + c.x, a.y b.y + c.y), each rounded once as fmaf: one instruction for two FP32 multiply-adds.
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)),
        "l"(*reinterpret_cast<unsigned long long *>(&c)));
  return *reinterpret_cast<float2 *>(&d);
}

// Accumulators of one dot product as in dot_seg (pcg.cuh): even and odd terms, each in increasing order.
struct Acc {
  float2 v = make_float2(0.0f, 0.0f);
  __device__ __forceinline__ void add(float m0, float m1, float s0, float s1) {
    v = ffma2(make_float2(m0, m1), make_float2(s0, s1), v);
  }
  __device__ __forceinline__ void add_even(float m, float s) { v.x = fmaf(m, s, v.x); }
  __device__ __forceinline__ void add_odd(float m, float s) { v.y = fmaf(m, s, v.y); }
  __device__ __forceinline__ float sum() const { return v.x + v.y; }
};

__device__ __forceinline__ float4 load_tile(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// Rows 2q, 2q+1 of M times seg; t: the block's tile row q.
template <int NX>
__device__ __forceinline__ Pair tile_rows(const float *t, const float *seg) {
  Acc r0, r1;
#pragma unroll
  for (int c = 0; c < NX; c += 2) {
    const float4 m = load_tile(t + 2 * c);
    if (c + 1 < NX) {
      r0.add(m.x, m.y, seg[c], seg[c + 1]);
      r1.add(m.z, m.w, seg[c], seg[c + 1]);
    } else {
      r0.add_even(m.x, seg[c]);
      r1.add_even(m.z, seg[c]);
    }
  }
  return {r0.sum(), r1.sum()};
}

// Rows 2c, 2c+1 of M^T times seg; t: the block's tile column c (tile rows ld values apart).
template <int NX>
__device__ __forceinline__ Pair tile_cols(const float *t, int ld, const float *seg) {
  Acc r0, r1;
#pragma unroll
  for (int q = 0; q < NX; q += 2) {
    const float4 m = load_tile(t + (q >> 1) * ld);
    r0.add_even(m.x, seg[q]);
    r1.add_even(m.y, seg[q]);
    if (q + 1 < NX) {
      r0.add_odd(m.z, seg[q + 1]);
      r1.add_odd(m.w, seg[q + 1]);
    }
  }
  return {r0.sum(), r1.sum()};
}

// Staging: nblk dense row-major blocks of NX x w (global) into tiles in shared memory, ``blk`` elements per
// block; TRANS: each (square) block transposed.  With a 16-byte aligned source (the packed layout aligns every
// problem's arrays) each thread takes 16 consecutive bytes per load and scatters the four values into the tiles;
// the rest, or an unaligned source, one element at a time.  The row and column past an odd NX or w are zeroed.
template <int NX, bool TRANS>
__device__ __forceinline__ void stage_tiles(float *dst, const float *src, int nblk, int w, int blk, int tid, int nthr) {
  const int ld4 = 4 * tile_ld(w);  // elements of a tile row
  const int count = nblk * NX * w;
  auto put = [&](int k, int i, int c, float v) {
    if (TRANS) { const int t = i; i = c; c = t; }
    dst[k * blk + (i >> 1) * ld4 + (c >> 1) * 4 + (i & 1) * 2 + (c & 1)] = v;
  };
  int done = 0;
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    const int nv = count / 4;
    const float4 *s4 = reinterpret_cast<const float4 *>(src);
    for (int v = tid; v < nv; v += nthr) {
      const float4 c4 = __ldg(s4 + v);
      const float vals[4] = {c4.x, c4.y, c4.z, c4.w};
      const int e = 4 * v;
      int r = e / w, col = e - r * w;
      int k = r / NX, i = r - k * NX;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        put(k, i, col, vals[q]);
        if (++col == w) {
          col = 0;
          if (++i == NX) { i = 0; ++k; }
        }
      }
    }
    done = 4 * nv;
  }
  for (int e = done + tid; e < count; e += nthr) {
    const int r = e / w, col = e - r * w;
    const int k = r / NX;
    put(k, r - k * NX, col, __ldg(src + e));
  }
  if (NX & 1) {  // the row past the last
    const int wp = (w + 1) & ~1;
    for (int e = tid; e < nblk * wp; e += nthr) put(e / wp, NX, e % wp, 0.0f);
  }
  if (w & 1)  // the column past the last
    for (int e = tid; e < nblk * NX; e += nthr) put(e / NX, e % NX, w, 0.0f);
}


template <int NX, int OP>
__device__ void pcg_one_solve(const PcgArgs &a, const ProbDesc &d, float *sm, df *slots) {
  using Sum = Red<kRedDf, float>;
  constexpr int NXP = (NX + 3) & ~3;
  constexpr int H = (NX + 1) / 2;     // row pairs of a block row
  constexpr int LD4 = 4 * (H | 1);    // values of a tile row of an nx x nx block
  constexpr int BLK = H * LD4;        // values of an nx x nx block
  constexpr int NUC = (NX + 1) / 2;   // nu = ceil(nx / 2), the usual input count: unrolled B-row products
  const int p = d.id;                 // output slot
  const int N = d.N, n = N + 1, nu = d.nu, R = n * NX, NUP = vec_stride(nu);
  const int hu = tile_half(nu), ldb4 = 4 * tile_ld(nu), blkb = tile_block(NX, nu);
  const int tid = (int)threadIdx.x, T = (int)blockDim.x;
  const OneLayout L = pcg_one_layout(OP, N, NX, nu);
  float *sp = sm + L.p, *sr = sm + L.r, *sv = sm + L.v, *svu = sm + L.vu, *siq = sm + L.iq, *sir = sm + L.ir;
  float *s0 = sm + L.m0, *s1 = sm + L.m1, *spd = sm + L.pd, *spe = sm + L.pe;
  // no off-diagonal preconditioner blocks (PE == nullptr): the preconditioner is block-diagonal
  const bool diag_only = a.PE == nullptr;
  const float *gam = a.gamma + d.ovec;
  float *lam = reinterpret_cast<float *>(a.lambda) + d.ovec;

  // The vectors, their zero segments before block row 0 and after block row N, and 1/q, 1/r start as zeros: the
  // entry past an odd nx (or nu) of a block row takes part in the pair arithmetic and stays zero.
  for (int e = tid; e < (int)L.m0; e += T) sm[e] = 0.0f;
  // a single knot has one zero off-diagonal slot of each kind
  auto zero = [&](float *s, int count) {
    for (int e = tid; e < count; e += T) s[e] = 0.0f;
  };
  if (N == 0) {
    if (OP == kOpQp) zero(s0, BLK);
    zero(s1, OP == kOpQp ? blkb : BLK);
    if (!diag_only) zero(spe, BLK);
  }
  __syncthreads();
  // PD and D are stored transposed: their products read by columns are then read by tile rows
  stage_tiles<NX, true>(spd, reinterpret_cast<const float *>(a.PD) + d.odiag, n, NX, BLK, tid, T);
  if (!diag_only) stage_tiles<NX, false>(spe, reinterpret_cast<const float *>(a.PE) + d.ooff, N, NX, BLK, tid, T);
  if constexpr (OP == kOpQp) {
    stage_tiles<NX, false>(s0, a.A + d.oA, N, NX, BLK, tid, T);
    if (nu > 0) stage_tiles<NX, false>(s1, a.B + d.oB, N, nu, blkb, tid, T);
    for (int e = tid; e < R; e += T) {
      const int k = e / NX, j = e - k * NX;
      siq[k * NXP + j] = 1.0f / a.qd[d.oq + e];
    }
    for (int e = tid; e < N * nu; e += T) {
      const int k = e / nu, j = e - k * nu;
      sir[k * NUP + j] = 1.0f / a.rd[d.orr + e];
    }
  } else {
    stage_tiles<NX, true>(s0, a.D + d.odiag, n, NX, BLK, tid, T);
    stage_tiles<NX, false>(s1, a.E + d.ooff, N, NX, BLK, tid, T);
  }

  // this thread's row pair c of block row k: rows 2c and 2c + 1 (the second past the end of an odd nx for c = H - 1)
  const bool on = tid < n * H;
  const int k = on ? tid / H : 0, c = on ? tid - k * H : 0, si = k * NXP + 2 * c, row = k * NX + 2 * c;
  const bool two = on && (NX % 2 == 0 || 2 * c + 1 < NX);
  const int km = k > 0 ? k - 1 : 0;                      // off-diagonal blocks, clamped into range: the segment they
  const int kp = k < N ? k : (N > 0 ? N - 1 : 0);        // multiply at the ends is zero (as in bt_row, pcg.cuh)

  // The thread's pair of a block-tridiagonal symmetric matrix times v (bt_row).
  auto bt_pair = [&](const float *Md, const float *Mo, const float *v) -> Pair {
    Seg<NX, float> v0, v1, v2;
    v0.load(v + k * NXP);
    v1.load(v + (k - 1) * NXP);
    v2.load(v + (k + 1) * NXP);
    const Pair da = tile_rows<NX>(Md + k * BLK + c * LD4, v0.v);
    const Pair db = tile_rows<NX>(Mo + km * BLK + c * LD4, v1.v);
    const Pair dc = tile_cols<NX>(Mo + kp * BLK + c * 4, LD4, v2.v);
    return {(da.a + db.a) + dc.a, (da.b + db.b) + dc.b};
  };
  auto apply_P = [&]() -> Pair {
    if (!diag_only) return bt_pair(spd, spe, sr);
    Seg<NX, float> s;
    s.load(sr + k * NXP);
    return tile_rows<NX>(spd + k * BLK + c * LD4, s.v);
  };
  // QP form, phase 1 (apply_S_phase1): v = G^-1 C^T src, x: the thread's pair of src; ends with a barrier.  The
  // column pairs of the B_k go to the threads from the last one down, which the row pairs may leave idle.
  const float inv_hu = hu > 0 ? 1.0f / (float)hu : 0.0f;
  auto phase1 = [&](const float *src, Pair x, Pair iq) {
    if constexpr (OP == kOpQp) {
      Seg<NX, float> s;
      if (on) {
        s.load(src + (k + 1) * NXP);
        const Pair ax = tile_cols<NX>(s0 + kp * BLK + c * 4, LD4, s.v);
        Pair{(-x.a + ax.a) * iq.a, (-x.b + ax.b) * iq.b}.store(sv + si);
      }
      for (int it = T - 1 - tid; it < N * hu; it += T) {
        const int kk = (int)(((float)it + 0.5f) * inv_hu), cc = it - kk * hu;
        s.load(src + (kk + 1) * NXP);
        const Pair bx = tile_cols<NX>(s1 + kk * blkb + cc * 4, ldb4, s.v), ir = Pair::load(sir + kk * NUP + 2 * cc);
        Pair{bx.a * ir.a, bx.b * ir.b}.store(svu + kk * NUP + 2 * cc);
      }
      __syncthreads();
    }
  };
  // The thread's pair of S src (QP form: of C v; apply_S_row).
  auto apply_S = [&](const float *src) -> Pair {
    if constexpr (OP == kOpQp) {
      Seg<NX, float> s;
      s.load(sv + (k - 1) * NXP);
      const Pair ax = tile_rows<NX>(s0 + km * BLK + c * LD4, s.v);
      Pair ab{0.0f, 0.0f};  // B terms: one accumulator per row, in order
      const float *vu = svu + (k - 1) * NUP, *tb = s1 + km * blkb + c * ldb4;
      auto b_tile = [&](int j, float v0, float v1, bool last) {  // last: nu is odd and j + 1 = nu
        const float4 m = load_tile(tb + 2 * j);
        ab = {fmaf(m.x, v0, ab.a), fmaf(m.z, v0, ab.b)};
        if (!last) ab = {fmaf(m.y, v1, ab.a), fmaf(m.w, v1, ab.b)};
      };
      if (nu == NUC) {  // unrolled, v_u in registers
        Seg<NUC, float> su;
        su.load(vu);
#pragma unroll
        for (int j = 0; j < NUC; j += 2) b_tile(j, su.v[j], su.v[j + 1], j + 1 >= NUC);
      } else {
        for (int j = 0; j < nu; j += 2) {
          const Pair v = Pair::load(vu + j);
          b_tile(j, v.a, v.b, j + 1 >= nu);
        }
      }
      const Pair vx = Pair::load(sv + si);
      return {(-vx.a + ax.a) + ab.a, (-vx.b + ax.b) + ab.b};
    } else {
      return bt_pair(s0, s1, src);
    }
  };

  // ---- r0 = gamma - S x0 ----
  Pair g{0.0f, 0.0f}, x = g, r, pv = g, w = g;
  if (on) {
    g = {gam[row], two ? gam[row + 1] : 0.0f};
    if (a.warm) {
      x = {lam[row], two ? lam[row + 1] : 0.0f};
      x.store(sp + si);
    }
  }
  r = g;
  df g1[1] = {dot(g, g)};
  block_sum<Sum, 1>(g1, slots);  // contains a barrier: staged blocks, reciprocals and sp complete
  const float gg = Sum::get(g1[0]);
  const float thresh = a.tol2 * gg;
  const int max_iter = a.max_iter > 0 ? a.max_iter : 10 * n * NX;
  if (gg == 0.0f) {
    if (on) lam[row] = 0.0f;
    if (two) lam[row + 1] = 0.0f;
    if (tid == 0) { a.iters[p] = 0; a.relres[p] = 0.0; a.status[p] = kOk; }
    __syncthreads();
    return;
  }
  const Pair iq = OP == kOpQp && on ? Pair::load(siq + si) : Pair{0.0f, 0.0f};
  bool warm = a.warm != 0;
  if (warm) {
    phase1(sp, x, iq);
    if (on) {
      w = apply_S(sp);
      r = {g.a - w.a, g.b - w.b};
    }
  }
  if (on) r.store(sr + si);
  __syncthreads();

  // ---- iterations ----
  float rz = 0.0f, rr = 0.0f;
  int it = 0, code = kOk;
  bool first = true;
  while (true) {
    // z = Phi^-1 r, r.z, r.r
    Pair z{0.0f, 0.0f};
    if (on) z = apply_P();
    df s2[2] = {dot(r, z), dot(r, r)};
    block_sum<Sum, 2>(s2, slots + 64);
    const float rz_old = rz;
    rz = Sum::get(s2[0]);
    rr = Sum::get(s2[1]);
    if (first) {
      if (warm && a.warm == 2 && !(rr < gg)) {  // warm start no better than zero: restart from lambda_0 = 0
        warm = false;
        x = {0.0f, 0.0f};
        r = g;
        if (on) r.store(sr + si);
        __syncthreads();
        continue;
      }
      first = false;
      pv = z;
    } else {
      const float beta = rz / rz_old;
      pv = {fmaf(beta, pv.a, z.a), fmaf(beta, pv.b, z.b)};
      ++it;
    }
    if (!(rr > thresh)) {
      if (!isfinite(rr)) code = kNonFinite;
      break;
    }
    if (it >= max_iter) { code = kMaxIter; break; }
    if (on) pv.store(sp + si);
    __syncthreads();
    // w = S p, p.w
    phase1(sp, pv, iq);
    if (on) w = apply_S(sp);
    df s1v[1] = {dot(pv, w)};
    block_sum<Sum, 1>(s1v, slots);
    const float pw = Sum::get(s1v[0]);
    if (!(pw > 0.0f) || !isfinite(pw)) { code = isfinite(pw) ? kBreakdown : kNonFinite; break; }
    const float alpha = rz / pw;
    x = {fmaf(alpha, pv.a, x.a), fmaf(alpha, pv.b, x.b)};
    r = {fmaf(-alpha, w.a, r.a), fmaf(-alpha, w.b, r.b)};
    if (on) r.store(sr + si);
    __syncthreads();
  }
  if (on) lam[row] = x.a;
  if (two) lam[row + 1] = x.b;
  if (tid == 0) {
    a.iters[p] = it;
    a.relres[p] = sqrt((double)rr / (double)gg);
    a.status[p] = code;
  }
  __syncthreads();
}

// Resident 512-thread CTAs per SM that the register allocation aims at: small blocks need few registers, and their
// problems run several to an SM.
template <int NX>
constexpr int one_min_ctas() { return NX <= 8 ? 2 : 1; }

// Persistent kernel: CTAs take problems from the work list as in pcg_kernel.
template <int NX, int OP>
__global__ void __launch_bounds__(512, one_min_ctas<NX>()) pcg_one_kernel(PcgArgs a) {
  extern __shared__ float4 smem4[];
  __shared__ __align__(16) df slots[4 * 32];
  __shared__ int s_next;
  for (int w = blockIdx.x;; w += gridDim.x) {
    if (a.counter) {
      if (threadIdx.x == 0) s_next = atomicAdd(a.counter, 1);
      __syncthreads();
      w = s_next;
      __syncthreads();
    }
    if (w >= a.nwork) break;
    const ProbDesc d = a.ps.get(a.work ? a.work[w] : w);
    if (a.status[d.id] != kOk) continue;  // preconditioner failed for this problem
    pcg_one_solve<NX, OP>(a, d, reinterpret_cast<float *>(smem4), slots);
  }
}

template <int NX, int OP>
struct PcgOneVariant {
  static cudaError_t prepare() {
    static std::atomic<uint64_t> attr_done{0};
    return smem_attr_once(attr_done, pcg_one_kernel<NX, OP>, pcg_max_smem_bytes());
  }
  static cudaError_t launch(const PcgArgs &a, int grid, int block, size_t smem, cudaStream_t st) {
    cudaError_t e = prepare();
    if (e != cudaSuccess) return e;
    pcg_one_kernel<NX, OP><<<grid, block, smem, st>>>(a);
    return cudaGetLastError();
  }
  static cudaError_t occupancy(int block, size_t smem, int *ctas) {
    cudaError_t e = prepare();
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, pcg_one_kernel<NX, OP>, block, smem);
  }
};

}  // namespace sspcg
