// Warm-start network products on the 5th-generation tensor cores:
// C[M][N] = epilogue(A[M][K] B[N][K]^T), bf16 operands, FP32 accumulation in
// tensor memory.  One CTA (4 warps) per MT x 128 rows and N (256, 64 or 32)
// columns of C: warp 0 streams A and B tiles of 64 columns (128 bytes) into a ring of
// shared-memory stages with TMA (128-byte swizzle); warp 1 issues
// tcgen05.mma (M = 128, K = 16 per instruction) from one thread and
// releases each stage with tcgen05.commit; then all four warps read the
// accumulators (tcgen05.ld, one TMEM lane per row) and apply the epilogue.
// Every mbarrier wait is bounded: on expiry the kernel records an error code,
// skips its remaining work, waits (bounded again) for its copies and products
// in flight, frees its tensor memory and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include "mlp.h"

namespace sspcg {
namespace mlp {
namespace {

constexpr int kTcM = 128;          // rows per tile (TMEM lanes)
constexpr int kTcK = 64;           // columns per stage: one 128-byte swizzle row of bf16
constexpr int kTcThreads = 128;
#ifndef SSPCG_TC_POLLS
#define SSPCG_TC_POLLS (1u << 26)
#endif
constexpr uint32_t kSpinLimit = SSPCG_TC_POLLS;  // polls of one mbarrier wait (well over a second)
constexpr uint32_t kDrainLimit = 1u << 26;       // of the waits that follow one that ran out

__device__ __forceinline__ uint32_t su32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(su32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(su32(bar)), "r"(bytes) : "memory");
}

// Wait until the phase of parity ``parity`` has completed; false when the bound expires.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint32_t limit = kSpinLimit) {
  const uint32_t a = su32(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];\n" ::"r"(su32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(su32(bar))
      : "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(const void *p) {
  const uint64_t addr = su32(p);
  uint64_t d = 0;
  d |= (addr >> 4) & 0x3FFFull;            // start address
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset: next 8-row group
  d |= (uint64_t)1 << 46;                  // descriptor version
  d |= (uint64_t)2 << 61;                  // 128-byte swizzle
  return d;
}

// Instruction descriptor of kind::f16: bf16 A and B (K-major), FP32 accumulator, M x N.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N) {
  return (1u << 4)                       // accumulator format F32
         | (1u << 7)                     // A format BF16
         | (1u << 10)                    // B format BF16
         | ((uint32_t)(N >> 3) << 17)    // N / 8
         | ((uint32_t)(M >> 4) << 24);   // M / 16
}

__device__ __forceinline__ void mma_issue(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
          tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(su32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

template <int N, int MT>
struct TcCfg {
  static constexpr int kStages = N >= 256 ? (MT == 2 ? 3 : 4) : N == 64 ? 8 : 6;
  static constexpr int kABytes = MT * kTcM * kTcK * 2;  // 16 KB per 128 rows
  static constexpr int kBBytes = N * kTcK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kTmemCols = MT * N;  // power of two >= 32
  static constexpr int kSmem = kStages * kStageBytes + 1024 /*alignment*/ + 256 /*barriers*/;
};

template <int N, int EPI, int MT>
__global__ void __launch_bounds__(kTcThreads, 1)
    gemm_nt_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, int64_t M,
                      int K, int ldc, const float *__restrict__ bias, bf16 *__restrict__ Cb, float *__restrict__ Cf,
                      int *__restrict__ err) {
  using C = TcCfg<N, MT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *stage_base = smem;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::kStages * C::kStageBytes);
  uint64_t *empty = full + C::kStages;
  uint64_t *acc_full = empty + C::kStages;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_full + 1);
  __shared__ int failed;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t m0 = (int64_t)blockIdx.x * kTcM * MT;
  const int n0 = blockIdx.y * N;  // first column of C
  const int KT = K / kTcK;

  if (threadIdx.x == 0) {
    failed = 0;
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(tmem_slot)),
                 "r"(C::kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  int issued = 0;  // the producer's stages on their way

  if (warp == 0 && lane == 0) {
    // producer: TMA loads of A rows [m0, m0 + 128 MT) and B rows [n0, n0 + N), 64 columns per stage
    for (int kt = 0; kt < KT; ++kt) {
      const int s = kt % C::kStages;
      if (kt >= C::kStages && !mbar_wait(&empty[s], ((kt / C::kStages) - 1) & 1)) {
        atomicExch(&failed, 1);
        break;
      }
      uint8_t *a = stage_base + s * C::kStageBytes;
      uint8_t *b = a + C::kABytes;
      mbar_expect_tx(&full[s], C::kStageBytes);
#pragma unroll
      for (int t = 0; t < MT; ++t)
        tma_load_2d(a + t * (C::kABytes / MT), &mapA, kt * kTcK, (int)m0 + t * kTcM, &full[s]);
      tma_load_2d(b, &mapB, kt * kTcK, n0, &full[s]);
      issued = kt + 1;
    }
  } else if (warp == 1 && lane == 0) {
    // MMA issuer
    constexpr uint32_t idesc = instr_desc(kTcM, N);
    bool ok = true;
    for (int kt = 0; kt < KT && ok; ++kt) {
      const int s = kt % C::kStages;
      if (!mbar_wait(&full[s], (kt / C::kStages) & 1)) {
        atomicExch(&failed, 1);
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const uint8_t *a = stage_base + s * C::kStageBytes;
      const uint8_t *b = a + C::kABytes;
#pragma unroll
      for (int t = 0; t < MT; ++t)
#pragma unroll
        for (int k = 0; k < kTcK / 16; ++k)
          mma_issue(tmem + t * N, smem_desc(a + t * (C::kABytes / MT) + k * 32), smem_desc(b + k * 32), idesc,
                    (kt > 0 || k > 0) ? 1u : 0u);
      mma_commit(&empty[s]);  // stage free once these products have read it
    }
    mma_commit(acc_full);  // accumulators complete
  }
  __syncwarp();

  // epilogue: warp w owns TMEM lanes (rows) 32w .. 32w + 31
  bool ready = mbar_wait(acc_full, 0);
  if (!ready) atomicExch(&failed, 1);
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (!failed) {
    const uint32_t tbase = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int cc = 0; cc < MT * N; cc += 16) {
      const int c0 = n0 + cc % N;
      const int64_t row = m0 + cc / N * kTcM + warp * 32 + lane;
      float v[16];
      tmem_ld16(tbase + (uint32_t)cc, v);
      if (row < M) {
        if (EPI == kEpiBiasRelu) {
          uint32_t packed[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float x0 = fmaxf(v[2 * i] + bias[c0 + 2 * i], 0.f);
            const float x1 = fmaxf(v[2 * i + 1] + bias[c0 + 2 * i + 1], 0.f);
            const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
            packed[i] = *reinterpret_cast<const uint32_t *>(&h);
          }
          uint4 *dst = reinterpret_cast<uint4 *>(Cb + row * ldc + c0);
          dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
          dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
        } else {
          float4 *dst = reinterpret_cast<float4 *>(Cf + row * ldc + c0);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            dst[i] = make_float4(v[4 * i] + bias[c0 + 4 * i], v[4 * i + 1] + bias[c0 + 4 * i + 1],
                                 v[4 * i + 2] + bias[c0 + 4 * i + 2], v[4 * i + 3] + bias[c0 + 4 * i + 3]);
        }
      }
    }
  } else if (threadIdx.x == 0) {  // what is in flight ends before the shared and the tensor memory go
    for (int kt = issued > C::kStages ? issued - C::kStages : 0; kt < issued; ++kt)
      mbar_wait(&full[kt % C::kStages], (kt / C::kStages) & 1, kDrainLimit);
    mbar_wait(acc_full, 0, kDrainLimit);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(C::kTmemCols));
  }
  if (threadIdx.x == 0 && failed) atomicExch(err, 1);
}

// ---------------------------------------------------------------------------
// Inference after its first layer, in one kernel:
//   lambda0 = rows of (relu(H1 W2^T + b2) W3^T + b3), H1 [M][256] of a span.
// As separate products and a scatter these were three launches that write and
// read H2 (0.5 KB per row each way) and Y, and the 256-column one spent its time
// between tiles: four stages of K, then an epilogue that nothing overlapped.
// Here a CTA per SM keeps both weight matrices (144 KB) in shared memory and
// walks the row tiles: TMA brings 128 rows of H1, the epilogue of the second
// layer writes H2 over them as the third layer's operand (128-byte swizzle: the
// 16-byte piece p of row r lies at piece p ^ (r % 8)), and the third layer's
// epilogue writes lambda0.  The next tile's H1 is on its way meanwhile.  The
// products and roundings are those of gemm_nt_tc_kernel in the same order, so
// lambda0 is bit-identical.  266,240 rows: 208 us in three launches before,
// 82 us now, bound by the serial chain of a tile: load, two products, two epilogues.
// ---------------------------------------------------------------------------
constexpr int kTailThreads = 256;  // eight warps: two per quarter of the TMEM lanes
constexpr int kTailKT = kHid / kTcK;
// bytes per 64 columns
constexpr int kTailABytes = kTcM * kTcK * 2, kTailW2Bytes = kHid * kTcK * 2, kTailW3Bytes = kOut * kTcK * 2;
constexpr int kTailSmem = kTailKT * (kTailABytes + kTailW2Bytes + kTailW3Bytes) + 1024 /*alignment*/;

__global__ void __launch_bounds__(kTailThreads, 1)
    tail_tc_kernel(const __grid_constant__ CUtensorMap mapH, const __grid_constant__ CUtensorMap mapW2,
                   const __grid_constant__ CUtensorMap mapW3, RowSpan rs, const float *__restrict__ b2,
                   const float *__restrict__ b3, float *__restrict__ lambda, int *__restrict__ err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *sW2 = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sA = sW2 + kTailKT * kTailW2Bytes, *sW3 = sA + kTailKT * kTailABytes;
  __shared__ uint64_t bar_w, bar_a, bar_2, bar_3;  // weights and H1 arrived; second and third layer done
  __shared__ uint32_t tmem_slot;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t tiles = (rs.nrows + kTcM - 1) / kTcM;
  const bool first = threadIdx.x == 0;
  auto load_tile = [&](int64_t tile) {
    mbar_expect_tx(&bar_a, kTailKT * kTailABytes);
    for (int kt = 0; kt < kTailKT; ++kt)
      tma_load_2d(sA + kt * kTailABytes, &mapH, kt * kTcK, (int)(tile * kTcM), &bar_a);
  };

  if (first) {
    mbar_init(&bar_w, 1);
    mbar_init(&bar_a, 1);
    mbar_init(&bar_2, 1);
    mbar_init(&bar_3, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    mbar_expect_tx(&bar_w, kTailKT * (kTailW2Bytes + kTailW3Bytes));
    for (int kt = 0; kt < kTailKT; ++kt) {
      tma_load_2d(sW2 + kt * kTailW2Bytes, &mapW2, kt * kTcK, 0, &bar_w);
      tma_load_2d(sW3 + kt * kTailW3Bytes, &mapW3, kt * kTcK, 0, &bar_w);
    }
    load_tile(blockIdx.x);  // the grid is at most the tiles
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(su32(&tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = tmem_slot, acc3 = tmem + kHid;  // accumulators: columns 0-255 and 256-287
  const int quarter = warp & 3, r = quarter * 32 + lane;
  const uint32_t tlane = (uint32_t)(quarter * 32) << 16;
  bool ok = true, second = false, third = false;  // thread 0: this tile's products have been issued
  uint32_t parity = 0;
  for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, parity ^= 1) {
    if (first) {
      third = false;
      second = ok = mbar_wait(&bar_w, 0) && mbar_wait(&bar_a, parity);
      if (ok) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        for (int kt = 0; kt < kTailKT; ++kt)
#pragma unroll
          for (int k = 0; k < kTcK / 16; ++k)
            mma_issue(tmem, smem_desc(sA + kt * kTailABytes + k * 32), smem_desc(sW2 + kt * kTailW2Bytes + k * 32),
                      instr_desc(kTcM, kHid), (kt > 0 || k > 0) ? 1u : 0u);
        mma_commit(&bar_2);
      }
    }
    __syncwarp();
    ok = mbar_wait(&bar_2, parity) && ok;
    ok = __all_sync(0xffffffffu, ok);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (ok) {
      // H2 over H1, which the second layer has read
#pragma unroll 1
      for (int c0 = (warp >> 2) * (kHid / 2); c0 < ((warp >> 2) + 1) * (kHid / 2); c0 += 16) {
        float v[16];
        tmem_ld16(tmem + tlane + (uint32_t)c0, v);
        uint32_t packed[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(fmaxf(v[2 * i] + __ldg(b2 + c0 + 2 * i), 0.f),
                                                         fmaxf(v[2 * i + 1] + __ldg(b2 + c0 + 2 * i + 1), 0.f));
          packed[i] = *reinterpret_cast<const uint32_t *>(&h);
        }
        uint8_t *row = sA + (c0 / kTcK) * kTailABytes + r * 128;
        const int piece = (c0 % kTcK) / 8;
        *reinterpret_cast<uint4 *>(row + ((piece ^ (r & 7)) << 4)) =
            make_uint4(packed[0], packed[1], packed[2], packed[3]);
        *reinterpret_cast<uint4 *>(row + (((piece + 1) ^ (r & 7)) << 4)) =
            make_uint4(packed[4], packed[5], packed[6], packed[7]);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
    if (first) {
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      for (int kt = 0; kt < kTailKT; ++kt)
#pragma unroll
        for (int k = 0; k < kTcK / 16; ++k)
          mma_issue(acc3, smem_desc(sA + kt * kTailABytes + k * 32), smem_desc(sW3 + kt * kTailW3Bytes + k * 32),
                    instr_desc(kTcM, kOut), (kt > 0 || k > 0) ? 1u : 0u);
      mma_commit(&bar_3);
      third = true;
    }
    __syncwarp();
    ok = __all_sync(0xffffffffu, mbar_wait(&bar_3, parity));
    if (__syncthreads_or(!ok)) {
      ok = false;
      break;
    }
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (first && tile + gridDim.x < tiles) load_tile(tile + gridDim.x);  // the third layer has read H2
    __syncwarp();
    if (warp < 4) {
      float v[32];
      tmem_ld16(acc3 + tlane, *reinterpret_cast<float(*)[16]>(v));
      tmem_ld16(acc3 + tlane + 16, *reinterpret_cast<float(*)[16]>(v + 16));
      const int64_t row = tile * kTcM + r;
      if (row < rs.nrows) {
        const int2 ref = rs.kref[rs.row0 + row];
        const ProbDesc d = rs.ps.get(ref.x);
        float *o = lambda + d.ovec + (int64_t)ref.y * d.nx;
#pragma unroll
        for (int i = 0; i < kPadX; ++i)
          if (i < d.nx) o[i] = v[i] + __ldg(b3 + i);
      }
    }
  }
  if (first && !ok) {  // what is in flight ends before the shared and the tensor memory go
    mbar_wait(&bar_w, 0, kDrainLimit);
    mbar_wait(&bar_a, parity, kDrainLimit);
    if (second) mbar_wait(&bar_2, parity, kDrainLimit);
    if (third) mbar_wait(&bar_3, parity, kDrainLimit);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512));
  }
  if (first && !ok) atomicExch(err, 1);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// 2-D bf16 tensor [rows][cols] (row-major), box of kTcK columns x box_rows rows, 128-byte swizzle.
bool make_map(CUtensorMap *map, const bf16 *base, int64_t rows, int cols, int box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * sizeof(bf16)};
  const cuuint32_t box[2] = {(cuuint32_t)kTcK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int N, int EPI, int MT>
cudaError_t launch_tc(const CUtensorMap &ma, const CUtensorMap &mb, int64_t M, int ldc, int K, const float *bias,
                      bf16 *Cb, float *Cf, int *err, cudaStream_t st) {
  using C = TcCfg<N, MT>;
  static std::atomic<uint64_t> attr_done{0};
  cudaError_t e = smem_attr_once(attr_done, gemm_nt_tc_kernel<N, EPI, MT>, C::kSmem);
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned)((M + MT * kTcM - 1) / (MT * kTcM)), (unsigned)(ldc / N));
  gemm_nt_tc_kernel<N, EPI, MT><<<grid, kTcThreads, C::kSmem, st>>>(ma, mb, M, K, ldc, bias, Cb, Cf, err);
  return cudaGetLastError();
}

}  // namespace

bool tc_available() { return encode_fn() != nullptr; }

cudaError_t launch_gemm_nt_tc(int epi, const bf16 *A, const bf16 *B, int64_t M, int N, int K, const float *bias,
                              bf16 *Cb, float *Cf, int *err, cudaStream_t st, int sms) {
  if (M <= 0) return cudaSuccess;
  if (K % kTcK != 0 || K <= 0) return cudaErrorInvalidValue;
  if (!(N == 256 || N == 32)) return cudaErrorInvalidValue;
  if (!(epi == kEpiBiasRelu || epi == kEpiBiasF32)) return cudaErrorInvalidValue;
  // TMA needs 16-byte aligned bases and row strides (K * 2 bytes: K % 64 == 0)
  if ((reinterpret_cast<uintptr_t>(A) & 15u) || (reinterpret_cast<uintptr_t>(B) & 15u)) return cudaErrorInvalidValue;
  // Few row tiles: each stage of a 256-column CTA is 48 KB, which one SM takes in at its own rate however idle the
  // others are, so four CTAs share a row tile's columns as long as all of them run at once.  2,080 rows: the
  // training step 156.8 to 144.6 us.
  const int64_t tiles = (M + kTcM - 1) / kTcM;
  const bool quarter = N == 256 && epi == kEpiBiasRelu && 4 * tiles <= sms;
  CUtensorMap ma, mb;
  if (!make_map(&ma, A, M, K, kTcM) || !make_map(&mb, B, N, K, quarter ? 64 : N)) return cudaErrorInvalidValue;
  if (quarter) return launch_tc<64, kEpiBiasRelu, 1>(ma, mb, M, N, K, bias, Cb, Cf, err, st);
  // Two row tiles per CTA share each stage's B rows (256 KB instead of 384 KB of L2 reads per 128 rows and 256 columns,
  // which is what bounds the first layer), once one tile per CTA no longer fits on the SMs in one wave.
  const bool pair = M > (int64_t)kTcM * sms;
  if (N == 256 && epi == kEpiBiasRelu && pair)
    return launch_tc<256, kEpiBiasRelu, 2>(ma, mb, M, N, K, bias, Cb, Cf, err, st);
  if (N == 256)
    return epi == kEpiBiasRelu ? launch_tc<256, kEpiBiasRelu, 1>(ma, mb, M, N, K, bias, Cb, Cf, err, st)
                               : launch_tc<256, kEpiBiasF32, 1>(ma, mb, M, N, K, bias, Cb, Cf, err, st);
  return epi == kEpiBiasRelu ? launch_tc<32, kEpiBiasRelu, 1>(ma, mb, M, N, K, bias, Cb, Cf, err, st)
                             : launch_tc<32, kEpiBiasF32, 1>(ma, mb, M, N, K, bias, Cb, Cf, err, st);
}

cudaError_t launch_tail_tc(const RowSpan &rs, const bf16 *H1, const bf16 *W2, const float *b2, const bf16 *W3,
                           const float *b3, float *lambda, int *err, cudaStream_t st, int sms) {
  if (rs.nrows <= 0) return cudaSuccess;
  CUtensorMap mh, m2, m3;
  if (!make_map(&mh, H1, rs.nrows, kHid, kTcM) || !make_map(&m2, W2, kHid, kHid, kHid) ||
      !make_map(&m3, W3, kOut, kHid, kOut))
    return cudaErrorInvalidValue;
  static std::atomic<uint64_t> attr_done{0};
  cudaError_t e = smem_attr_once(attr_done, tail_tc_kernel, kTailSmem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (rs.nrows + kTcM - 1) / kTcM;
  tail_tc_kernel<<<(unsigned)(tiles < sms ? tiles : sms), kTailThreads, kTailSmem, st>>>(mh, m2, m3, rs, b2, b3, lambda,
                                                                                         err);
  return cudaGetLastError();
}

}  // namespace mlp
}  // namespace sspcg
