// The PCG launches of one nx: the compiled variants and the dispatch among them.
#pragma once

#include "pcg.cuh"
#include "pcg_one.cuh"

namespace sspcg {

// The variant of one nx for an operator form, reduction mode and precision: FP32 with three reduction modes
// for both operator forms, and the FP64 path (QP form, FP64 reductions); vectors in a global workspace (gv)
// for the QP form only; single-reduction PCG (cg) for the QP form with FP32 arithmetic and double-float sums.
// f(PcgVariant<...>{}) is called on it; cudaErrorInvalidValue when no variant exists.
// warp: one problem per warp, for the QP form with textbook PCG: FP32 with double-float sums, and the FP64
// path.  one: a thread per row pair (pcg_one.cuh), both operator forms.
template <int NX, typename F>
cudaError_t with_pcg_variant(int op, int red, bool f64, bool gv, bool cg, bool warp, bool one, F &&f) {
  if (one) {
    if (f64 || gv || warp || red != kRedDf || (cg && op == kOpQp)) return cudaErrorInvalidValue;
    if (op == kOpBlock) return f(PcgOneVariant<NX, kOpBlock>{});
    return f(PcgOneVariant<NX, kOpQp>{});
  }
  if (warp) {
    if (op != kOpQp || gv || (cg && !f64)) return cudaErrorInvalidValue;
    if (f64) return f(PcgVariant<NX, kOpQp, kRedF64, double, false, false, true>{});
    if (red == kRedDf) return f(PcgVariant<NX, kOpQp, kRedDf, float, false, false, true>{});
    return cudaErrorInvalidValue;
  }
  if (cg && op == kOpQp && !f64) {  // single-reduction PCG (the FP64 and block-form launches stay textbook)
    if (red != kRedDf) return cudaErrorInvalidValue;
    if (gv) return f(PcgVariant<NX, kOpQp, kRedDf, float, true, true>{});
    return f(PcgVariant<NX, kOpQp, kRedDf, float, false, true>{});
  }
  if (gv) {
    if (op != kOpQp) return cudaErrorInvalidValue;
    if (f64) return f(PcgVariant<NX, kOpQp, kRedF64, double, true, false>{});
    if (red == kRedDf) return f(PcgVariant<NX, kOpQp, kRedDf, float, true, false>{});
    if (red == kRedF32) return f(PcgVariant<NX, kOpQp, kRedF32, float, true, false>{});
    if (red == kRedF64) return f(PcgVariant<NX, kOpQp, kRedF64, float, true, false>{});
    return cudaErrorInvalidValue;
  }
  if (f64) {
    if (op != kOpQp) return cudaErrorInvalidValue;
    return f(PcgVariant<NX, kOpQp, kRedF64, double, false, false>{});
  }
#define SSPCG_PCG_CASE(OPV, REDV) \
  if (op == OPV && red == REDV) return f(PcgVariant<NX, OPV, REDV, float, false, false>{});
  SSPCG_PCG_CASE(kOpQp, kRedDf)
  SSPCG_PCG_CASE(kOpQp, kRedF32)
  SSPCG_PCG_CASE(kOpQp, kRedF64)
  SSPCG_PCG_CASE(kOpBlock, kRedDf)
  SSPCG_PCG_CASE(kOpBlock, kRedF32)
  SSPCG_PCG_CASE(kOpBlock, kRedF64)
#undef SSPCG_PCG_CASE
  return cudaErrorInvalidValue;
}

template <int NX>
cudaError_t launch_pcg_for_nx(int op, int red, bool f64, const PcgArgs &a, int grid, int block, size_t smem,
                              cudaStream_t st) {
  return with_pcg_variant<NX>(op, red, f64, a.gscratch != nullptr, a.cg != 0, a.warp != 0, a.one != 0,
                              [&](auto v) { return decltype(v)::launch(a, grid, block, smem, st); });
}

template <int NX>
cudaError_t occupancy_pcg_for_nx(int op, int red, bool f64, bool gv, bool cg, bool warp, bool one, int block,
                                 size_t smem, int *ctas) {
  return with_pcg_variant<NX>(op, red, f64, gv, cg, warp, one,
                              [&](auto v) { return decltype(v)::occupancy(block, smem, ctas); });
}

}  // namespace sspcg

#define SSPCG_INSTANTIATE_PCG(NXV) SSPCG_INSTANTIATE_PCG_(NXV)  // expands a macro argument
#define SSPCG_INSTANTIATE_PCG_(NXV)                                                                            \
  namespace sspcg {                                                                                           \
  cudaError_t launch_pcg_nx##NXV(int op, int red, bool f64, const PcgArgs &a, int grid, int block, size_t smem, \
                                 cudaStream_t st) {                                                           \
    return launch_pcg_for_nx<NXV>(op, red, f64, a, grid, block, smem, st);                                     \
  }                                                                                                           \
  cudaError_t occupancy_pcg_nx##NXV(int op, int red, bool f64, bool gv, bool cg, bool warp, bool one,          \
                                    int block, size_t smem, int *ctas) {                                      \
    return occupancy_pcg_for_nx<NXV>(op, red, f64, gv, cg, warp, one, block, smem, ctas);                      \
  }                                                                                                           \
  }
