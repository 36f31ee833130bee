"""A tcgen05 product whose bounded waits run out: it sets the error flag, writes nothing, waits for the copies it has
issued, frees its tensor memory and returns, so that the GPU and the context stay usable.  The kernels are compiled here
with waits of no polls at all, so that every wait runs out at once; the wait for what is in flight keeps its length.
Every size that picks another kernel (a quarter of the columns, one and two row tiles per CTA, 32 columns, the rest of
the inference), with one, part of and several tiles; afterwards the library's own inference runs on the same GPU."""
import ctypes
import os
import shutil
import subprocess

import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg

PROGRAM = r'''
#include "mlp_tc.cu"
using namespace sspcg;
using namespace sspcg::mlp;
extern "C" int product(int epi, const void *A, const void *B, long long M, int N, int K, const float *bias, void *Cb,
                       float *Cf, int *err, int sms) {
  cudaError_t e = launch_gemm_nt_tc(epi, (const bf16 *)A, (const bf16 *)B, M, N, K, bias, (bf16 *)Cb, Cf, err, 0, sms);
  return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
extern "C" int tail(const int *kref, long long rows, const void *H1, const void *W2, const float *b2, const void *W3,
                    const float *b3, float *lambda, int *err, int sms) {
  RowSpan rs{};
  rs.ps.single.nx = 3;
  rs.ps.nprob = 1;
  rs.kref = (const int2 *)kref;
  rs.nrows = rows;
  cudaError_t e = launch_tail_tc(rs, (const bf16 *)H1, (const bf16 *)W2, b2, (const bf16 *)W3, b3, lambda, err, 0, sms);
  return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    folder = tmp_path_factory.mktemp("tc")
    src, so = folder / "tc.cu", folder / "tc.so"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, *_build.ARCH, *_build.FLAGS, f"-I{_build.CSRC}", "-DSSPCG_TC_POLLS=0u", "-shared", str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1
ptr = lambda t: ctypes.c_void_p(t.data_ptr())


def _library_runs():
    probs = P.custom_problems([(40, 14, 7)] * 8, config=88)
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    qp = d["A"], d["B"], d["qd"], d["rd"]
    sspcg.sspcg_build_schur_batched(plan, *qp, b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    net = sspcg.sspcg_mlp_create(8 * 41)
    sspcg.sspcg_mlp_set_params(net, torch.from_numpy(P.mlp_initial_params(5)).cuda())
    sspcg.sspcg_mlp_infer(net, plan, *qp, d["gamma"], b.PD, b.lam)
    torch.cuda.synchronize()
    assert sspcg.sspcg_mlp_status(net) == 0


# (epilogue: bias and ReLU to bf16, or bias to FP32; rows; columns; K): K of fewer stages than the ring holds, and of more
@pytest.mark.parametrize("relu,M,N,K", [(1, 1, 256, 64), (1, 130, 256, 1344), (1, 128 * SMS, 256, 256),
                                        (1, 128 * SMS, 256, 1344), (1, 128 * SMS + 1, 256, 1344), (0, 300, 256, 512),
                                        (0, 1000, 32, 256), (1, 1000, 32, 1344)])
def test_product_returns_when_its_waits_run_out(lib, relu, M, N, K):
    A = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    B = torch.zeros((N, K), dtype=torch.bfloat16, device="cuda")
    bias = torch.zeros(N, device="cuda")
    out = torch.full((M, N), 7.0, dtype=torch.bfloat16 if relu else torch.float32, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    none = ctypes.c_void_p(None)
    epi = 0 if relu else 1  # Epilogue of csrc/mlp.h
    for _ in range(3):
        err.zero_()
        torch.cuda.synchronize()
        assert lib.product(epi, ptr(A), ptr(B), ctypes.c_longlong(M), N, K, ptr(bias), ptr(out) if relu else none,
                           none if relu else ptr(out), ptr(err), SMS) == 0
        assert int(err.item()) == 1
    assert bool((out == 7.0).all())
    _library_runs()


@pytest.mark.parametrize("rows", [1, 128, 300, 128 * SMS * 2 + 5])
def test_inference_tail_returns_when_its_waits_run_out(lib, rows):
    kref = torch.stack([torch.zeros(rows, dtype=torch.int32), torch.arange(rows, dtype=torch.int32)], 1).cuda()
    H1 = torch.zeros((rows, 256), dtype=torch.bfloat16, device="cuda")
    W2 = torch.zeros((256, 256), dtype=torch.bfloat16, device="cuda")
    W3 = torch.zeros((32, 256), dtype=torch.bfloat16, device="cuda")
    b2, b3 = torch.zeros(256, device="cuda"), torch.zeros(32, device="cuda")
    out = torch.full((rows * 3,), 7.0, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert lib.tail(ptr(kref), ctypes.c_longlong(rows), ptr(H1), ptr(W2), ptr(b2), ptr(W3), ptr(b3), ptr(out), ptr(err),
                    SMS) == 0
    assert int(err.item()) == 1
    assert bool((out == 7.0).all())
    _library_runs()
