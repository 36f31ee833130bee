"""The PCG kernel with a thread per row pair (csrc/pcg_one.cuh) at the ends of what it takes: the last size whose layout
fits in the device's shared memory and the first that does not, the last with 512 pairs and the next, in both operator
forms, for even and odd nx and nu.  Against the general kernel (the STREAM schedule) with the bars of the parity tests:
both form the same block products and sum them in double-float, so lambda agrees to 1e-5 and the counts to one.

The sizes come from the library's layout and the device's limit, and the plan's schedule says which kernel runs."""
import numpy as np
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg
    from _gpu_helpers import LAMBDA_RTOL, rel
    from _layout import STATIC_SMEM, largest
    BUDGET = torch.cuda.get_device_properties(0).shared_memory_per_block_optin - STATIC_SMEM


def _solve(probs, op, **kw):
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs],
                                   sspcg.options(tol=1e-6, **kw))
    b = sspcg.Batch(plan, probs)
    d = b.dev
    sspcg.sspcg_build_schur_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    if op == 1:
        sspcg.sspcg_solve_qp_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.PD, b.PE, d["gamma"], b.lam, b.iters,
                                     b.relres, b.status)
    else:
        sspcg.sspcg_solve_batched(plan, b.D, b.E, b.PD, b.PE, d["gamma"], b.lam, b.iters, b.relres, b.status)
    torch.cuda.synchronize()
    return plan, b.lambdas(), b.iters.cpu().numpy(), b.status.cpu().numpy()


# (nx, nu): the memory ends the range for all but nx = 2, 3, 4 and, in the block form, nx = 5, which 512 pairs end
@pytest.mark.parametrize("op", [1, 0], ids=["qp", "block"])
@pytest.mark.parametrize("nx,nu", [(14, 7), (13, 7), (21, 4), (21, 11), (28, 14), (27, 0), (12, 28), (24, 5), (28, 28),
                                   (2, 1), (3, 2), (4, 2), (5, 28)])
def test_last_and_first_size(op, nx, nu):
    N, _, total = largest(op, nx, nu, BUDGET)
    probs = P.custom_problems([(N, nx, nu), (N + 1, nx, nu)], config=83)
    plan, lam, it, st = _solve(probs, op)
    _, lam0, it0, st0 = _solve(probs, op, schedule="stream")
    assert (st == sspcg.SOLVE_OK).all() and (st0 == sspcg.SOLVE_OK).all()
    for i, p in enumerate(probs):
        assert abs(int(it[i]) - int(it0[i])) <= 1, (p.N, it[i], it0[i])
        assert rel(lam[i], lam0[i]) <= LAMBDA_RTOL, p.N
    if op == 1:  # the plan's schedule lists the groups of the QP form
        assert any(g["max_N"] == N and g["smem"] == total and g["stream"] == 0 for g in
                   sspcg.sspcg_plan_schedule(plan, "solve_qp"))
        assert not any(g["max_N"] == N + 1 and g["smem"] == total for g in sspcg.sspcg_plan_schedule(plan, "solve_qp"))
