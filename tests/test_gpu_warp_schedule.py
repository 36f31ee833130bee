"""The WARP schedule at the end of what fits in shared memory whole: one problem per warp only for problems that the
per-warp kernel's layout holds whole.  The layout of the kernel with a thread per row pair is the smaller one, so some
problems fit whole in that one alone: they run there, not by 32 threads with part of their blocks staged.  Solutions
against the automatic schedule with the bars of the parity tests."""
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


def _solve(shapes, schedule):
    probs = P.custom_problems(shapes, config=84)
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs],
                                   sspcg.options(tol=1e-6, schedule=schedule))
    b = sspcg.Batch(plan, probs)
    d = b.dev
    sspcg.sspcg_build_schur_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    sspcg.sspcg_solve_qp_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.PD, b.PE, d["gamma"], b.lam, b.iters,
                                 b.relres, b.status)
    torch.cuda.synchronize()
    return plan, b.lambdas(), b.iters.cpu().numpy(), b.status.cpu().numpy()


@pytest.mark.parametrize("nx,nu", [(14, 7), (14, 14)])
def test_only_whole_problems_run_one_per_warp(nx, nu):
    pairs, general, _ = largest(1, nx, nu, BUDGET)
    assert pairs > general  # the window this test is about
    sizes = [general - 8, general, general + 1, pairs, pairs + 1]
    shapes = [(N, nx, nu) for N in sizes]
    plan, lam, it, st = _solve(shapes, "warp")
    by_warp = {}
    for g in sspcg.sspcg_plan_schedule(plan, "solve_qp"):
        by_warp[g["max_N"]] = (g["problems"], g["warps"] > 0)
    assert by_warp == {general: (2, True), pairs: (2, False), pairs + 1: (1, False)}
    _, lam0, it0, st0 = _solve(shapes, "auto")
    assert (st == sspcg.SOLVE_OK).all() and (st0 == sspcg.SOLVE_OK).all()
    for i, s in enumerate(shapes):
        assert abs(int(it[i]) - int(it0[i])) <= 1, (s, it[i], it0[i])
        assert rel(lam[i], lam0[i]) <= LAMBDA_RTOL, s
