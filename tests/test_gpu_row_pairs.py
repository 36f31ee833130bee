"""The PCG kernel with a thread per row pair (csrc/pcg_one.cuh) against the general kernel on the same inputs, where
tiles, pairs and lanes are cut: odd and even nx, the smallest horizons, nu that is odd, zero or not ceil(nx / 2), the
largest problems it takes and the first it does not, both operator forms, warm starts and block-diagonal
preconditioners.

The STREAM schedule takes the general kernel.  Both form the same products in the same order and sum them in
double-float, so alpha and beta differ by an FP32 rounding at most now and then: lambda within 1e-5 of each other
(the parity bar against the oracle) and iteration counts within one."""
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

# (N, nx, nu): single knots, one and two block rows, odd tails, pairs across warps, 512 pairs and just past, the
# largest that fits whole and just past it
SHAPES = [(0, 1, 1), (0, 5, 2), (0, 28, 14), (1, 1, 0), (1, 2, 3), (2, 3, 2), (3, 28, 14), (7, 13, 7), (9, 5, 28),
          (20, 21, 11), (31, 21, 4), (16, 27, 14), (255, 4, 2), (256, 4, 2), (72, 14, 7), (73, 14, 7), (84, 12, 6),
          (85, 12, 6), (40, 15, 0)]


def _solve(probs, op, kind, **kw):
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs],
                                   sspcg.options(tol=1e-6, **kw))
    b = sspcg.Batch(plan, probs)
    d = b.dev
    sspcg.sspcg_build_schur_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, kind, b.D, b.E, b.PD, b.PE, b.status)
    if kw.get("warm_start"):
        b.lam.copy_(0.01 * d["gamma"])
    PE = None if kind == "bj" else b.PE
    if op == "qp":
        sspcg.sspcg_solve_qp_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.PD, PE, d["gamma"], b.lam, b.iters,
                                     b.relres, b.status)
    else:
        sspcg.sspcg_solve_batched(plan, b.D, b.E, b.PD, PE, d["gamma"], b.lam, b.iters, b.relres, b.status)
    torch.cuda.synchronize()
    return b.lambdas(), b.iters.cpu().numpy(), b.status.cpu().numpy()


@pytest.mark.parametrize("op,kind,warm", [("qp", "sym", 0), ("qp", "sym", 2), ("qp", "bj", 0), ("block", "sym", 0),
                                          ("block", "bj", 1)])
def test_row_pairs_match_general_kernel(op, kind, warm):
    probs = P.custom_problems(SHAPES, config=81)
    lam, it, st = _solve(probs, op, kind, warm_start=warm)
    lam0, it0, st0 = _solve(probs, op, kind, warm_start=warm, schedule="stream")
    assert np.array_equal(st, st0)
    for i, s in enumerate(SHAPES):
        assert abs(int(it[i]) - int(it0[i])) <= 1, (s, it[i], it0[i])
        assert rel(lam[i], lam0[i]) <= LAMBDA_RTOL, s
