"""Which problems of nx 1 and 5 run with a thread per row pair: with more than one or two to an SM only the shorter ones.
The plan's schedule tells the groups apart; the solutions of both kernels agree with the bars of the parity tests, with
a plan and without allocation."""
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

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1


def _solve(probs, noalloc=False):
    opts = sspcg.options(tol=1e-6)
    shapes = [p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs]
    plan = sspcg.sspcg_plan_create(*shapes, opts)
    b = sspcg.Batch(plan, probs)
    d = b.dev
    qp = d["A"], d["B"], d["qd"], d["rd"]
    sspcg.sspcg_build_schur_batched(plan, *qp, b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    out = b.lam, b.iters, b.relres, b.status
    if noalloc:
        sspcg.sspcg_solve_qp_batched_noalloc(*shapes, *qp, b.PD, b.PE, d["gamma"], b.lam, opts, *out[1:])
    else:
        sspcg.sspcg_solve_qp_batched(plan, *qp, b.PD, b.PE, d["gamma"], *out)
    torch.cuda.synchronize()
    assert (b.status == sspcg.SOLVE_OK).all()
    return sspcg.sspcg_plan_schedule(plan, "solve_qp"), b.lambdas(), b.iters.cpu().numpy()


@pytest.mark.parametrize("nx,short,long", [(1, 64, 65), (5, 140, 141)])
def test_many_long_problems_take_the_general_kernel(nx, short, long):
    a, b = P.custom_problems([(short, nx, 3), (long, nx, 3)], config=97)
    few = _solve([a, b])
    assert len(few[0]) == 1  # one group: both with a thread per row pair
    many = _solve([a] * SMS + [b] * (SMS + 1))
    assert sorted(g["max_N"] for g in many[0]) == [short, long]
    direct = _solve([a] * SMS + [b] * (SMS + 1), noalloc=True)
    for got in (many, direct):
        for i, k in ((0, 0), (SMS - 1, 0), (SMS, 1), (2 * SMS, 1)):
            assert rel(got[1][i], few[1][k]) <= LAMBDA_RTOL
            assert abs(int(got[2][i]) - int(few[2][k])) <= 1
