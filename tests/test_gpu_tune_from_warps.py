"""The tuner on a plan whose groups run one problem per warp already: it also times one problem per CTA and keeps the
faster.  A lone problem of 256 rows takes a warp eight rows per lane, several times as long as a CTA."""
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg


@pytest.mark.parametrize("shape", [(31, 8, 4), (63, 4, 2)])
def test_tuner_leaves_one_problem_per_warp(shape):
    probs = P.custom_problems([shape], config=85)
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs],
                                   sspcg.options(tol=1e-6, schedule="warp", precision="f32"))
    assert [g["warps"] > 0 for g in sspcg.sspcg_plan_schedule(plan, "pipeline")] == [True]
    b = sspcg.Batch(plan, probs)
    d = b.dev
    try:
        sspcg.sspcg_plan_autotune(plan, "sym", d["A"], d["B"], d["qd"], d["rd"], d["gamma"], b.D, b.E, b.PD, b.PE,
                                  b.lam, b.iters, b.relres, b.status, which="pipeline")
    finally:
        sspcg.sspcg_autotune_cache_clear()
    assert [g["warps"] for g in sspcg.sspcg_plan_schedule(plan, "pipeline")] == [0]
    b.pipeline()
    torch.cuda.synchronize()
    assert int(b.status[0]) == sspcg.SOLVE_OK
