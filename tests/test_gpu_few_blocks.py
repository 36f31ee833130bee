"""FP32 Schur and off-diagonal preconditioner blocks by a warp per knot, which a few small blocks take, and by chunks:
the same values, bit for bit (the same operations in the same order), on both sides of the line between them."""
import numpy as np
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg

SHAPES = [(0, 1, 0), (0, 8, 8), (1, 1, 1), (5, 2, 1), (7, 3, 8), (20, 4, 2), (31, 5, 3), (40, 7, 7), (64, 8, 8), (100, 8, 0)]


def _blocks(probs, kind):
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    sspcg.sspcg_build_schur_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, kind, b.D, b.E, b.PD, b.PE, b.status)
    torch.cuda.synchronize()
    assert (b.status == 0).all()
    return [plan.unpack(a, t, [(p.n if a == sspcg.ARRAY_DIAG else p.N, p.nx, p.nx) for p in probs])
            for a, t in ((sspcg.ARRAY_DIAG, b.D), (sspcg.ARRAY_OFF, b.E), (sspcg.ARRAY_DIAG, b.PD),
                         (sspcg.ARRAY_OFF, b.PE))]


@pytest.mark.parametrize("kind", ["sym", "add", "bj"])
def test_both_kernels_give_the_same_blocks(kind):
    probs = P.custom_problems(SHAPES, config=91)
    filler = P.custom_problems([(440, 2, 1)], config=92)
    few = _blocks(probs, kind)                        # 278 knots of at most 8 rows: a warp each
    many = _blocks(probs + 20 * filler, kind)         # 9,098 knots: chunks
    large = _blocks(probs + P.custom_problems([(3, 9, 9)], config=93), kind)  # nx, nu past 8: chunks
    for x, y, z in zip(few, many, large):
        for i, s in enumerate(SHAPES):
            assert np.array_equal(x[i], y[i]), s
            assert np.array_equal(x[i], z[i]), s


# knots in three problems around 4,500 (Schur blocks) and 8,003 (8,000 off-diagonal blocks)
@pytest.mark.parametrize("knots", [4499, 4500, 4501, 8002, 8003, 8004])
def test_at_the_lines(knots):
    probs = P.custom_problems([(knots - 1 - 4000, 2, 1), (1999, 2, 1), (1999, 2, 1)], config=94)
    got = _blocks(probs, "sym")
    for i in range(3):
        want = _blocks([probs[i]], "sym")  # at most 4,004 knots: a warp each
        for x, y in zip(got, want):
            assert np.array_equal(x[i], y[0])
