"""Feature rows where a warp walks several (more than 12 per SM): horizons, block sizes and input counts that change from
row to row, no inputs, horizon 0.  All problems in one call against one call per problem, where a warp has one row at
most; those rows are checked against the oracle in test_gpu_mlp.py.  Each row is the same arithmetic: bit-identical."""
import numpy as np
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg

SHAPES = [(0, 1, 0), (0, 28, 14), (1, 1, 1), (3, 28, 14), (2, 27, 0), (5, 2, 14), (40, 14, 7), (90, 5, 3), (129, 21, 11)]


@pytest.mark.parametrize("rep", [7, 23])
def test_rows_of_one_call_and_of_many(rep):
    probs = P.custom_problems(SHAPES, config=87) * rep
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    qp = d["A"], d["B"], d["qd"], d["rd"]
    sspcg.sspcg_build_schur_batched(plan, *qp, b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    rows = sum(p.n for p in probs)
    net = sspcg.sspcg_mlp_create(rows)
    sspcg.sspcg_mlp_fit_normalisation(net, plan, *qp, d["gamma"], b.PD)
    X = torch.zeros((rows, sspcg.MLP_IN), dtype=torch.bfloat16, device="cuda")
    sspcg.sspcg_mlp_features(net, plan, 0, len(probs), *qp, d["gamma"], b.PD, X)
    Y = torch.zeros_like(X)
    r = 0
    for i, p in enumerate(probs):
        sspcg.sspcg_mlp_features(net, plan, i, i + 1, *qp, d["gamma"], b.PD, Y[r:])
        r += p.n
    assert torch.equal(X.view(torch.int16), Y.view(torch.int16))
    assert X.float().abs().sum().item() > 0
