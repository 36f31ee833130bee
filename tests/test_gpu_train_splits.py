"""Gradients over row chunks (splits of 512 rows and more, tiles of 512 rows of a column sum): a step over P problems
against the mean of the steps over each alone.  P is a power of two, so that every bf16 value of the backward pass is
the single problem's times 1/P exactly, and the gradients differ by FP32 summation only: at most 1,100 terms in a row,
1,100 * 2^-24 = 6.6e-5 of the terms' magnitude."""
import numpy as np
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg

# block rows per problem: 511, 512, 513 and 1,025 rows; 33,024 rows are more than 64 splits of 512
ROWS = [[255, 256], [256, 256], [256, 257], [256, 256, 256, 257], [516] * 64]


@pytest.mark.parametrize("weights", ["initial", "random"])
@pytest.mark.parametrize("rows", ROWS, ids=[str(sum(r)) for r in ROWS])
def test_gradients_are_the_mean_of_single_steps(rows, weights):
    probs = P.custom_problems([(n - 1, 3, 2) for n in rows], config=86)
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    qp = d["A"], d["B"], d["qd"], d["rd"]
    sspcg.sspcg_build_schur_batched(plan, *qp, b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    net = sspcg.sspcg_mlp_create(sum(rows))
    w = P.mlp_initial_params(6)  # W3 = b3 = 0: no gradient at lambda* = 0
    if weights == "random":
        w[-(32 * 256 + 32):] = 0.05 * P.normals(P.config_key(86, 1000), 32 * 256 + 32)
    sspcg.sspcg_mlp_set_params(net, torch.from_numpy(w).cuda())
    sspcg.sspcg_mlp_fit_normalisation(net, plan, *qp, d["gamma"], b.PD)
    star = torch.zeros_like(d["gamma"])
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")

    def grads(p0, p1):
        sspcg.sspcg_mlp_train_step(net, plan, p0, p1, *qp, d["gamma"], b.D, b.E, b.PD, star, sspcg.adam(lr=0.0), loss)
        g = torch.zeros(sspcg.MLP_PARAMS, device="cuda")
        sspcg.sspcg_mlp_get_grads(net, g)
        return g.cpu().numpy().astype(np.float64)

    each = [grads(i, i + 1) / len(rows) for i in range(len(rows))]
    got, want = grads(0, len(rows)), sum(each)
    edges = np.cumsum([256 * 1344, 256, 256 * 256, 256, 32 * 256])
    for x, y, *e in zip(np.split(got, edges), np.split(want, edges), *(np.split(g, edges) for g in each)):
        assert np.linalg.norm(x - y) <= 6.6e-5 * sum(np.linalg.norm(v) for v in e)
        assert weights == "initial" or np.linalg.norm(y) > 0
