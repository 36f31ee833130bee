"""The loss of a training step where the width of its CTAs changes: with the number of problems (two, four CTAs' worth
per SM and one more) and with the rows of the longest.  The loss of P problems is the mean of their losses alone; each is
a sum of squares of the same FP32 values in FP64, so the two differ by FP64 rounding only: at most 1,300 additions in
a row, 1,300 * 2^-53 = 1.5e-13 of a sum of positive terms."""
import numpy as np
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1
# (problems, N, nx): one knot; 31 and 33 knots of 32 outputs around 1,024 entries; 8 rows of 32 entries (256); around
# the limits of 1,024, 512 and 256 threads by the number of problems
CASES = [(1, 0, 1), (3, 30, 5), (3, 32, 28), (2, 7, 3), (2, 8, 3), (2, 300, 4), (2 * SMS, 40, 3), (2 * SMS + 1, 40, 3),
         (4 * SMS, 40, 3), (4 * SMS + 1, 40, 3)]


@pytest.mark.parametrize("count,N,nx", CASES)
def test_loss_is_the_mean_of_single_losses(count, N, nx):
    probs = P.custom_problems([(N, nx, 2)] * min(count, 4), config=87)
    probs = [probs[i % len(probs)] for i in range(count)]
    plan = sspcg.sspcg_plan_create([N] * count, [nx] * count, [2] * count, sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    qp = d["A"], d["B"], d["qd"], d["rd"]
    sspcg.sspcg_build_schur_batched(plan, *qp, b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    net = sspcg.sspcg_mlp_create(count * (N + 1))
    w = P.mlp_initial_params(6)
    w[-(32 * 256 + 32):] = 0.05 * P.normals(P.config_key(87, 1000), 32 * 256 + 32)  # W3 and b3 are zero at first
    sspcg.sspcg_mlp_set_params(net, torch.from_numpy(w).cuda())
    sspcg.sspcg_mlp_set_engine(net, "mma_sync")  # the products' widths do not depend on the number of rows
    sspcg.sspcg_mlp_fit_normalisation(net, plan, *qp, d["gamma"], b.PD)
    star = torch.zeros_like(d["gamma"])

    def loss(p0, p1):
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        sspcg.sspcg_mlp_train_step(net, plan, p0, p1, *qp, d["gamma"], b.D, b.E, b.PD, star, sspcg.adam(lr=0.0), out)
        return float(out.item())

    each = [loss(i, i + 1) for i in range(min(count, 4))]
    want = sum(each[i % len(each)] for i in range(count)) / count
    assert want > 0
    assert abs(loss(0, count) - want) <= 1.5e-13 * want
