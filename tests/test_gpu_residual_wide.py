"""The true residual of problems with more inputs than states, whose chunks hold at least 128 rows where they fit
(residual_rows in csrc/common.cuh): horizons at the ends of those chunks, against the dense FP64 residual with the bar of
the other chunk tests, alone and in a batch with problems of fewer inputs, which leaves every value as it is alone."""
import numpy as np
import pytest
import torch

from oracle import dense
from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg
    from _gpu_helpers import dev

# chunks of 64, 64, 43, 32, 16, 10, 8 and 7 block rows; two problems of no more inputs than states
SHAPES = [(N, nx, nu) for c, nx, nu in [(64, 1, 28), (64, 2, 3), (43, 3, 28), (32, 4, 28), (16, 8, 28), (10, 14, 28),
                                        (8, 17, 28), (7, 20, 28)] for N in (c - 1, c, c + 1)]
SHAPES += [(0, 1, 28), (20, 14, 7), (9, 28, 28)]
RES_RTOL = 1.4e-11  # FP64: some 120 roundings of 2^-53 along a sum, whose terms are at most 1e3 times the result


def test_wide_problems_alone_and_batched():
    probs = P.custom_problems(SHAPES, config=89)
    lams = [(0.1 * P.normals(P.config_key(89, 1000 + i), p.gamma.size)).astype(np.float32) for i, p in enumerate(probs)]
    alone = []
    for p, lam in zip(probs, lams):
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        sspcg.sspcg_residual_qp(p.N, p.nx, p.nu, dev(p.A), dev(p.B), dev(p.qd), dev(p.rd), dev(p.gamma), dev(lam), out)
        g = p.gamma.astype(np.float64).ravel()
        want = np.linalg.norm(g - dense.schur(p.A, p.B, p.qd, p.rd) @ lam.astype(np.float64)) / np.linalg.norm(g)
        assert abs(out.item() - want) <= RES_RTOL * want, (p.N, p.nx, p.nu)
        alone.append(out.item())
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    b.lam.copy_(torch.from_numpy(plan.pack(sspcg.ARRAY_VEC, lams)))
    sspcg.sspcg_residual_qp_batched(plan, d["A"], d["B"], d["qd"], d["rd"], d["gamma"], b.lam, b.relres)
    torch.cuda.synchronize()
    assert np.array_equal(b.relres.cpu().numpy(), np.array(alone))
