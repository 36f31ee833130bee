"""The right-hand side and the primal step around a solve by a warp per knot and by chunks: the same values, bit for bit
(the same operations in the same order).  A batch of few small knots and a lone problem of small blocks take the warps;
a batch of many small knots and a lone problem of large blocks take chunks, whatever the other sizes."""
import numpy as np
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg
    from _gpu_helpers import dev

SHAPES = [(0, 1, 0), (0, 28, 14), (1, 1, 1), (2, 3, 28), (5, 2, 1), (13, 28, 28), (20, 14, 7), (31, 21, 11), (40, 17, 0),
          (64, 8, 16), (65, 4, 2), (100, 12, 6), (128, 1, 28)]


def _inputs(i, p):
    n = lambda k, count: P.normals(P.config_key(95, 10 * i + k), max(count, 1))[:count].astype(np.float32)
    return {"c": n(0, p.n * p.nx), "q": n(1, p.n * p.nx), "r": n(2, p.N * p.nu), "mu": n(3, p.n * p.nx)}


# copies of the filler: 482 knots, too few for chunks; past 10,000 (right-hand side), past 16,000 (both), many
@pytest.mark.parametrize("copies", [0, 24, 39, 600])
def test_both_kernels_give_the_same_steps(copies):
    probs = P.custom_problems(SHAPES, config=95) + copies * P.custom_problems([(399, 2, 1)], config=96)
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    data = [_inputs(min(i, len(SHAPES)), p) for i, p in enumerate(probs)]
    put = lambda kind, k: torch.from_numpy(plan.pack(kind, [x[k] for x in data])).cuda()
    c, q, mu = (put(sspcg.ARRAY_VEC, k) for k in ("c", "q", "mu"))
    r = put(sspcg.ARRAY_RD, "r")
    gamma, dx, du = torch.zeros_like(c), torch.zeros_like(c), torch.zeros_like(r)
    sspcg.sspcg_form_gamma_batched(plan, d["A"], d["B"], d["qd"], d["rd"], c, q, r, gamma)
    sspcg.sspcg_recover_step_batched(plan, d["A"], d["B"], d["qd"], d["rd"], q, r, mu, dx, du)
    torch.cuda.synchronize()
    vec = [(p.n * p.nx,) for p in probs]
    gamma, dx = plan.unpack(sspcg.ARRAY_VEC, gamma, vec), plan.unpack(sspcg.ARRAY_VEC, dx, vec)
    du = plan.unpack(sspcg.ARRAY_RD, du, [(p.N * p.nu,) for p in probs])
    for i, (s, p) in enumerate(zip(SHAPES, probs)):
        A, B, qd, rd = dev(p.A), dev(p.B), dev(p.qd), dev(p.rd)
        x = {k: dev(v) for k, v in data[i].items()}
        g1, x1, u1 = torch.zeros_like(x["c"]), torch.zeros_like(x["c"]), torch.zeros_like(x["r"])
        sspcg.sspcg_form_gamma(p.N, p.nx, p.nu, A, B, qd, rd, x["c"], x["q"], x["r"], g1)
        sspcg.sspcg_recover_step(p.N, p.nx, p.nu, A, B, qd, rd, x["q"], x["r"], x["mu"], x1, u1)
        torch.cuda.synchronize()
        k, m = p.n * p.nx, p.N * p.nu
        assert np.array_equal(gamma[i], g1.cpu().numpy()[:k]), s
        assert np.array_equal(dx[i], x1.cpu().numpy()[:k]), s
        assert np.array_equal(du[i], u1.cpu().numpy()[:m]), s
