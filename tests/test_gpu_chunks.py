"""The QP step around the solve and the FP64 true residual, whose CTAs walk chunks of block rows: sizes at the ends of
chunks, the largest and smallest blocks, no inputs, more inputs than states, values the residual's integer widening and
its division treat apart, and batches with one CTA per problem against the singly launched calls."""
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
    from _gpu_helpers import dev, rel

# A chunk has min(64, 256 / (nx + nu)) block rows: 64, 64, 42, 21, 12, 8, 8, 4.
SHAPES = [(N, nx, nu) for c, nx, nu in [(64, 1, 0), (64, 1, 1), (42, 4, 2), (21, 8, 4), (12, 14, 7), (8, 28, 4),
                                        (8, 2, 28), (4, 28, 28)] for N in (c - 1, c, c + 1)] + [(0, 1, 0), (1, 28, 28)]
# FP64: some 120 roundings of 2^-53 along a sum, whose terms are at most 1e3 times the result here
RES_RTOL = 1.4e-11


def _residual(p, lam, **kw):
    a = {k: getattr(p, k) for k in ("A", "B", "qd", "rd", "gamma")} | kw
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    sspcg.sspcg_residual_qp(p.N, p.nx, p.nu, dev(a["A"]), dev(a["B"]), dev(a["qd"]), dev(a["rd"]), dev(a["gamma"]),
                            dev(lam), out)
    g = a["gamma"].astype(np.float64).ravel()
    with np.errstate(all="ignore"):
        Sx = dense.schur(a["A"], a["B"], a["qd"], a["rd"]) @ lam.astype(np.float64).ravel()
    return out.item(), np.linalg.norm(g - Sx) / np.linalg.norm(g)


def _lam(p, seed):
    return (0.1 * P.normals(P.config_key(82, seed), p.gamma.size)).astype(np.float32).reshape(p.gamma.shape)


def test_chunk_edges_singly_and_batched():
    probs = P.custom_problems(SHAPES, config=82)
    vecs = [P.qp_vectors(p, seed=3) for p in probs]
    lams = [_lam(p, i) for i, p in enumerate(probs)]
    single = []
    for p, (c, q, r), lam in zip(probs, vecs, lams):
        n, m = p.n, p.nx
        A, B, qd, rd = dev(p.A), dev(p.B), dev(p.qd), dev(p.rd)
        g, dx, du = (torch.zeros(max(k, 4), device="cuda") for k in (n * m, n * m, p.N * p.nu))
        sspcg.sspcg_form_gamma(p.N, m, p.nu, A, B, qd, rd, dev(c), dev(q), dev(r), g)
        sspcg.sspcg_recover_step(p.N, m, p.nu, A, B, qd, rd, dev(q), dev(r), dev(lam), dx, du)
        g, dx, du = g.cpu().numpy()[:n * m], dx.cpu().numpy()[:n * m], du.cpu().numpy()[:p.N * p.nu]
        dx_ref, du_ref = dense.recover_step(p.A, p.B, p.qd, p.rd, q, r, lam)
        # FP32 sums of at most 2 * 28 products of FP32 inputs
        assert rel(g, dense.form_gamma(p.A, p.B, p.qd, p.rd, c, q, r)) <= 1e-6
        assert rel(dx, dx_ref) <= 1e-6
        if du.size:
            assert rel(du, du_ref) <= 1e-6
        got, want = _residual(p, lam)
        assert abs(got - want) <= RES_RTOL * want, (p.N, m, p.nu)
        single.append((g, dx, du, got))

    rep = 100  # 2600 problems: one CTA each, which walks all of its chunks
    many = probs * rep
    plan = sspcg.sspcg_plan_create([p.N for p in many], [p.nx for p in many], [p.nu for p in many], sspcg.options())
    b = sspcg.Batch(plan, many)
    d = b.dev
    ones = np.ones(max(int(plan.sizes[sspcg.ARRAY_RD]), 4), np.float32)
    cv, qv, lv = (torch.from_numpy(plan.pack(sspcg.ARRAY_VEC, x * rep)).cuda()
                  for x in ([v[0] for v in vecs], [v[1] for v in vecs], lams))
    rv = torch.from_numpy(plan.pack(sspcg.ARRAY_RD, [v[2] for v in vecs] * rep, ones)).cuda()
    gam, dx, du = plan.empty(sspcg.ARRAY_VEC), plan.empty(sspcg.ARRAY_VEC), plan.empty(sspcg.ARRAY_RD)
    res = torch.zeros(len(many), dtype=torch.float64, device="cuda")
    sspcg.sspcg_form_gamma_batched(plan, d["A"], d["B"], d["qd"], d["rd"], cv, qv, rv, gam)
    sspcg.sspcg_recover_step_batched(plan, d["A"], d["B"], d["qd"], d["rd"], qv, rv, lv, dx, du)
    sspcg.sspcg_residual_qp_batched(plan, d["A"], d["B"], d["qd"], d["rd"], d["gamma"], lv, res)
    gs = plan.unpack(sspcg.ARRAY_VEC, gam, [p.gamma.shape for p in many])
    dxs = plan.unpack(sspcg.ARRAY_VEC, dx, [p.gamma.shape for p in many])
    dus = plan.unpack(sspcg.ARRAY_RD, du, [(p.N, p.nu) for p in many])
    res = res.cpu().numpy()
    for i in range(len(many)):
        g, x, u, r = single[i % len(probs)]
        assert np.array_equal(gs[i].ravel(), g) and np.array_equal(dxs[i].ravel(), x), SHAPES[i % len(probs)]
        assert np.array_equal(dus[i].ravel(), u) and res[i] == r, SHAPES[i % len(probs)]


def test_residual_of_values_apart():
    """Zeros and subnormals among the inputs, costs whose FP32 reciprocal is subnormal or infinite, and infinities."""
    p = P.custom_problems([(9, 5, 3)], config=83)[0]
    lam = _lam(p, 50)
    A = p.A.copy()
    A.flat[::3], A.flat[1::7] = 0.0, 1e-41
    lam.flat[::4], lam.flat[1::5] = -0.0, -1e-44
    for scale, gscale in ((1.0, 1.0), (1.5e38, 1e-38), (1e-40, 1e30)):
        u = (0.5 + P.uniform01(P.config_key(83, 1), p.qd.size)).reshape(p.qd.shape)
        w = (0.5 + P.uniform01(P.config_key(83, 2), p.rd.size)).reshape(p.rd.shape)
        got, want = _residual(p, lam, A=A, qd=(u * scale).astype(np.float32), rd=(w * scale).astype(np.float32),
                              gamma=(p.gamma * gscale).astype(np.float32))
        assert np.isfinite(want) and abs(got - want) <= RES_RTOL * want, scale
    for bad in (np.inf, np.nan):
        A.flat[4] = bad
        assert not np.isfinite(_residual(p, lam, A=A)[0])
