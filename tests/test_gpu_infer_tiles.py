"""Inference on the tcgen05 engine where its row tiles are cut: one row, one more and one less than a tile of 128, one
wave of tiles and the first size past it (pairs of tiles per CTA, CTAs that walk several), with last tiles and last pairs
that are nearly empty or full.  Against the mma.sync engine, whose products round the same operands to bf16 and differ by
the order of FP32 sums and rare rounding flips of hidden activations (bar 5e-4, as between the engines elsewhere)."""
import numpy as np
import pytest
import torch

from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg
    from _gpu_helpers import rel

SHAPES = [(0, 1, 0), (0, 28, 14), (1, 1, 1), (3, 28, 14), (2, 27, 0), (5, 2, 14), (40, 14, 7), (90, 5, 3), (129, 21, 11)]
WAVE = 128 * 152


def _check(shapes, max_rows):
    probs = P.custom_problems(shapes, config=88)
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    qp = d["A"], d["B"], d["qd"], d["rd"]
    sspcg.sspcg_build_schur_batched(plan, *qp, b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, "sym", b.D, b.E, b.PD, b.PE, b.status)
    net = sspcg.sspcg_mlp_create(max_rows)
    w = P.mlp_initial_params(5)
    w[-(32 * 256 + 32):] = 0.05 * P.normals(P.config_key(88, 1000), 32 * 256 + 32)  # W3 and b3 are zero at first
    sspcg.sspcg_mlp_set_params(net, torch.from_numpy(w).cuda())
    sspcg.sspcg_mlp_fit_normalisation(net, plan, *qp, d["gamma"], b.PD)
    out = {}
    for engine in ("tcgen05", "mma_sync"):
        sspcg.sspcg_mlp_set_engine(net, engine)
        lam0 = plan.empty(sspcg.ARRAY_VEC)
        sspcg.sspcg_mlp_infer(net, plan, *qp, d["gamma"], b.PD, lam0)
        torch.cuda.synchronize()
        out[engine] = plan.unpack(sspcg.ARRAY_VEC, lam0, [p.gamma.shape for p in probs])
    assert sspcg.sspcg_mlp_status(net) == 0
    x, y = (np.concatenate([v.ravel() for v in out[e]]) for e in ("tcgen05", "mma_sync"))
    assert np.isfinite(x).all() and np.abs(y).max() > 0
    assert rel(x, y) <= 5e-4


@pytest.mark.parametrize("max_rows", [1, 127, 128, 129, 1000])
def test_small_tiles(max_rows):
    _check(SHAPES[3:6] if max_rows == 1 else SHAPES, max_rows)


@pytest.mark.parametrize("rows", [WAVE // 4, WAVE // 4 + 1])  # four CTAs per row tile, and the first size with one
def test_around_a_quarter_wave(rows):
    _check([(1023, 3, 2)] * (rows // 1024) + [(rows % 1024 - 1, 3, 2)], rows)


@pytest.mark.parametrize("rows", [WAVE, WAVE + 1, WAVE + 128, WAVE + 129, 2 * WAVE + 256])
def test_around_a_wave(rows):
    _check([(1023, 3, 2)] * (rows // 1024) + [(rows % 1024 - 1, 3, 2)] * (rows % 1024 > 0), rows)
