"""The FP32 Schur and off-diagonal preconditioner blocks (csrc/build_f32.cu), made in chunks of blocks and 4 x 4 tiles:
block sizes at the ends of tiles, horizons at the ends of chunks, no inputs, more inputs than states.  Singly against
the oracle at its bars (1e-6 relative; PE's with PD's magnitude, from which it is formed); batched bit-identical."""
import numpy as np
import pytest
import torch

from oracle import block
from paper_2309_06427_gb300 import problems as P

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg
    from _gpu_helpers import gpu_precond, gpu_schur, oracle_blocks32, dev, rel

# (blocks in a chunk, nx, nu): of the Schur kernel, then of the off-diagonal kernel
SHAPES = [(N, nx, nu) for c, nx, nu in [(3, 28, 28), (6, 28, 0), (19, 5, 28), (213, 4, 2),
                                        (4, 28, 14), (7, 21, 11), (16, 14, 7), (64, 5, 3), (239, 4, 1), (256, 1, 1)]
          for N in (c - 1, c, c + 1)] + [(0, 28, 14), (1, 1, 0), (1, 3, 2), (2, 8, 4), (5, 9, 5), (5, 25, 13)]


@pytest.mark.parametrize("kind", ["sym", "add", "bj", "jacobi"])
def test_blocks_at_tile_and_chunk_ends(kind):
    probs = P.custom_problems(SHAPES, config=84) * 170  # 6,120 problems: one CTA each, in full chunks
    plan = sspcg.sspcg_plan_create([p.N for p in probs], [p.nx for p in probs], [p.nu for p in probs], sspcg.options())
    b = sspcg.Batch(plan, probs)
    d = b.dev
    sspcg.sspcg_build_schur_batched(plan, d["A"], d["B"], d["qd"], d["rd"], b.D, b.E)
    sspcg.sspcg_build_precond_batched(plan, kind, b.D, b.E, b.PD, b.PE, b.status)
    assert (b.status.cpu().numpy() == 0).all()
    diag, off = [(p.n, p.nx, p.nx) for p in probs], [(p.N, p.nx, p.nx) for p in probs]
    Ds, PDs = plan.unpack(sspcg.ARRAY_DIAG, b.D, diag), plan.unpack(sspcg.ARRAY_DIAG, b.PD, diag)
    Es, PEs = plan.unpack(sspcg.ARRAY_OFF, b.E, off), plan.unpack(sspcg.ARRAY_OFF, b.PE, off)
    for i in range(len(SHAPES), len(probs)):
        j = i % len(SHAPES)
        for x in (Ds, Es, PDs, PEs):
            assert np.array_equal(x[i], x[j]), SHAPES[j]
    for i, p in enumerate(probs[:len(SHAPES)]):
        nd, no = p.n * p.nx ** 2, p.N * p.nx ** 2
        _, D, E = gpu_schur(p)
        assert np.array_equal(Ds[i].ravel(), D.cpu().numpy()[:nd]), SHAPES[i]
        assert np.array_equal(Es[i].ravel(), E.cpu().numpy()[:no]), SHAPES[i]
        assert np.array_equal(Ds[i], np.transpose(Ds[i], (0, 2, 1)))
        PD, PE, _ = gpu_precond(p, D, E, kind)
        assert np.array_equal(PDs[i].ravel(), PD.cpu().numpy()[:nd]), SHAPES[i]
        assert np.array_equal(PEs[i].ravel(), PE.cpu().numpy()[:no]), SHAPES[i]
        S = block.build_schur(p.A, p.B, p.qd, p.rd)
        assert rel(Ds[i], S.d) <= 1e-6, SHAPES[i]
        D32, E32, So = oracle_blocks32(p)
        Mo = block.build_precond(So, kind)
        if p.N:
            assert rel(Es[i], S.l[1:]) <= 1e-6, SHAPES[i]
            PD, PE, _ = gpu_precond(p, dev(D32.ravel()), dev(E32.ravel()), kind)
            bar = 1e-6 * max(1.0, np.abs(Mo.d).max() / max(np.abs(Mo.l).max(), 1e-30))
            assert rel(PE.cpu().numpy()[:no], Mo.l[1:]) <= bar, SHAPES[i]
