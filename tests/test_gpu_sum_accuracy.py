"""Accuracy of the double-float block sums of the kernel with a thread per row pair (csrc/pcg_one.cuh): no worse than
the general kernel's on the same terms.

With S = I, block-diagonal Phi^-1 = diag(d) and one iteration, lambda = alpha z with z = d gamma (one rounding each) and
alpha = (gamma . z) / (z . z).  The last two entries of d cancel gamma . z to about 2e-13 of its terms' magnitude, so
the error of that sum, some 1e-16 of the magnitude, is a thousandth of alpha, which FP32 shows to 6e-8.  Both kernels
add the same terms in groups of another order; their mean errors over 600 sums differ by the spread of two such means
(standard deviation of an error about 0.8 of its mean, so 0.8 sqrt(2 / 600) = 4.6 %): five of those is the bar."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg

COUNT = 600


def _terms(R, rng):
    """gamma, d (float32, R entries): gamma . fl(d gamma) cancels down to about 2^-42 of the terms' magnitude."""
    g = rng.standard_normal(R).astype(np.float32)
    d = rng.standard_normal(R).astype(np.float32)
    g[-2:] = 1.0
    total = math.fsum((g[:-2].astype(np.float64) * (d[:-2] * g[:-2]).astype(np.float64)).tolist())
    d[-2] = -np.float32(total)
    rest = total + float(d[-2])
    d[-1] = -np.float32(rest) * np.float32(1 - 2.0 ** -12)
    return g, d


def _errors(N, nx, schedule):
    """Error of gamma . z relative to the sum of its terms' magnitudes, one per problem."""
    rng = np.random.default_rng(17)
    n = N + 1
    terms = [_terms(n * nx, rng) for _ in range(COUNT)]
    plan = sspcg.sspcg_plan_create([N] * COUNT, [nx] * COUNT, [1] * COUNT,
                                   sspcg.options(tol=0.0, max_iter=1, schedule=schedule))
    eye = np.broadcast_to(np.eye(nx, dtype=np.float32), (n, nx, nx))
    put = lambda kind, arrays: torch.from_numpy(plan.pack(kind, arrays)).cuda()
    D = put(sspcg.ARRAY_DIAG, [eye] * COUNT)
    E = plan.empty(sspcg.ARRAY_OFF)
    PD = put(sspcg.ARRAY_DIAG, [eye * d.reshape(n, nx, 1) for _, d in terms])
    gamma = put(sspcg.ARRAY_VEC, [g for g, _ in terms])
    lam = plan.empty(sspcg.ARRAY_VEC)
    iters = torch.zeros(COUNT, dtype=torch.int32, device="cuda")
    relres = torch.zeros(COUNT, dtype=torch.float64, device="cuda")
    status = torch.zeros(COUNT, dtype=torch.int32, device="cuda")
    sspcg.sspcg_solve_batched(plan, D, E, PD, None, gamma, lam, iters, relres, status)
    torch.cuda.synchronize()
    assert (iters == 1).all() and (status == sspcg.SOLVE_MAXITER).all()
    out = []
    for (g, d), x in zip(terms, plan.unpack(sspcg.ARRAY_VEC, lam, [(n * nx,)] * COUNT)):
        z = (d * g).astype(np.float64)
        t = g.astype(np.float64) * z  # exact: two FP32 factors
        i = int(np.argmax(np.abs(z)))
        got = float(x[i]) / z[i] * math.fsum((z * z).tolist())
        out.append(abs(got - math.fsum(t.tolist())) / np.abs(t).sum())
    return np.array(out)


@pytest.mark.parametrize("N,nx", [(127, 8), (64, 2)])  # 512 pairs and 65: sixteen warps and three
def test_row_pair_sums_are_as_accurate_as_the_general_kernels(N, nx):
    pairs, general = _errors(N, nx, "auto").mean(), _errors(N, nx, "stream").mean()
    assert general < 1e-15  # the sums cancel as intended: the errors are seen at all
    assert pairs <= 1.23 * general, (pairs, general)
