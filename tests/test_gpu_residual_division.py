"""The FP64 quotients of the true residual (csrc/residual.cu divides by an FP32 value in seven instructions) against IEEE
division, over the whole range of its arguments.

A problem of one knot and one unknown has (S lambda) = lambda / q, so its residual is |gamma - lambda / q| / |gamma|.  With
gamma the quotient rounded to FP32 the subtraction is exact and leaves at most 2^-24 of gamma: one unit in the last place
of the quotient changes the residual by more than 2^-53 / 2^-24 = 1.8e-9 of itself, a correctly rounded one leaves four
roundings of square, quotient and root: 4 * 2^-53 = 4.5e-16."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2309_06427_gb300 import build as _build
    _build.build()
    from paper_2309_06427_gb300 import sspcg


def _residuals(gamma, lam, q):
    n = len(q)
    plan = sspcg.sspcg_plan_create([0] * n, [1] * n, [0] * n, sspcg.options())
    put = lambda kind, v: torch.from_numpy(plan.pack(kind, list(v.reshape(n, 1)))).cuda()
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    sspcg.sspcg_residual_qp_batched(plan, None, None, put(sspcg.ARRAY_QD, q), None, put(sspcg.ARRAY_VEC, gamma),
                                    put(sspcg.ARRAY_VEC, lam), out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _expected(gamma, lam, q):
    with np.errstate(all="ignore"):
        g = gamma.astype(np.float64)
        r = g - lam.astype(np.float64) / q.astype(np.float64)
        return np.sqrt((r * r) / (g * g))


def _check(gamma, lam, q):
    got, want = _residuals(gamma, lam, q), _expected(gamma, lam, q)
    with np.errstate(invalid="ignore"):  # inf - inf where both are
        same = (got == want) | (np.isnan(got) & np.isnan(want)) | (np.abs(got - want) <= 4.5e-16 * want)
    assert same.all(), [(lam[i], q[i], got[i], want[i]) for i in np.flatnonzero(~same)[:5]]


@pytest.mark.parametrize("low,high", [(-20, 20), (-126, 127)])
def test_quotients_are_correctly_rounded(low, high):
    rng = np.random.default_rng(high)
    q = np.ldexp(rng.uniform(1, 2, 200000), rng.integers(low, high, 200000)).astype(np.float32)
    lam = (np.ldexp(rng.uniform(1, 2, 200000), rng.integers(-60, 60, 200000))
           * rng.choice([-1, 1], 200000)).astype(np.float32)
    with np.errstate(all="ignore"):
        gamma = (lam.astype(np.float64) / q.astype(np.float64)).astype(np.float32)
    use = np.isfinite(gamma) & (np.abs(gamma) >= np.float32(2.0 ** -126))
    assert use.sum() > 50000
    _check(gamma[use], lam[use], q[use])


def test_special_values():
    tiny, low, top = np.float32(2.0 ** -149), np.float32(2.0 ** -126), np.float32(3.4028235e38)
    qs = np.array([1, 3, low, tiny, 3 * tiny, low / 2, top, top / 2, 2.0 ** 126, 2.0 ** 127, np.inf, 0, -2, np.nan],
                  np.float32)
    xs = np.array([0, 1, -1, 0.3, tiny, -7 * tiny, low, top, -top, np.inf, -np.inf, np.nan], np.float32)
    lam, q = (v.ravel() for v in np.meshgrid(xs, qs))
    _check(np.ones_like(lam), lam, q)
