"""Accuracy of FP64-form windows in 64-bit fixed point: no mean error on weakly dominant systems, and every
component as good as the FP64 recurrences give it, against the binary128 oracle."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_2469_gb300 as pkg
    return pkg


def roots(t):
    q = (abs(t[1]) + math.sqrt(t[1] * t[1] - 4.0 * t[0] * t[2])) / 2.0
    return abs(t[0]) / q, abs(t[2]) / q, 1.0 / q


def error(x, t, F):
    """x - exact and the binary128 solution rounded to FP64 (that rounding is taken out by one step of
    refinement, its residual in extended precision)."""
    xq = oracle.thomas_q(t, F)
    X = np.concatenate([[0], xq, [0]]).astype(np.longdouble)
    r = (F.astype(np.longdouble) - np.longdouble(t[0]) * X[:-2] - np.longdouble(t[1]) * X[1:-1]
         - np.longdouble(t[2]) * X[2:]).astype(np.float64)
    return (x - xq) - oracle.thomas(t, r), xq


@pytest.mark.parametrize("t", [(-1.0, 2.0013, -1.0), (-1.0, 2.002, -1.0), (-1.0, 2.005, -1.0), (1.0, 2.005, 1.0),
                               (-1.0, 2.005, -1.004), (-1.0, 2.1, -1.0), (-1.0, 2.5, -1.0), (-1.2, 2.5, -0.8),
                               (-0.9, 1.9, 0.0)])
def test_weak_systems_have_no_mean_error(D, t):
    """Mean error over 2^20 rows of a right-hand side without a sign, in units of the words.  The few
    products between threads leave at most half a unit each on average, at most eight of them on either
    way: 4 units into u, hence 4 / (1 - B) + 4 into X, one more for the output's constant; the random
    part (below 64 units, uncorrelated beyond 256 rows) averages to 64 / sqrt(4096) = 1."""
    N = 1 << 20
    F = np.random.default_rng(5).standard_normal(N)
    s = np.where(np.arange(N) % 2 == 1, -1.0, 1.0) if t[0] * t[1] > 0 else np.ones(N)
    x = D.Plan(*t, N).solve(torch.from_numpy(F).cuda()).cpu().numpy()
    err, _ = error(x, t, F)
    R, B, g = roots(t)
    hb = 63 + math.floor(math.log2((1.0 - R) * (1.0 - B)))
    unit = g * 2.0 ** (math.frexp(np.max(np.abs(F)))[1] - hb)
    assert abs(np.mean(s * err)) <= (4.0 / (1.0 - B) + 4.0 + 2.0) * unit
