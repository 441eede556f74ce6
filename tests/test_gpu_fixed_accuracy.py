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


def component_bound(t, F):
    """A priori bound of the FP64 recurrences' errors, row by row: with s, t the two recurrences run on
    |F| (g t = |T^-1| |F|), constants good to an ulp and their powers to an ulp per row, and 32 roundings of
    quantities below t for the block ends, the scan and the corrections of the block solves."""
    R, B, g = roots(t)

    def conv(a, r, order):
        out, c = np.empty_like(a), np.zeros(a.shape[1:], dtype=a.dtype)
        for i in order:
            c = c * r + a[i]
            out[i] = c
        return out

    N = F.shape[0]
    up, down = range(N), range(N - 1, -1, -1)
    s = conv(np.abs(F).astype(np.longdouble), R, up)
    y = conv(s, B, down)
    e = 4.0 * conv(conv(s, R, up), B, down) + 4.0 * conv(y, B, down) + 32.0 * y
    return g * 2.0 ** -53 * e


def sparse(N, rng):
    """Right-hand sides whose rows differ by many orders of magnitude within a few rows, and ordinary ones."""
    i = np.arange(N)
    out = {}
    out["one value in 32 rows"] = np.where(i % 32 == 7, 1.0 + np.abs(rng.standard_normal(N)), 0.0)
    out["rows 64 k and 64 k + 63"] = np.where((i % 64 == 0) | (i % 64 == 63), 1.0, 0.0)
    out["small background"] = np.where(i % 32 == 31, 1.0, 1e-12 * rng.uniform(0.5, 1.0, N))
    out["large values"] = np.where(i % 32 == 16, 1e10, rng.standard_normal(N))
    F = rng.standard_normal(N)
    at = 40
    while at < N - 100:   # stretches weakened by up to 2^-30
        n = int(rng.integers(2, 60))
        F[at:at + n] *= 2.0 ** -rng.uniform(0.0, 30.0)
        at += n + int(rng.integers(20, 120))
    out["weak stretches"] = F
    out["zero stretch at a warp's edge"] = np.where((i % 1024 > 990) | (i % 1024 < 3), 0.0, rng.standard_normal(N))
    out["sine"] = np.sin(2.0 * np.pi * 5.3 * (i + 0.37) / 4096.0)
    out["steep"] = rng.uniform(1.0, 2.0, N) * 2.0 ** (-(i % 4096) / 8.0)
    out["random"] = rng.standard_normal(N)
    return out


@pytest.mark.parametrize("t", [(-1.0, 4.0, -1.0), (-0.5, 8.0, -0.5), (-1.0, 20.0, -1.0), (-1.2, 2.5, -0.8), (1.0, 4.0, 1.0),
                               (0.7, -2.5, 1.1), (-1.0, 2.05, -1.0), (-1.0, 2.005, -1.0), (0.0, 2.0, -1.0),
                               (-1.0, 2.0, 0.0)])
def test_every_row_is_as_good_as_fp64_recurrences_give_it(D, t):
    N = 4093
    cases = sparse(N, np.random.default_rng(23))
    bounds = component_bound(t, np.stack(list(cases.values()), axis=1))
    # one window, whose block solves leave nothing out
    plan = D.Plan(*t, N, block_size=64, threads=64, trunc_eps=1e-290)
    for k, (name, F) in enumerate(cases.items()):
        x = plan.solve(torch.from_numpy(F).cuda()).cpu().numpy()
        err, _ = error(x, t, F)
        assert (np.abs(err) <= bounds[:, k] + 1e-290).all(), (name, float(np.max(np.abs(err) / (bounds[:, k] + 1e-290))))


@pytest.mark.parametrize("N", [4096, 100003])
def test_zero_and_subnormal_windows(D, N):
    """Windows of zeros have the zero solution; values near the lower end of the FP64 range (whose upper bits
    are those of zero too) are solved: spacing 2^-1074, at most a few roundings of it."""
    t = (-1.0, 4.0, -1.0)
    plan = D.Plan(*t, N, block_size=64, threads=64)
    x = plan.solve(torch.zeros(N, dtype=torch.float64, device="cuda"))
    assert (x == 0.0).all()
    F = np.zeros(N)
    F[N // 2:N // 2 + 40] = 1000.0 * 2.0 ** -1074
    F[N // 3] = -3e-310
    x = plan.solve(torch.from_numpy(F).cuda()).cpu().numpy()
    ref = oracle.thomas(t, F * 2.0 ** 600) * 2.0 ** -600
    assert np.max(np.abs(x - ref)) <= 16 * 2.0 ** -1074
    assert np.max(np.abs(x)) > 1e-311


@pytest.mark.parametrize("t", [(-1.0, 4.0, -1.0), (-1.2, 2.5, -0.8), (1.0, 4.0, 1.0), (0.7, -2.5, 1.1)])
@pytest.mark.parametrize("N", [1984, 3001, 4031, 4096, 100005])
def test_rows_of_varying_scale(D, t, N):
    """A right-hand side that falls by 9 to 20 decades from block to block (windows whose threads each have
    their own unit), a slope with sign changes and one with a noisy tail: every row against the bound of the
    values around it, so a wrong unit in the tail shows.  Halos truncate at 2^-64 of values at most 2^8
    times the row's own, far below the bound."""
    rng = np.random.default_rng(N)
    i = np.arange(N)
    m = np.minimum(i % 4096, 4096 - i % 4096) / 4096.0
    cases = {"gaussian": rng.uniform(1.0, 2.0, N) * np.exp(-46.0 * (i / N - 0.4) ** 2 / 0.36),
             "triangle": rng.uniform(1.0, 2.0, N) * 2.0 ** (-100.0 * m),
             "signs": np.sin(0.013 * i + 0.1) * 2.0 ** (-60.0 * m)}
    bounds = component_bound(t, np.stack(list(cases.values()), axis=1))
    n = -(-N // 64)
    plan = D.Plan(*t, N, block_size=n + (N % n == 1), threads=64) if N <= 4096 else D.Plan(*t, N, block_size=64, threads=64)
    for k, (name, F) in enumerate(cases.items()):
        x = plan.solve(torch.from_numpy(F).cuda()).cpu().numpy()
        err, _ = error(x, t, F)
        assert (np.abs(err) <= bounds[:, k]).all(), (name, float(np.max(np.abs(err) / bounds[:, k])))
