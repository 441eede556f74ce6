"""FP64-form windows solved in 64-bit fixed point (32 rows per thread): the sizes, alignments, signs and
right-hand sides where that form's cases meet, against the binary128 oracle.

Tolerance.  One unit of a window's words is at most u = 2 max|F| 2^-hb with 2^hb <= 2^63 (1 - R)(1 - B)
(R = |rs|, B = |ib|).  Every product truncates at most 3 units; a row takes at most three products into
u and X and two into the output, and the recurrences amplify a row's error by at most
1 / ((1 - R)(1 - B)) <= 2^(64 - hb); conversions add one unit each.  So |x - exact| is at most
2^-53 |x| (the final rounding) + 16 u 2^(64 - hb) |g|; windows of varying scale spend two more bits.
Rows solved in FP64 instead (values that do not suit fixed point) are held to the suite's 1e-12.
"""
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


def bound(t, F, xq, extra_bits=0):
    tm1, t0, tp1 = (abs(v) for v in t)
    q = (t0 + math.sqrt(t0 * t0 - 4.0 * t[0] * t[2])) / 2.0
    head = (1.0 - tm1 / q) * (1.0 - tp1 / q)
    hb = 63 + math.floor(math.log2(head)) - extra_bits
    unit = 2.0 * np.max(np.abs(F)) * 2.0 ** -hb
    return 2.0 ** -53 * np.max(np.abs(xq)) + 16.0 * unit * 2.0 ** (64 - hb) / q


def distance(x, t, F):
    """max |x - exact| and the binary128 solution rounded to FP64: that rounding (as large as the bound
    itself) is taken out again with one step of refinement, its residual in extended precision."""
    xq = oracle.thomas_q(t, F)
    X = np.concatenate([[0], xq, [0]]).astype(np.longdouble)
    r = (F.astype(np.longdouble) - np.longdouble(t[0]) * X[:-2] - np.longdouble(t[1]) * X[1:-1]
         - np.longdouble(t[2]) * X[2:]).astype(np.float64)
    return np.max(np.abs((x - xq) - oracle.thomas(t, r))), xq


T = [(-1.2, 2.5, -0.8), (-1.0, 4.0, -1.0), (1.0, 4.0, 1.0), (0.7, -2.5, 1.1), (0.0, 2.0, -1.0), (-1.0, 2.0, 0.0),
     (-1.0, 2.2, -1.0)]


def one_window(D, t, N):
    """A plan of one window of 64 blocks (the default would take shorter windows for so short a system)."""
    n = -(-N // 64)
    return D.Plan(*t, N, block_size=n + (N % n == 1), threads=64)


def rhs(shape, N, rng):
    if shape == "random":
        return rng.standard_normal(N)
    if shape == "smooth":        # 20 decades over the system, a little from block to block: varying scale
        return rng.uniform(1.0, 2.0, N) * np.exp(-46.0 * (np.arange(N) / N - 0.4) ** 2 / 0.36)
    F = rng.standard_normal(N)   # zero stretches and a spike: windows solved in FP64 beside others
    F[N // 4:N // 2] = 0.0
    F[N // 3] = 1e9
    return F


# one window (n = ceil(N / 64) rows per block) up to 4096 rows, its thread, warp and block edges; windows
# with halos, a single last row in a slot, an odd block size (N mod 64 = 1)
SIZES = [1984, 2017, 2048, 3001, 4031, 4064, 4096]
LONG = [1 << 20, (1 << 20) + 1, 1200005, 1249983]


@pytest.mark.parametrize("shape", ["random", "smooth", "holes"])
@pytest.mark.parametrize("t", T)
def test_windows_against_binary128(D, t, shape):
    rng = np.random.default_rng(17)
    for N in SIZES + (LONG if t in T[:2] or t == T[6] else LONG[1:2]):
        F = rhs(shape, N, rng)
        plan = one_window(D, t, N) if N <= 4096 else D.Plan(*t, N)
        x = plan.solve(torch.from_numpy(F).cuda()).cpu().numpy()
        assert plan.status() == 0
        err, xq = distance(x, t, F)
        if shape == "holes":
            assert err <= 1e-12 * np.max(np.abs(xq)), N
        else:
            assert err <= bound(t, F, xq, 2 if shape == "smooth" else 0), (N, plan.info["n"])


@pytest.mark.parametrize("scale", [1e-200, 1.0, 1e15, 1e200])
def test_scales_and_odd_offsets(D, scale):
    """Rows at odd offsets (8-byte copies), next to canaries; scales inside and outside the words' range."""
    t, N = (-1.2, 2.5, -0.8), 4001
    F = np.random.default_rng(3).standard_normal(N) * scale
    plan = one_window(D, t, N)
    for off in (0, 1):
        buf = torch.full((N + 3,), float("nan"), dtype=torch.float64, device="cuda")
        out = torch.full((N + 3,), 7.0, dtype=torch.float64, device="cuda")
        buf[off:off + N] = torch.from_numpy(F).cuda()
        D.dichotomy_solve(plan.handle, buf[off:off + N], out[off:off + N])
        o = out.cpu().numpy()
        assert plan.status() == 0
        assert (o[:off] == 7.0).all() and (o[off + N:] == 7.0).all()
        err, xq = distance(o[off:off + N], t, F)
        assert err <= (bound(t, F, xq) if scale < 1e100 else 1e-12 * np.max(np.abs(xq)))


def test_nonfinite_stays_local_and_is_reported(D):
    t, N = (-1.2, 2.5, -0.8), 1 << 20
    F = np.random.default_rng(4).standard_normal(N)
    F[N // 2] = np.inf
    plan = D.Plan(*t, N, flags=D.FLAG_CHECK_FINITE)
    x = plan.solve(torch.from_numpy(F).cuda()).cpu().numpy()
    assert plan.status() == 5
    assert not np.isfinite(x[N // 2])
    ref = oracle.thomas(t, np.where(np.isfinite(F), F, 0.0))
    assert np.max(np.abs(x[:N // 4] - ref[:N // 4])) < 1e-12


@pytest.mark.parametrize("t", [T[0], T[2], T[6]])
def test_adjoint_batch_and_series(D, t):
    """The transposed solve with its gradient sums, a batch with systems of both forms of a window, and
    a series on the plan's second geometry."""
    rng = np.random.default_rng(8)
    N = 600001
    F, w = rng.standard_normal(N), rng.uniform(-1, 1, N)
    plan = D.Plan(*t, N)
    x = plan.solve(torch.from_numpy(F).cuda())
    gF, gt = plan.adjoint(torch.from_numpy(w).cuda(), x)
    xq = oracle.thomas_q(t, F)
    err, lq = distance(gF.cpu().numpy(), t[::-1], w)
    assert err <= bound(t, w, lq)
    ref = -np.array([math.fsum(lq[1:] * xq[:-1]), math.fsum(lq * xq), math.fsum(lq[:-1] * xq[1:])])
    # n products rounded and summed: n 2^-53 sum |lambda x| at worst, sqrt(n) of it in earnest
    assert np.max(np.abs(gt.cpu().numpy() - ref)) <= 2.0 ** -53 * math.sqrt(N) * np.sum(np.abs(lq * xq))
    Ns = np.array([4096, 5, 2049, 100, 9001, 1, 4095, 70000], dtype=np.int64)
    off = np.concatenate([[0], np.cumsum(Ns)[:-1]])
    Fb = rng.standard_normal(int(Ns.sum()))
    k = np.full(Ns.size, 1.0)
    b = D.Batch(Ns, t[0] * k, t[1] * k, t[2] * k)
    xb = b.solve(torch.from_numpy(Fb).cuda()).cpu().numpy()
    assert b.status() == 0
    for n, o in zip(Ns, off):
        err, q = distance(xb[o:o + n], t, Fb[o:o + n])
        # systems shorter than the form's smallest window are solved in FP64
        assert err <= max(bound(t, Fb[o:o + n], q), 1e-14 * np.max(np.abs(q))), n
    M, Nr = 200, 9001
    Fs = rng.standard_normal((M, Nr))
    xs = D.Plan(*t, Nr).solve_series(torch.from_numpy(Fs).cuda()).cpu().numpy()
    for r in (0, 1, M - 1):
        err, q = distance(xs[r], t, Fs[r])
        assert err <= bound(t, Fs[r], q)


def test_high_gain_windows(D):
    """Coupling longer than a default window (one pass over wider ones), and a solution far below the
    words' bound there (solved in FP64)."""
    t, N = (-1.0, 2.001, -1.0), 1 << 21
    rng = np.random.default_rng(9)
    for F in (rng.standard_normal(N), np.where(np.arange(N) % 2 == 0, 1.0, -1.0) * rng.uniform(1.0, 1.01, N)):
        plan = D.Plan(*t, N)
        x = plan.solve(torch.from_numpy(F).cuda()).cpu().numpy()
        xq = oracle.thomas_q(t, F)
        assert np.max(np.abs(x - xq)) <= 1e-12 * np.max(np.abs(xq))
