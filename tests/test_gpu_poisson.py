"""The 2-D Dirichlet Poisson driver (separation of variables, Sec. 3.2 and Sec. 4): DST-I along x,
the batch of mode systems through the Dichotomy kernels, inverse DST-I; against the oracle's
pipeline (scipy DST + Thomas per mode) and against manufactured solutions."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import poisson as OP  # noqa: E402


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_2469_gb300 import poisson
    return poisson


def rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def test_dst1_matches_scipy_and_is_involutory(P):
    import scipy.fft
    a = np.random.default_rng(0).standard_normal((37, 29))
    for dim in (0, 1):
        x = P.dst1(torch.from_numpy(a).cuda(), dim).cpu().numpy()
        assert rel(x, scipy.fft.dst(a, type=1, norm="ortho", axis=dim)) < 1e-14
    back = P.dst1(P.dst1(torch.from_numpy(a).cuda(), 0), 0).cpu().numpy()
    assert rel(back, a) < 1e-14


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("M", [1, 2, 31, 255])
def test_poisson2d_matches_oracle_pipeline(P, M, prec):
    f = np.random.default_rng(M).standard_normal((M, M))
    solver = P.Poisson2D(M, precision=prec)
    u = solver.solve(torch.from_numpy(f).cuda()).cpu().numpy()
    assert solver.status() == 0
    # both pipelines are FP64; the lowest mode's conditioning (~0.4 (M + 1)^2) amplifies the
    # rounding of the two DST implementations
    assert rel(u, OP.poisson2d(f)) < max(1e-13, 4e-16 * 0.4 * (M + 1) ** 2 * 10)


@pytest.mark.parametrize("p,q", [(1, 1), (7, 3)])
def test_poisson2d_single_mode(P, p, q):
    M = 511
    h = 1.0 / (M + 1)
    x = np.arange(1, M + 1) * h
    f = np.outer(np.sin(p * math.pi * x), np.sin(q * math.pi * x))
    lam = (4 * math.sin(p * math.pi * h / 2) ** 2 + 4 * math.sin(q * math.pi * h / 2) ** 2) / h ** 2
    u = P.Poisson2D(M).solve(torch.from_numpy(f).cuda()).cpu().numpy()
    assert rel(u, f / lam) < 1e-12


def test_poisson2d_manufactured(P):
    M = 1023
    us = np.random.default_rng(1).uniform(-1, 1, (M, M))
    f = OP.laplacian5(us)
    u = P.Poisson2D(M).solve(torch.from_numpy(f).cuda()).cpu().numpy()
    assert rel(u, us) < 1e-9        # kappa ~ 0.4 (M + 1)^2 = 4e5 times the FP64 unit roundoff


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("M,My", [(1, 2), (31, 17), (255, 300)])
def test_poisson2d_neumann_y_matches_oracle_pipeline(P, M, My, prec):
    """Neumann in y: every mode a quasi-Toeplitz system (eq. 21) in one batch."""
    f = np.random.default_rng(M + My).standard_normal((M, My))
    solver = P.Poisson2D(M, precision=prec, My=My, bc_y="neumann")
    u = solver.solve(torch.from_numpy(f).cuda()).cpu().numpy()
    assert solver.status() == 0
    assert rel(u, OP.poisson2d_neumann_y(f)) < max(1e-13, 4e-16 * 0.4 * max(M + 1, My) ** 2 * 10)
    assert rel(OP.laplacian5_neumann_y(u), f) < 1e-9


def test_poisson2d_neumann_y_manufactured(P):
    M, My = 511, 400
    us = np.random.default_rng(2).uniform(-1, 1, (M, My))
    f = OP.laplacian5_neumann_y(us)
    u = P.Poisson2D(M, My=My, bc_y="neumann").solve(torch.from_numpy(f).cuda()).cpu().numpy()
    assert rel(u, us) < 1e-10


@pytest.mark.parametrize("M,My", [(1, 1), (1, 5), (2, 3), (3, 64), (62, 65), (63, 63), (64, 129), (255, 17), (256, 16),
                                  (257, 130), (511, 33), (1022, 31), (130, 1000), (511, 1), (1023, 64), (2047, 35),
                                  (4095, 66)])
def test_transform_steps_against_scipy(P, M, My):
    """The transform of Poisson2D at the edges of its tiles (32 values of k and their mirror images by 64
    columns; 128 values of m by 16 columns), odd and even lengths.  A DST of length M sums M products:
    each output within (log2(M + 1) + 8) 2^-53 of the columns' 2-norm, the running sums of the odd
    outputs within sqrt(M + 1) times that."""
    import scipy.fft
    a = np.random.default_rng(M + 7 * My).standard_normal((M, My))
    solver = P.Poisson2D(M, My=My)
    x = solver._dst(torch.from_numpy(a).cuda(), 1.0).cpu().numpy()
    ref = scipy.fft.dst(a, type=1, norm="ortho", axis=0)
    tol = (math.log2(M + 1) + 8) * 2.0 ** -53 * np.linalg.norm(a, axis=0) * math.sqrt(M + 1)
    assert np.all(np.abs(x - ref) <= tol)
    scaled = solver._dst(torch.from_numpy(a).cuda(), solver.hy ** 2).cpu().numpy()
    assert np.all(np.abs(scaled - solver.hy ** 2 * ref) <= 2 * solver.hy ** 2 * tol)


@pytest.mark.parametrize("M", [511, 1023, 2047, 4095])
def test_fixed_point_transform_of_uneven_columns(P, M):
    """Columns of very different magnitudes in one pair (each has its own unit), zero columns, single
    spikes, constants and alternating signs (the largest growth a pass can see), the ends of the FP64
    range.  Per column: two units (below 2^-55 of the largest |a| times the growth sqrt(M) of its 2-norm)
    per pass, product and running sum stay within (log2(M + 1) + 8) 2^-53 of its 2-norm times sqrt(M + 1),
    as for the FP64 transform."""
    import scipy.fft
    rng = np.random.default_rng(M)
    cols = [rng.standard_normal(M) * 1e-280, rng.standard_normal(M) * 1e280, np.zeros(M), np.ones(M),
            (-1.0) ** np.arange(M), np.eye(M)[M // 2], np.eye(M)[0] * 5e-300, rng.standard_normal(M),
            np.sin(np.arange(1, M + 1) * (math.pi / (M + 1))), 1e12 + rng.standard_normal(M),
            np.exp(-0.05 * np.arange(M))]
    a = np.stack(cols, axis=1)
    solver = P.Poisson2D(M, My=a.shape[1])
    x = solver._dst(torch.from_numpy(a).cuda(), 1.0).cpu().numpy()
    unit = np.max(np.abs(a), axis=0)
    unit[unit == 0.0] = 1.0
    ref = scipy.fft.dst(a / unit, type=1, norm="ortho", axis=0)
    tol = (math.log2(M + 1) + 8) * 2.0 ** -53 * np.linalg.norm(a / unit, axis=0) * math.sqrt(M + 1)
    assert np.all(np.abs(x / unit - ref) <= tol)
    bad = a.copy()
    bad[3, 7] = np.nan
    y = solver._dst(torch.from_numpy(bad).cuda(), 1.0).cpu().numpy()
    assert np.isnan(y[:, 7]).all()   # and the pair's other column stands
    assert np.all(np.abs(y[:, 6] / unit[6] - ref[:, 6]) <= tol[6])


@pytest.mark.parametrize("M", [511, 1023])
def test_fixed_point_transform_errors_do_not_gather_over_rows(M):
    """Rows of one scale go through the same roundings: what mean error they keep must not be common to
    the rows, or a solve along the other axis adds it up.  The mean over the rows of every output's
    error, in units of its standard error: 6 of these over M outputs have a chance below 2e-6 (normal);
    a common offset of a fifth of the rounding noise would show as 9."""
    sf = pytest.importorskip("scipy.fft")
    from paper_1002_2469_gb300 import poisson as PS
    rows = 2048
    a = np.random.default_rng(M).uniform(-4.0, 4.0, (M, rows))
    solver = PS.Poisson2D(M, My=rows)
    got = solver._dst(torch.from_numpy(a).cuda(), 1.0).cpu().numpy()
    want = sf.dst(a.astype(np.longdouble), type=1, axis=0, norm="ortho")
    e = (got - want).astype(np.float64)
    assert np.sqrt(np.mean(e * e)) < 3e-15
    assert np.max(np.abs(e.mean(axis=1)) / (e.std(axis=1) / np.sqrt(rows))) < 6.0
