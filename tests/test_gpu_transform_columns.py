"""Transforms of lengths that go through the FFT library: every column has errors of its own size only."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M", [1, 2, 62, 255, 599, 1001, 1999, 3071])
def test_columns_of_very_different_magnitudes(M):
    """Per column, as for columns of one size: (log2(M + 1) + 8) 2^-53 of its 2-norm times sqrt(M + 1) for
    the running sums; a column with a NaN leaves the others alone.  (Odd lengths M + 1 above 256 are not among
    these: there the FFT library itself takes two rows at a time.)"""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sf = pytest.importorskip("scipy.fft")
    from paper_1002_2469_gb300 import poisson as PS
    rng = np.random.default_rng(M)
    cols = [rng.standard_normal(M) * 1e20, rng.standard_normal(M), rng.standard_normal(M) * 1e-30, np.ones(M), np.zeros(M),
            rng.standard_normal(M) * 1e100, np.eye(M)[M // 2], 1e12 + rng.standard_normal(M), rng.standard_normal(M) * 1e-100]
    for order in (cols, cols[1:]):   # both neighbours of every column
        a = np.stack(order, axis=1)
        solver = PS.Poisson2D(M, My=a.shape[1])
        unit = np.max(np.abs(a), axis=0)
        unit[unit == 0.0] = 1.0
        ref = sf.dst(a / unit, type=1, norm="ortho", axis=0)
        tol = (math.log2(M + 1) + 8) * 2.0 ** -53 * np.linalg.norm(a / unit, axis=0) * math.sqrt(M + 1)
        x = solver._dst(torch.from_numpy(a).cuda(), 1.0).cpu().numpy()
        assert np.all(np.abs(x / unit - ref) <= tol)
        for bad in range(a.shape[1]):
            b = a.copy()
            b[M // 3, bad] = np.nan
            y = solver._dst(torch.from_numpy(b).cuda(), 1.0).cpu().numpy()
            assert np.isnan(y[:, bad]).any()
            rest = np.arange(a.shape[1]) != bad
            assert np.array_equal(y[:, rest], x[:, rest])
