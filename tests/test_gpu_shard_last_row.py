"""MIXED systems of 16 k + 1 rows keep a last block of a single row: that row by itself, from whole and
sharded solves and from the adjoint, against the binary128 oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from test_gpu_shard import sharded_separate_buffers  # noqa: E402


@pytest.mark.parametrize("nshards", [1, 2, 3])
@pytest.mark.parametrize("t,N,kw", [((-1.2, 2.5, -0.8), 300001, {}), ((0.7, 2.5, -1.1), 65537, {}),
                                    ((0.7, 2.5, -1.1), 65537, {"flags": 1}), ((-1.0, 2.001, -1.0), 200001, {}),
                                    ((-1.2, 2.5, -0.8), 16 * 127 * 2 + 1, {})])
def test_last_row_of_16k_plus_1(t, N, kw, nshards):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_2469_gb300 as D
    plan = D.Plan(*t, N, precision=1, threads=64, **kw)   # (else a short system takes shorter blocks)
    assert plan.info["n"] == 16 and plan.info["n_last"] == 1
    F = np.random.default_rng(N).standard_normal(N)
    F[-1] = 10.0   # (the last row's solution is not small)
    ref = oracle.thomas_q(t, F)
    tol = 1e-12 * abs(ref[-1])   # the suite's norm-wise tolerance, on one component of the solution's size
    x, _ = sharded_separate_buffers(D, plan, F, nshards)
    assert abs(x[-1] - ref[-1]) <= tol
    xd = plan.solve(torch.from_numpy(F).cuda())
    assert abs(float(xd[-1]) - ref[-1]) <= tol
    gF, _ = plan.adjoint(torch.from_numpy(F).cuda(), xd)
    lam = oracle.thomas_q(t[::-1], F)
    assert abs(float(gF[-1]) - lam[-1]) <= 1e-12 * abs(lam[-1])
