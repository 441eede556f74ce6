"""A weakly dominant plan that reports the general path leaves its intermediates (beta of eq. 16, the blocks'
first and last values) in the workspace after every solve, adjoint and series, whatever windows solved it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402

TOL = 1e-12


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_2469_gb300 as pkg
    return pkg


def check(plan, t, F, scale_of):
    info = plan.info
    P, n = info["P"], info["n"]
    torch.cuda.synchronize()
    ref = oracle.dich_eq15(t, F, oracle.even_starts(plan.N, n))
    scale = np.max(np.abs(ref["x"]))
    at = lambda o: plan.workspace[o:o + 16 * P].view(torch.float64).cpu().numpy().reshape(P, 2)  # noqa: E731
    beta, iface = at(info["beta_offset"]), at(info["iface_offset"])
    for got, want in ((beta[:, 0], "beta_L"), (beta[:, 1], "beta_R"), (iface[:, 0], "x_first"), (iface[:, 1], "x_last")):
        assert np.max(np.abs(got - ref[want])) / scale < TOL, (scale_of, want)


@pytest.mark.parametrize("t,N", [((-1.0, 2.001, -1.0), 5894), ((-1.0, 2.005, -1.004), 20011), ((-1.0, 2.001, -1.0), 30001)])
def test_intermediates_of_weak_plans(D, t, N):
    rng = np.random.default_rng(N)
    plan = D.Plan(*t, N)
    assert plan.info["path"] == 2 and plan.info["beta_offset"] > 0 and plan.info["iface_offset"] > 0
    F, w = rng.standard_normal(N), rng.uniform(-1.0, 1.0, N)
    plan.workspace[plan.info["beta_offset"]:].fill_(255)   # (NaN)
    x = plan.solve(torch.from_numpy(F).cuda())
    check(plan, t, F, "solve")
    plan.adjoint(torch.from_numpy(w).cuda(), x)
    check(plan, t[::-1], w, "adjoint")
    Fs = rng.standard_normal((3, N))
    plan.solve_series(torch.from_numpy(Fs).cuda())
    check(plan, t, Fs[-1], "series")
