"""dichotomy_solve_noalloc near the size of its static array: the general path's systems leave the
fixed-point table, which that path does not use, out of it."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("t,N", [((-1.0, 2.001, -1.0), 504907), ((-1.0, 2.0013, -1.0), 506567), ((-0.99, 1.0, 0.0), 514259)])
def test_largest_general_systems_are_accepted(t, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    from paper_1002_2469_gb300 import _lib
    F = np.random.default_rng(N).standard_normal(N)
    d, x = torch.from_numpy(F).cuda(), torch.empty(N, dtype=torch.float64, device="cuda")
    rc = _lib.load().dichotomy_solve_noalloc(*t, N, ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(x.data_ptr()),
                                             ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    ref = oracle.thomas_q(t, F)
    assert np.max(np.abs(x.cpu().numpy() - ref)) <= 1e-12 * np.max(np.abs(ref))
