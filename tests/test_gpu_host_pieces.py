"""Solves from host memory: how much is enqueued for them."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_2469_gb300 as pkg
    return pkg


def enqueued(call, stream):
    """The nodes (kernels, copies) of what `call` enqueues on `stream`, by stream capture."""
    cu = ctypes.CDLL("libcuda.so.1")
    h = ctypes.c_void_p(stream.cuda_stream)
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    stream.synchronize()
    assert cu.cuStreamBeginCapture_v2(h, 2) == 0    # relaxed
    try:
        call()
    finally:
        rc = cu.cuStreamEndCapture(h, ctypes.byref(graph))
    assert rc == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    cu.cuGraphDestroy(graph)
    return n.value


@pytest.mark.parametrize("N", [600, 3001, 4096])
def test_short_system_is_copied_whole(D, N):
    """One default window of rows: one copy in, one launch, one copy out, though the plan splits it into
    several short windows; a system of many default windows goes in pieces."""
    s = torch.cuda.Stream()
    for n, pieces in ((N, 1), (100003, 4)):
        plan = D.Plan(-1.0, 4.0, -1.0, n)
        assert plan.info["path"] == 1
        F = torch.randn(n, dtype=torch.float64).pin_memory()
        x = torch.empty(n, dtype=torch.float64, pin_memory=True)
        stage = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)]
        torch.cuda.synchronize()
        call = lambda: D.dichotomy_solve_host(plan.handle, F, x, *stage, 4, s.cuda_stream)  # noqa: E731
        call()   # (the plan makes its streams and events)
        want = plan.solve(F.cuda()).cpu()
        s.synchronize()
        assert torch.equal(x, want)
        assert enqueued(call, s) == 3 * pieces
