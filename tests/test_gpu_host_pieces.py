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


def enqueued(call, stream, block_of_first=False):
    """The number of nodes (kernels, copies) that `call` enqueues on `stream`, or the first one's threads per
    block, by stream capture."""
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
    threads = 0
    if block_of_first:
        nodes = (ctypes.c_void_p * n.value)()
        params = (ctypes.c_uint32 * 64)()   # function (8 bytes), grid x y z, block x y z, ...
        assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(nodes[0]), params) == 0
        threads = params[5]
    cu.cuGraphDestroy(graph)
    return threads if block_of_first else n.value


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


@pytest.mark.parametrize("N", [100003, 1 << 20])
def test_pinned_memory_is_read_by_the_fp64_sweeps(D, N):
    """FP64-form windows that read and write host memory: one thread per block of the plan's windows (the
    fixed-point form's blocks of 32 rows each would have more)."""
    s = torch.cuda.Stream()
    plan = D.Plan(-1.2, 2.5, -0.8, N, block_size=64, threads=64)
    F = torch.randn(N, dtype=torch.float64).pin_memory()
    x = torch.empty(N, dtype=torch.float64, pin_memory=True)
    call = lambda: D.dichotomy_solve_host(plan.handle, F, x, None, None, 0, s.cuda_stream)  # noqa: E731
    call()
    s.synchronize()
    want = plan.solve(F.cuda()).cpu()
    assert torch.max(torch.abs(x - want)) <= 1e-13 * torch.max(torch.abs(want))
    assert enqueued(call, s, block_of_first=True) == 64
