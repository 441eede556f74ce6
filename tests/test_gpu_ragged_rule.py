"""Which kernel a MIXED system with a shorter last block takes: the one that has such blocks on the register
path while all of its windows run at once, by the window's width and the device's SMs."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def first_kernel(call, stream):
    cu = ctypes.CDLL("libcuda.so.1")
    h = ctypes.c_void_p(stream.cuda_stream)
    graph, n = ctypes.c_void_p(), ctypes.c_size_t(1)
    stream.synchronize()
    assert cu.cuStreamBeginCapture_v2(h, 2) == 0    # relaxed
    try:
        call()
    finally:
        rc = cu.cuStreamEndCapture(h, ctypes.byref(graph))
    assert rc == 0
    node, params, name = ctypes.c_void_p(), (ctypes.c_uint64 * 32)(), ctypes.c_char_p()
    assert cu.cuGraphGetNodes(graph, ctypes.byref(node), ctypes.byref(n)) == 0
    assert cu.cuGraphKernelNodeGetParams_v2(node, params) == 0
    func = params[0] or params[7]   # CUfunction, or a CUkernel of it
    if params[0]:
        assert cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(func)) == 0
    else:
        assert cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(func)) == 0
    out = name.value.decode()
    cu.cuGraphDestroy(graph)
    return out


@pytest.mark.parametrize("NT,per_sm", [(64, 11), (128, 6), (256, 3)])
def test_kernel_by_windows_at_once(NT, per_sm):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1002_2469_gb300 as D
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    t = (-1.2, 2.5, -0.8)
    s = torch.cuda.Stream()
    i = D.Plan(*t, 1 << 22, precision=1, threads=NT, block_size=16).info
    rows = 16 * (2 * NT - i["halo_l"] - i["halo_r"])
    for windows, kind in ((per_sm * sms - 1, 4), (per_sm * sms + 1, 0)):
        N = rows * windows - 5
        plan = D.Plan(*t, N, precision=1, threads=NT, block_size=16)
        assert plan.info["tiles"] == windows and plan.info["n_last"] == 11
        F = torch.randn(N, dtype=torch.float64, device="cuda")
        x = torch.empty_like(F)
        torch.cuda.synchronize()
        name = first_kernel(lambda: D.dichotomy_solve(plan.handle, F, x, s.cuda_stream), s)
        assert "k_window2" in name and "ILi%dELi%dE" % (NT, kind) in name, name
