"""dptq_launch_plan against the launches themselves: the grid and the shared memory of captured
calls, read from the graph.  K = 384 and 1152 have an odd number of 128-element blocks, which
layers pad to an even one."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class KernelNodeParams(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def launches(call, stream):
    """(grid, dynamic shared memory) of each kernel that call() puts on `stream`."""
    cu = ctypes.CDLL("libcuda.so.1")
    graph, num, s = ctypes.c_void_p(), ctypes.c_size_t(0), ctypes.c_void_p(stream.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(s, 2) == 0   # relaxed
    call()
    assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(num)) == 0
    nodes = (ctypes.c_void_p * num.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(num)) == 0
    out = []
    for n in nodes:
        p = KernelNodeParams()
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(n), ctypes.byref(p)) == 0
        out.append((p.grid[0], p.smem))
    assert cu.cuGraphDestroy(graph) == 0
    return out


@pytest.mark.parametrize("M,N,K", [(5, 4096, 384), (16, 1024, 1152), (64, 12288, 384), (700, 1024, 384), (700, 1024, 4096),
                                   (1025, 12176, 1152), (100, 512, 128)])
@pytest.mark.parametrize("bits", [4, 8])
def test_captured_launches_are_the_plan(M, N, K, bits):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_12487_gb300 import dptq
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    layer = dptq.dptq_pack_weights(torch.zeros((N, K), dtype=torch.float16, device="cuda"), 128)
    x = torch.zeros((M, K), dtype=torch.float16, device="cuda")
    out = torch.empty((M, N), dtype=torch.float16, device="cuda")
    dptq.dptq_reserve(M, K, 0)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    got = launches(lambda: dptq.dptq_qlinear(layer, x, bits, out, stream=s), s)
    if len(got) == 1:   # one launch: a CTA rotates each row
        p = dptq.dptq_launch_plan(M, N, K, bits, sms, M)
        assert M <= 64 and p["fused"] == 1
    else:
        p = dptq.dptq_launch_plan(M, N, K, bits, sms, 0)
        assert M > 64 and len(got) == 2
    assert (p["grid"], p["smem_bytes"]) in got
    layer.close()
