"""Whether a decode launch takes clusters must not depend on which layer ran first: one kernel
serves clusters of two and of four, and how many of each are resident at once are different
questions.  Read off captured launches (their cluster attribute), in fresh processes."""
import os
import subprocess
import sys
import textwrap

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Captures one call per shape, in the order given, and prints the cluster size of each launch.
CHILD = """
import ctypes, sys
import torch
from paper_2606_12487_gb300 import dptq
cu = ctypes.CDLL("libcuda.so.1")
def check(r):
    assert r == 0, r
dptq.dptq_reserve(32, 4096, 0)
layers, ins, outs, s = [], [], [], torch.cuda.Stream()
for n in map(int, sys.argv[1].split(",")):
    layers.append(dptq.dptq_pack_weights(torch.randn((n, 4096), device="cuda").half(), 4096))
    ins.append(torch.randn((32, 4096), device="cuda").half())
    outs.append(torch.empty((32, n), dtype=torch.float16, device="cuda"))
torch.cuda.synchronize()
for layer, x, out in zip(layers, ins, outs):
    graph, num = ctypes.c_void_p(), ctypes.c_size_t(1)
    check(cu.cuStreamBeginCapture_v2(ctypes.c_void_p(s.cuda_stream), 2))   # relaxed
    dptq.dptq_qlinear(layer, x, 4, out, stream=s)
    check(cu.cuStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)))
    node = ctypes.c_void_p()
    check(cu.cuGraphGetNodes(graph, ctypes.byref(node), ctypes.byref(num)))
    assert num.value == 1, "one launch expected"
    value = (ctypes.c_uint * 16)()
    check(cu.cuGraphKernelNodeGetAttribute(node, 4, value))                # 4: cluster dimension
    print(layer.N, value[0] or 1)                                          # (0: no cluster)
"""


def clusters(*ns):
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(CHILD), ",".join(map(str, ns))], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return dict(map(int, line.split()) for line in r.stdout.splitlines())


def test_clusters_do_not_depend_on_the_order_of_layers():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_12487_gb300 import dptq
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # 4736 channels: the most CTAs that clusters of four can ask for (37 tiles, 148 CTAs)
    ns = (4096, 6144, 4736)
    plan = {n: dptq.dptq_launch_plan(32, n, 4096, 4, sms, 32)["cluster"] for n in ns}
    if sms == 152:
        assert plan == {4096: 4, 6144: 2, 4736: 4}
    alone = {}
    for n in ns:
        alone.update(clusters(n))
    assert all(alone[n] in (1, plan[n]) for n in ns), alone   # none only where they do not all fit
    if sms == 152:
        assert alone[6144] == 2 and alone[4096] == 4, alone
    assert clusters(4096, 6144, 4736) == alone
    assert clusters(6144, 4736, 4096) == alone
