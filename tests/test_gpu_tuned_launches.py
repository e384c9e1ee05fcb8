"""The kernels of a step run with the heap's tuning: threads per CTA, and CTAs
per SM where it fixes them. The launches are read from a captured graph."""
import ctypes as C

import pytest
import torch

from paper_1809_07444_gb300 import workloads as WL
from paper_1809_07444_gb300.apps import Traffic

pytestmark = pytest.mark.gpu

KERNEL_NODE = 0


class KernelParams(C.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", C.c_void_p), ("grid", C.c_uint * 3), ("block", C.c_uint * 3), ("smem", C.c_uint),
                ("params", C.c_void_p), ("extra", C.c_void_p), ("kern", C.c_void_p), ("ctx", C.c_void_p)]


def launches(call):
    """[(grid, block)] of the kernels that call(stream) queues, none of which runs."""
    cu = C.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    graph, n = C.c_void_p(), C.c_size_t(0)
    assert cu.cuStreamBeginCapture_v2(C.c_void_p(s.cuda_stream), 2) == 0  # relaxed
    try:
        call(s)
    finally:
        assert cu.cuStreamEndCapture(C.c_void_p(s.cuda_stream), C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, C.byref(n)) == 0
    out = []
    for node in nodes:
        kind = C.c_int()
        assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(kind)) == 0
        if kind.value == KERNEL_NODE:
            p = KernelParams()
            assert cu.cuGraphKernelNodeGetParams_v2(C.c_void_p(node), C.byref(p)) == 0
            out.append((p.grid[0], p.block[0]))
    assert cu.cuGraphDestroy(graph) == 0
    return out


SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 0


@pytest.mark.parametrize("tuning", [{"threads": 128, "ctas_per_sm": 2}, {"threads": 1024, "ctas_per_sm": 1},
                                    {"threads": 512, "ctas_per_sm": 2}, {"ctas_per_sm": 3}])
def test_traffic_step(tuning):
    R, L = 1000, 1000
    g = Traffic(R, L, WL.traffic_initial(R, L, 1, density=0.2, vmax=5), 1, tuning=tuning)
    g.step(1)
    torch.cuda.synchronize()
    # list, cars, sources
    got = launches(lambda s: g.step(1, stream=s))
    assert got[1:] == [(tuning["ctas_per_sm"] * SMS, tuning.get("threads", 256))] * 2
