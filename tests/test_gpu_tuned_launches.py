"""The kernels of a step and of a dump run with the heap's tuning: threads per
CTA, and CTAs per SM where it fixes them. The launches are read from a captured
graph."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1809_07444_gb300 import _lib as L
from paper_1809_07444_gb300 import workloads as WL
from paper_1809_07444_gb300.apps import Traffic
from paper_1809_07444_gb300.heap import Heap, _stream_ptr, heap_bytes_for_blocks

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
    R, W = 1000, 1000
    g = Traffic(R, W, WL.traffic_initial(R, W, 1, density=0.2, vmax=5), 1, tuning=tuning)
    g.step(1)
    torch.cuda.synchronize()
    # list, cars, sources
    got = launches(lambda s: g.step(1, stream=s))
    assert got[1:] == [(tuning["ctas_per_sm"] * SMS, tuning.get("threads", 256))] * 2


@pytest.mark.parametrize("tuning", [{"threads": 64, "ctas_per_sm": 1}, {"threads": 128, "ctas_per_sm": 2},
                                    {"threads": 1024, "ctas_per_sm": 1}, {"threads": 768}, {"ctas_per_sm": 3}])
@pytest.mark.parametrize("fields", [[4, 4], [4] + [8] * 15])
def test_dump(tuning, fields):
    h = Heap([fields], heap_bytes_for_blocks([fields], 40_000, tuning), tuning=tuning)
    threads = tuning.get("threads", 256)
    row = h.lib.dsr_row_words(h.handle, 0)
    out = torch.empty(16, dtype=torch.int64, device="cuda")
    got = launches(lambda s: L.check(h.lib.dsr_heap_dump(h.handle, 0, C.c_void_p(out.data_ptr()), 1,
                                                         C.c_void_p(out.data_ptr() + 16 * 8 - 8), _stream_ptr(s)), "dump"))
    assert row <= 34 and got[1][1] == threads
    if "ctas_per_sm" in tuning:
        assert got[1][0] == tuning["ctas_per_sm"] * SMS
    # every object, whatever the tuning
    refs = torch.zeros(100_003, dtype=torch.int64, device="cuda")
    h.bench_alloc(refs, 1, 3)
    _, handles = h.dump(0)
    assert np.array_equal(np.sort(handles), np.sort(refs.cpu().numpy().view(np.uint64)))
    assert h.stats()["error_flags"] == 0
