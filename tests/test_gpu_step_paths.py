"""Every route a step or a read-out can take, at the sizes where the route
changes: life and wa-tor heaps around the largest one that steps in a single
cluster (csrc/dsr_gol.cu, dsr_wator.cu: kSmallBlocks), the pair-force kernels
around their tiles, rows and limits (csrc/dsr_nbody.cu), the traffic gap scan's
8-byte words, and dumps whose rows are not all 4-byte words."""
import ctypes as C
import os

import numpy as np
import pytest

import oracle as O
from paper_1809_07444_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

# 128 threads per CTA and a fixed number of CTAs keep to the general path
TUNINGS = [None, {"threads": 128}, {"ctas_per_sm": 2}, {"cap_min": 32, "fanout": 16}]


@pytest.mark.parametrize("blocks", [1023, 1024, 1025])
@pytest.mark.parametrize("tuning", TUNINGS)
def test_wator_around_the_single_cluster_heap(blocks, tuning):
    from paper_1809_07444_gb300.apps import WATOR_TYPES, Wator
    from paper_1809_07444_gb300.heap import heap_bytes_for_blocks

    from helpers import check_invariants

    W, H = 131, 97
    k0 = WL.wator_initial(W, H, blocks)
    g = Wator(W, H, k0, 7, heap_bytes=heap_bytes_for_blocks(WATOR_TYPES, blocks, tuning), tuning=tuning)
    assert g.heap.layout().n_blocks == blocks
    o = O.Wator(W, H, k0, 7)
    for n in (1, 2, 3, 1, 19, 30):  # odd and even numbers of steps in a call
        c0 = g.heap.counters()
        g.step(n)
        ev = np.sum([o.step(1)[0] for _ in range(n)], axis=0)
        c1 = g.heap.counters()
        assert c1["allocs"] - c0["allocs"] == ev[0] + ev[2]
        assert c1["frees"] - c0["frees"] == ev[1] + ev[3]
        assert g.hash() == o.hash()
    for a, b in zip(g.dump(), o.dump()):
        assert np.array_equal(a, b)
    check_invariants(g.heap, list(o.counts()))


@pytest.mark.parametrize("blocks", [767, 768, 769])
@pytest.mark.parametrize("tuning", TUNINGS)
def test_life_around_the_single_cluster_heap(blocks, tuning):
    from paper_1809_07444_gb300.apps import GOL_TYPES, Gol
    from paper_1809_07444_gb300.heap import heap_bytes_for_blocks

    from helpers import check_invariants

    W, H = 83, 61
    s0 = WL.gol_initial(W, H, blocks)
    g = Gol(W, H, s0, heap_bytes=heap_bytes_for_blocks(GOL_TYPES, blocks, tuning), tuning=tuning)
    assert g.heap.layout().n_blocks == blocks
    o = O.Gol(W, H, s0)
    for n in (1, 2, 3, 1, 40):
        g.step(n)
        o.step(n)
        assert g.hash() == o.hash()
    for a, b in zip(g.dump(), o.dump()):
        assert np.array_equal(a, b)
    check_invariants(g.heap, [W * H, o.alive_count()])


# One step against the FP64 oracle, at the bar of the other n-body tests (1e-4
# relative; the bodies start at rest, so their velocities are the forces).
@pytest.mark.parametrize("pairs", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [2, 127, 128, 129, 255, 257, 511, 513, 1023, 1025, 2049])
def test_nbody_around_tiles_and_rows(n, pairs):
    from test_gpu_nbody import _run

    rows, _ = WL.nbody_initial(n, n)
    _run(rows, 1, pairs=pairs)


@pytest.mark.parametrize("n,kw", [(16383, {}), (16385, {}), (32769, {}), (4097, {"eps": 0.0}), (4097, {"eps": 0.0, "pairs": "fp64"}),
                                  (4097, {"r_near": 0.0})])
def test_nbody_around_the_shape_limits(n, kw):
    from test_gpu_nbody import _run

    rows, _ = WL.nbody_initial(n, n)
    _run(rows, 1, threads=os.cpu_count() or 8, **kw)


@pytest.mark.parametrize("n", [163840, 163841])
def test_nbody_around_the_most_symmetric_positions(n):
    # uniform positions; no two bodies come within the merge distance
    from test_gpu_nbody import _run

    rng = np.random.default_rng(n)
    rows = np.zeros((n, 7))
    rows[:, :3] = rng.random((n, 3))
    rows[:, 6] = 10 ** rng.uniform(-3, 0, n)
    rows = rows.astype(np.float32).astype(np.float64)
    _run(rows, 1, threads=os.cpu_count() or 8, r_merge=1e-6)


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("L,vmax", [(2, 1), (7, 6), (8, 7), (9, 8), (17, 15), (24, 16), (33, 17), (128, 127)])
def test_traffic_gaps_around_eight_cells(L, vmax, periodic):
    from paper_1809_07444_gb300.apps import Traffic

    R = 61
    v0 = WL.traffic_initial(R, L, L, density=0.15, vmax=vmax)
    kw = dict(vmax=vmax, p=0.2, alpha=0.6, periodic=periodic)
    g, o = Traffic(R, L, v0, 11, **kw), O.Traffic(R, L, v0, 11, **kw)
    for s in range(30):
        g.step(1)
        o.step(1)
        assert g.hash() == o.hash(), s
    for a, b in zip(g.dump(), o.dump()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("fields", [[4], [4, 8], [4, 8, 4], [4] * 5, [4] + [8] * 3, [4] * 16])
@pytest.mark.parametrize("n", [1, 31, 64, 4097])
@pytest.mark.parametrize("narrow", [False, True])  # a small second type: few objects of the first to a block
def test_dump_rows_and_capacity(fields, n, narrow):
    import torch

    from paper_1809_07444_gb300 import _lib as L
    from paper_1809_07444_gb300.heap import Heap, heap_bytes_for_blocks

    types = [fields, [4]] if narrow else [fields]
    h = Heap(types, heap_bytes_for_blocks(types, 4096))
    refs = torch.zeros(n, dtype=torch.int64, device="cuda")
    h.bench_alloc(refs, 1, 3)
    torch.cuda.synchronize()
    keep = refs[::2].contiguous() if n > 1 else refs
    if n > 1:
        h.bench_free(refs[1::2].contiguous())
    # every object's fields: its handle and the field's number, read back below
    lay = h.layout()
    handles = np.sort(keep.cpu().numpy().view(np.uint64))
    data = h.arena[lay.off_data:].cpu().numpy()
    for k in handles:
        b, s = int(k) >> 6, int(k) & 63
        for f, w in enumerate(fields):
            at = b * lay.block_bytes + lay.field_offset[0][f] + s * w
            data[at: at + w] = np.frombuffer(np.uint64(int(k) * 31 + f).tobytes()[:w], np.uint8)
    h.arena[lay.off_data:].copy_(torch.from_numpy(data))
    rows, got = h.dump(0)
    order = np.argsort(got)
    assert np.array_equal(got[order], handles)
    want = []
    for k in handles:
        words = []
        for f, w in enumerate(fields):
            v = int(k) * 31 + f
            words += [v & 0xFFFFFFFF] + ([v >> 32] if w == 8 else [])
        want.append(words)
    assert np.array_equal(rows[order], np.array(want, dtype=np.uint32).reshape(len(handles), -1))
    assert h.stats()["error_flags"] == 0
    # a buffer too small for the rows: the count is complete, nothing is written past it
    row = h.lib.dsr_row_words(h.handle, 0)
    cap = len(handles) // 2
    out = torch.full((max(len(handles), 1) * row,), -1, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    L.check(h.lib.dsr_heap_dump(h.handle, 0, C.c_void_p(out.data_ptr()), cap, C.c_void_p(cnt.data_ptr()), None), "dump")
    torch.cuda.synchronize()
    assert int(cnt.item()) == len(handles)
    assert (out[cap * row:] == -1).all()
    assert h.stats()["error_flags"] != 0


@pytest.mark.parametrize("R,L,density", [(1, 2, 1.0), (3, 85, 0.5), (64, 64, 1.0), (63, 65, 0.01), (701, 997, 0.03),
                                         (4096, 300, 0.2), (128, 8192, 1.0)])
@pytest.mark.parametrize("tuning", [None, {"cap_min": 32}, {"fanout": 16}])
def test_traffic_initial_cars(R, L, density, tuning):
    from paper_1809_07444_gb300.apps import TRAFFIC_TYPES, Traffic
    from paper_1809_07444_gb300.heap import heap_bytes_for_blocks

    from helpers import check_stats

    v0 = WL.traffic_initial(R, L, R + L, density=density, vmax=1)
    road, x = np.nonzero(v0 >= 0)
    # a heap with few more slots than cars, and one with room
    cap = 32 if tuning and "cap_min" in tuning else 64
    for blocks in (17 * len(x) // (16 * cap) + 64, 4 * (len(x) // cap) + 256):
        g = Traffic(R, L, v0, 1, vmax=1, periodic=True, tuning=tuning,
                    heap_bytes=heap_bytes_for_blocks(TRAFFIC_TYPES, blocks, tuning))
        cars, _ = g.dump()
        assert np.array_equal(cars, np.stack([road, x, v0[road, x]], 1))
        st = check_stats(g.heap)
        assert st["error_flags"] == 0 and st["live_objects"][0] == len(x)
