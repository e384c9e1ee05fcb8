"""N-body steps of a heap with more bodies than its handle placed there, and of
the largest heaps that the kernels of unordered pairs serve (csrc/dsr_nbody.cu,
kSymPositions): one step against the FP64 oracle, at the bar of the other
n-body tests (1e-4 relative; the bodies start at rest, so their velocities are
the forces)."""
import ctypes as C
import os

import numpy as np
import pytest
import torch

import oracle as O
from paper_1809_07444_gb300 import _lib as L
from paper_1809_07444_gb300.apps import NBODY_TYPES, NBody
from paper_1809_07444_gb300.heap import heap_bytes_for_blocks

from helpers import check_invariants
from test_gpu_nbody import _compare

pytestmark = pytest.mark.gpu


def _rows(n, seed):
    """Uniform positions, at rest; no two bodies come within a merge distance of 1e-6."""
    rng = np.random.default_rng(seed)
    rows = np.zeros((n, 7))
    rows[:, :3] = rng.random((n, 3))
    rows[:, 6] = 10 ** rng.uniform(-3, 0, n)
    return rows.astype(np.float32).astype(np.float64)


def _add_bodies(g, rows):
    """Place `rows` in g's heap as a program of its own would, with ids from g.n0 on."""
    ws = torch.empty(g.workspace.numel(), dtype=torch.uint8, device="cuda")
    dev = torch.from_numpy(rows.astype(np.float32)).cuda()
    h = C.c_void_p()
    L.check(g.lib.dsr_nbody_create(g.heap.handle, C.byref(g.params), C.c_void_p(dev.data_ptr()), len(rows),
                                   C.c_void_p(ws.data_ptr()), g.log_cap, None, C.byref(h)), "dsr_nbody_create")
    torch.cuda.synchronize()
    L.check(g.lib.dsr_nbody_destroy(h))
    # the second placement numbered its bodies from 0 as well
    f, refs = g.heap.dump(0)
    xyz = f[:, 1:4].view(np.float32)
    first = {tuple(p): i for i, p in enumerate(rows[:, :3].astype(np.float32))}
    lay = g.heap.layout()
    data = g.heap.arena[lay.off_data:].cpu().numpy()
    for p, r in zip(xyz, refs):
        i = first.get(tuple(p))
        if i is not None:
            at = (int(r) >> 6) * lay.block_bytes + lay.field_offset[0][0] + 4 * (int(r) & 63)
            data[at: at + 4] = np.frombuffer(np.int32(g.n0 + i).tobytes(), np.uint8)
    g.heap.arena[lay.off_data:].copy_(torch.from_numpy(data))


def _step_and_compare(g, rows):
    O.set_threads(os.cpu_count() or 8)
    o = O.NBody(rows, r_merge=1e-6)
    g.step(1)
    o.step(1)
    _compare(g.dump(), o.dump())
    assert g.heap.stats()["error_flags"] == 0
    check_invariants(g.heap, [len(rows)])


@pytest.mark.parametrize("n0,n,pairs", [
    (100, 8200, "fp32"), (4097, 8200, "fp32"), (100, 20480, "fp32"),  # tile groups of 1 tile -> 2, 3
    (16385, 40000, "fp32"),                                           # the form for many bodies: 3 -> 5
    (100, 8200, "fp64"), (8000, 16385, "fp64"), (8000, 40000, "fp64"),  # 1 -> 1, 5, 10
])
def test_more_bodies_than_at_creation(n0, n, pairs):
    rows = _rows(n, n0 + n)
    g = NBody(rows[:n0], pairs=pairs, r_merge=1e-6, heap_bytes=heap_bytes_for_blocks(NBODY_TYPES, -(-n // 64) + 8))
    _add_bodies(g, rows[n0:])
    _step_and_compare(g, rows)


# 2560 blocks have exactly the most positions; one more takes the other kernels
@pytest.mark.parametrize("blocks", [2560, 2561])
def test_largest_heap_of_unordered_pairs(blocks):
    rows = _rows(163800, blocks)
    g = NBody(rows, r_merge=1e-6, heap_bytes=heap_bytes_for_blocks(NBODY_TYPES, blocks))
    assert g.heap.layout().n_blocks == blocks
    _step_and_compare(g, rows)


@pytest.mark.parametrize("n", [16385, 33000])
def test_fp64_pairs_of_many_bodies(n):
    # beyond 16,384 positions a body has 32 entries a side, and groups several tiles
    rows = _rows(n, n)
    g = NBody(rows, pairs="fp64", r_merge=1e-6, heap_bytes=heap_bytes_for_blocks(NBODY_TYPES, -(-n // 64) + 8))
    _step_and_compare(g, rows)
