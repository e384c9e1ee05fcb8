"""The workloads whose speed this framework is measured by.

Every case is a whole pass of a user's program over device-resident inputs: a
simulation is placed in a heap that the program keeps (heap reset, the
application's create call), advanced by a number of steps, and its final state
is read out of the heap (dsr_heap_dump) and put in an order that does not
depend on where the allocator placed an object. The streaming do-all works in
place on a heap that stays as it is.

listed(), draw(rng)   the cases: plain dicts of sizes and options
prepare(case, seed)   what the program has in hand before a pass
run(state)            one pass
work(case)            the bytes and operations a pass cannot do without
exact(case, seed)     the n-body result in FP64; the other cases are integer
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_1809_07444_gb300 import _lib as L
from paper_1809_07444_gb300.apps import Gol, NBody, Sugarscape, Traffic, Wator, WatorBatch
from paper_1809_07444_gb300.heap import Heap, heap_bytes_for_blocks


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest board of the configurations, 100 generations: every
        # generation is a handful of tiny kernels, so latency is all there is
        {"name": "gol_64", "app": "gol", "W": 64, "H": 64, "steps": 100},
        # an ordinary, non-square board of the served jobs' range
        {"name": "gol_1500x1000", "app": "gol", "W": 1500, "H": 1000, "steps": 20},
        # a small ragged torus, as the tests and the short served jobs use
        {"name": "wator_200x130", "app": "wator", "W": 200, "H": 130, "steps": 100},
        # the benchmark's workload: births and deaths all over a large torus
        {"name": "wator_2048", "app": "wator", "W": 2048, "H": 2048, "steps": 20},
        # many independent instances of mixed sizes in one captured step
        {"name": "wator_batch_32", "app": "batch", "n": 32, "lo": 64, "hi": 1024, "sides_seed": 7, "steps": 20},
        # a few thousand bodies: the launches and the spatial sort show
        {"name": "nbody_4097", "app": "nbody", "n": 4097, "pairs": "fp32", "steps": 5},
        # the configurations' n-body, all pairs in FP32 (the default mode)
        {"name": "nbody_65536", "app": "nbody", "n": 65536, "pairs": "fp32", "steps": 2},
        # the FP64 pair mode, which long runs with close encounters need
        {"name": "nbody_8000_fp64", "app": "nbody", "n": 8000, "pairs": "fp64", "steps": 1},
        # open roads at the benchmark's size: cars leave and enter all the time
        {"name": "traffic_8192x4096", "app": "traffic", "R": 8192, "L": 4096, "periodic": False, "steps": 16},
        # agents that look around, move, die and are replaced
        {"name": "sugarscape_4096", "app": "sugar", "W": 4096, "H": 4096, "steps": 8},
        # the allocator by itself: objects of two types created, half of them
        # deleted and replaced, all deleted
        {"name": "alloc_churn_free_4m", "app": "alloc", "n": 1 << 22, "types": 2},
        # a do-all that only streams fields, over a heap with holes
        {"name": "stream_k2_fill75", "app": "stream", "n": 1 << 26, "fields": 2, "fill": 75},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    app = rng.choice(["gol", "wator", "batch", "nbody", "traffic", "sugar", "alloc", "stream"])
    if app in ("gol", "wator"):
        W, H = _log(rng, 24, 2000), _log(rng, 24, 2000)
        return {"app": app, "W": W, "H": H, "steps": 100 if W * H <= 65536 else 20}
    if app == "batch":
        return {"app": app, "n": rng.randint(3, 32), "lo": 64, "hi": _log(rng, 128, 1024),
                "sides_seed": rng.randrange(1000), "steps": rng.randint(10, 20)}
    if app == "nbody":
        if rng.random() < 0.3:
            return {"app": app, "n": _log(rng, 300, 8000), "pairs": "fp64", "steps": 1}
        return {"app": app, "n": _log(rng, 300, 65000), "pairs": "fp32", "steps": 2}
    if app == "traffic":
        return {"app": app, "R": _log(rng, 64, 8000), "L": _log(rng, 64, 4000), "periodic": rng.random() < 0.4,
                "steps": 16}
    if app == "sugar":
        return {"app": app, "W": _log(rng, 64, 4000), "H": _log(rng, 64, 4000), "steps": 8}
    if app == "alloc":
        return {"app": app, "n": _log(rng, 1 << 12, 1 << 22), "types": rng.randint(1, 4)}
    return {"app": app, "n": _log(rng, 1 << 16, 1 << 26), "fields": rng.choice([2, 3, 4, 8]),
            "fill": rng.choice([100, 75])}


# ---------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(n, seed):
    return torch.rand(n, generator=_gen(seed), device="cuda")


def _wator_kinds(W, H, seed):
    """30% of the cells hold a fish, 3% a shark."""
    u = _uniform(W * H, seed)
    return ((u < 0.33).to(torch.uint8) + ((u >= 0.30) & (u < 0.33)).to(torch.uint8)).contiguous()


def _nbody_rows(n, seed):
    """Positions uniform in the unit cube, masses log-uniform in [1e-3, 1], at rest."""
    rng = np.random.default_rng(seed)
    rows = np.zeros((n, 7), dtype=np.float32)
    rows[:, 0:3] = rng.random((n, 3))
    rows[:, 6] = 10.0 ** rng.uniform(-3.0, 0.0, n)
    return rows


def _sugar_inputs(W, H, seed):
    """Two sugar hills; a tenth of the cells hold an agent."""
    y = torch.arange(H, device="cuda", dtype=torch.float32).view(-1, 1)
    x = torch.arange(W, device="cuda", dtype=torch.float32).view(1, -1)
    cap = torch.zeros(H, W, device="cuda")
    for px, py in ((W / 4, H / 4), (3 * W / 4, 3 * H / 4)):
        dx, dy = (x - px).abs(), (y - py).abs()
        dx, dy = torch.minimum(dx, W - dx), torch.minimum(dy, H - dy)
        cap = torch.maximum(cap, 4 - torch.floor(torch.hypot(dx, dy) / (max(W, H) / 10.0)))
    cap = cap.clamp(0, 4).to(torch.uint8)
    g = _gen(seed)
    n = W * H // 10
    cells = torch.randperm(W * H, generator=g, device="cuda")[:n].sort().values
    u = torch.rand(5, n, generator=g, device="cuda", dtype=torch.float64)
    max_age = 60 + (u[0] * 41).long()
    agents = torch.stack([cells % W, cells // W, 5 + (u[1] * 21).long(), 1 + (u[2] * 4).long(), 1 + (u[3] * 6).long(),
                          (u[4] * max_age).long(), max_age], 1).to(torch.int32).contiguous()
    return cap.contiguous(), agents


def _sides(case):
    rng = np.random.default_rng(case["sides_seed"])
    return [int(s) for s in np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["n"]))]


# ---------------------------------------------------------------------------
# reading a state out of its heap
# ---------------------------------------------------------------------------
def _stream():
    return C.c_void_p(torch.cuda.current_stream().cuda_stream)


def _ptr(t, byte_offset=0):
    return C.c_void_p(t.data_ptr() + byte_offset)


class _Dump:
    """Device buffers that the live objects of one type are dumped to: one
    range of rows per heap, a row being the fields and the handle."""

    def __init__(self, words, caps):
        self.words, self.caps = words, caps
        self.first = [0]
        for c in caps:
            self.first.append(self.first[-1] + c)
        self.rows = torch.zeros(max(1, self.first[-1]), words, dtype=torch.int32, device="cuda")
        self.counts = torch.zeros(len(caps), dtype=torch.int64, device="cuda")
        in_range = torch.cat([torch.arange(c, device="cuda") for c in caps]) if len(caps) > 1 else \
            torch.arange(self.first[-1], device="cuda")
        self.at = in_range
        self.heap_of = torch.repeat_interleave(torch.arange(len(caps), device="cuda"),
                                               torch.tensor(caps, device="cuda")) if len(caps) > 1 else None

    def read(self, lib, heap, type_id, k=0):
        L.check(lib.dsr_heap_dump(heap, type_id, _ptr(self.rows, 4 * self.words * self.first[k]), self.caps[k],
                                  _ptr(self.counts, 8 * k), _stream()), "dsr_heap_dump")

    def live(self):
        """Which rows hold an object."""
        return self.at < (self.counts if self.heap_of is None else self.counts[self.heap_of])

    def scatter(self, index, columns, size, empty):
        """The columns of the live rows at `index` of arrays of `size` entries, `empty` elsewhere."""
        index = torch.where(self.live(), index, size)
        out = []
        for c in columns:
            a = torch.full((size + 1,), empty, dtype=torch.int32, device="cuda")
            out.append(a.index_copy_(0, index, c)[:size])
        return out


# ---------------------------------------------------------------------------
# the applications: prepare and run
# ---------------------------------------------------------------------------
def _restart(sim, create, destroy, *args):
    """Places a new simulation in the program's heap: the old handle goes, the heap is emptied, create() fills it."""
    s = _stream()
    L.check(getattr(sim.lib, destroy)(sim.handle), destroy)
    sim.handle = None
    L.check(sim.lib.dsr_heap_reset(sim.heap.handle, s), "dsr_heap_reset")
    h = C.c_void_p()
    L.check(getattr(sim.lib, create)(sim.heap.handle, *args, s, C.byref(h)), create)
    sim.handle = h


class _Gol:
    def __init__(self, case, seed):
        self.W, self.H, self.steps = case["W"], case["H"], case["steps"]
        n = self.W * self.H
        self.alive0 = (_uniform(n, seed) < 0.25).to(torch.uint8)
        self.sim = Gol(self.W, self.H, self.alive0.cpu().numpy())
        self.cells, self.alive = _Dump(5, [n]), _Dump(4, [n])

    def run(self):
        sim, n = self.sim, self.W * self.H
        _restart(sim, "dsr_gol_create", "dsr_gol_destroy", self.W, self.H, _ptr(self.alive0), _ptr(sim.workspace))
        sim.step(self.steps)
        self.cells.read(sim.lib, sim.heap.handle, 0)
        self.alive.read(sim.lib, sim.heap.handle, 1)
        c, a = self.cells.rows, self.alive.rows
        state = self.cells.scatter(c[:, 2].long(), [c[:, 0], c[:, 1]], n, -1)
        objects = self.alive.scatter(a[:, 1].long() * self.W + a[:, 0], [a[:, 0]], n, -1)
        return {"alive": state[0], "count": state[1], "objects": objects[0]}


class _WatorState:
    """Per-cell timers and energies of the agents of one or many tori."""

    def __init__(self, shapes):
        n = [w * h for w, h in shapes]
        self.size = sum(n)
        self.fish, self.sharks = _Dump(5, n), _Dump(6, n)
        one = len(n) == 1
        self.W = shapes[0][0] if one else torch.tensor([w for w, _ in shapes], device="cuda")[self.fish.heap_of]
        self.base = 0 if one else torch.tensor(self.fish.first[:-1], device="cuda")[self.fish.heap_of]

    def read(self, lib, heap, k=0):
        self.fish.read(lib, heap, 0, k)
        self.sharks.read(lib, heap, 1, k)

    def cells(self):
        f, s = self.fish.rows, self.sharks.rows
        fish = self.fish.scatter(f[:, 1].long() * self.W + f[:, 0] + self.base, [f[:, 2]], self.size, -1)
        sharks = self.sharks.scatter(s[:, 1].long() * self.W + s[:, 0] + self.base, [s[:, 2], s[:, 3]], self.size, -1)
        return {"fish_timer": fish[0], "shark_timer": sharks[0], "shark_energy": sharks[1]}


class _Wator:
    def __init__(self, case, seed):
        self.W, self.H, self.steps = case["W"], case["H"], case["steps"]
        self.kind0 = _wator_kinds(self.W, self.H, seed)
        self.sim = Wator(self.W, self.H, self.kind0.cpu().numpy(), seed)
        self.state = _WatorState([(self.W, self.H)])
        self.kinds = torch.zeros(self.W * self.H, dtype=torch.uint8, device="cuda")

    def run(self):
        sim = self.sim
        _restart(sim, "dsr_wator_create", "dsr_wator_destroy", C.byref(sim.params), _ptr(self.kind0),
                 _ptr(sim.workspace))
        sim.step(self.steps)
        L.check(sim.lib.dsr_wator_kinds(sim.handle, _ptr(self.kinds), _stream()), "dsr_wator_kinds")
        self.state.read(sim.lib, sim.heap.handle)
        return dict(self.state.cells(), kinds=self.kinds)


class _Batch:
    """The batch is rewound by copying back the bytes of its arena, which hold
    the heaps and workspaces of all instances (see dsr_wator_attach)."""

    def __init__(self, case, seed):
        sides, self.steps = _sides(case), case["steps"]
        need = sum(WatorBatch.blocks_for(s, s) * 1100 + s * s * 24 for s in sides) + (64 << 20)
        self.batch = WatorBatch(need, max_instances=len(sides))
        self.slots = []
        for i, s in enumerate(sides):
            slot = self.batch.add(s, s, _wator_kinds(s, s, seed * 1000 + i).cpu().numpy(), seed + i)
            if slot is None:
                raise RuntimeError("the arena is too small")
            self.slots.append(slot)
        self.batch.prepare()
        torch.cuda.synchronize()
        self.used = need - self.batch.free_bytes()[1]  # first fit: the free bytes are the arena's end
        self.saved = self.batch.arena[: self.used].clone()
        self.state = _WatorState([(s, s) for s in sides])
        self.kinds = torch.zeros(self.state.size, dtype=torch.uint8, device="cuda")

    def run(self):
        b = self.batch
        b.arena[: self.used].copy_(self.saved)
        b.step(self.steps)
        h = C.c_void_p()
        for k, slot in enumerate(self.slots):
            L.check(b.lib.dsr_wator_batch_heap(b.handle, slot, C.byref(h)), "dsr_wator_batch_heap")
            L.check(b.lib.dsr_wator_batch_kinds(b.handle, slot, _ptr(self.kinds, self.state.fish.first[k]), _stream()),
                    "dsr_wator_batch_kinds")
            self.state.read(b.lib, h, k)
        return dict(self.state.cells(), kinds=self.kinds)


class _NBody:
    def __init__(self, case, seed):
        self.n, self.steps = case["n"], case["steps"]
        rows = _nbody_rows(self.n, seed)
        self.rows = torch.from_numpy(rows).cuda()
        self.sim = NBody(rows, pairs=case["pairs"])
        self.bodies = _Dump(17, [self.n])

    def run(self):
        sim, n = self.sim, self.n
        _restart(sim, "dsr_nbody_create", "dsr_nbody_destroy", C.byref(sim.params), _ptr(self.rows), n,
                 _ptr(sim.workspace), sim.log_cap)
        sim.step(self.steps)
        self.bodies.read(sim.lib, sim.heap.handle, 0)
        rows = self.bodies.rows
        index = torch.where(self.bodies.live(), rows[:, 0].long(), n)
        out = torch.zeros(n + 1, 7, dtype=torch.int32, device="cuda")
        out.index_copy_(0, index, rows[:, 1:8])  # the high words: a component's value rounded to FP32
        out = out[:n].view(torch.float32)
        return {"position": out[:, 0:3], "velocity": out[:, 3:6], "mass": out[:, 6]}


class _Traffic:
    def __init__(self, case, seed):
        self.R, self.L, self.steps, self.open = case["R"], case["L"], case["steps"], not case["periodic"]
        n, g = self.R * self.L, _gen(seed)
        car = torch.rand(n, generator=g, device="cuda") < 0.2
        v = torch.randint(0, 6, (n,), generator=g, device="cuda", dtype=torch.int8)
        self.v0 = torch.where(car, v, torch.full_like(v, -1))
        self.sim = Traffic(self.R, self.L, self.v0.cpu().numpy(), seed, periodic=case["periodic"])
        self.cars = _Dump(5, [int(car.sum().item()) + self.R * (self.steps if self.open else 0)])
        self.sources = _Dump(5, [self.R])

    def run(self):
        sim = self.sim
        _restart(sim, "dsr_traffic_create", "dsr_traffic_destroy", C.byref(sim.params), _ptr(self.v0),
                 _ptr(sim.workspace))
        sim.step(self.steps)
        self.cars.read(sim.lib, sim.heap.handle, 0)
        c, s = self.cars.rows, self.sources.rows
        out = {"velocity": self.cars.scatter(c[:, 0].long() * self.L + c[:, 1], [c[:, 2]], self.R * self.L, -1)[0]}
        if self.open:
            self.sources.read(sim.lib, sim.heap.handle, 1)
            out["entered"], out["blocked"] = self.sources.scatter(s[:, 0].long(), [s[:, 1], s[:, 2]], self.R, -1)
        return out


class _Sugar:
    def __init__(self, case, seed):
        self.W, self.H, self.steps = case["W"], case["H"], case["steps"]
        self.cap, self.agents0 = _sugar_inputs(self.W, self.H, seed)
        self.sim = Sugarscape(self.W, self.H, self.cap.cpu().numpy(), self.agents0.cpu().numpy(), seed)
        self.n = self.agents0.shape[0]  # each death is a birth: the population is constant
        self.agents = _Dump(10, [self.n])
        self.sugar = torch.zeros(self.W * self.H, dtype=torch.int32, device="cuda")

    def run(self):
        sim = self.sim
        _restart(sim, "dsr_sugarscape_create", "dsr_sugarscape_destroy", C.byref(sim.params), _ptr(self.cap),
                 _ptr(self.agents0), self.n, _ptr(sim.workspace))
        sim.step(self.steps)
        L.check(sim.lib.dsr_sugarscape_sugar(sim.handle, _ptr(self.sugar), _stream()), "dsr_sugarscape_sugar")
        self.agents.read(sim.lib, sim.heap.handle, 0)
        a = self.agents.rows
        order = torch.argsort(a[:, 1] * self.W + a[:, 0])  # one agent per cell
        return {"agents": a[:, :8][order], "sugar": self.sugar}


class _Alloc:
    FIELDS = [[4, 4], [4, 4, 4], [4, 4, 4, 4], [4, 4, 4, 4, 4, 4]]

    def __init__(self, case, seed):
        self.n, self.k, self.seed = case["n"], case["types"], int(seed)
        types = self.FIELDS[: self.k]
        blocks = sum(-(-self.n * len(t) // (64 * 2)) for t in types) * 2 // self.k + 4096
        self.heap = Heap(types, heap_bytes_for_blocks(types, blocks))
        self.refs = torch.zeros(self.n, dtype=torch.int64, device="cuda")
        self.dumps = [_Dump(len(t) + 2, [self.n]) for t in types]
        self.replaced = torch.zeros(1, dtype=torch.int64, device="cuda")
        self.left = torch.zeros(self.k, dtype=torch.int64, device="cuda")

    def run(self):
        h, n = self.heap, self.n
        h.reset()
        h.bench_alloc(self.refs, self.k, self.seed)
        self.replaced.zero_()
        L.check(h.lib.dsr_bench_churn(h.handle, n, self.k, self.seed + 17, _ptr(self.refs), _ptr(self.replaced),
                                      _stream()), "dsr_bench_churn")
        kinds = []
        for t, d in enumerate(self.dumps):
            d.read(h.lib, h.handle, t)
            kinds.append(d.scatter(d.rows[:, 0].long(), [d.rows[:, 0]], n, -1)[0])
        h.bench_free(self.refs)
        self.left.zero_()
        for t in range(self.k):
            h.parallel_do(t, L.METHOD_COUNT, L.CountArgs(_ptr(self.left, 8 * t)))
        return {"of_type": kinds, "replaced": self.replaced, "left": self.left}


class _Stream:
    """A heap whose every block is allocated, its fields filled from the seed;
    with 75% fill a quarter of the objects (those whose first field is 1
    modulo 4) have been deleted."""

    def __init__(self, case, seed):
        k, blocks = case["fields"], -(-case["n"] // 64)
        types = [[4] * k]
        self.heap = Heap(types, heap_bytes_for_blocks(types, blocks))
        lay = self.heap.layout()
        refs = torch.zeros(int(lay.n_blocks) * 64, dtype=torch.int64, device="cuda")
        self.heap.bench_alloc(refs, 1, 0)
        if self.heap.stats()["live_objects"][0] != refs.numel():
            raise RuntimeError("the heap is not full")
        first = int(lay.off_data)
        self.data = self.heap.arena[first: first + int(lay.n_blocks) * int(lay.block_bytes)].view(torch.int32)
        self.data.random_(0, 1 << 30, generator=_gen(seed))
        if case["fill"] < 100:
            self.heap.parallel_do(0, L.METHOD_DELETE_IF, L.DeleteIfArgs(4, 1))

    def run(self):
        self.heap.parallel_do(0, L.METHOD_STREAM_ADD)
        return self.data


_APPS = {"gol": _Gol, "wator": _Wator, "batch": _Batch, "nbody": _NBody, "traffic": _Traffic, "sugar": _Sugar,
         "alloc": _Alloc, "stream": _Stream}


def prepare(case, seed):
    return _APPS[case["app"]](case, seed)


def run(state):
    return state.run()


# ---------------------------------------------------------------------------
# work and exact results
# ---------------------------------------------------------------------------
def work(case):
    """Per step, every live object's fields and its cell read and written once
    (populations as at the start); the initial state read and the final state
    written once; n-body: 20 operations a pair."""
    app = case["app"]
    if app == "nbody":
        n, t = case["n"], case["steps"]
        return {"bytes": t * n * 60 * 2 + n * 28 * 2, "flops": 20.0 * n * n * t}
    if app == "gol":  # a cell's three words, a quarter as many Alive objects
        n, t = case["W"] * case["H"], case["steps"]
        return {"bytes": t * n * (12 + 8 + 0.25 * 16) + n * (1 + 12), "flops": 0}
    if app in ("wator", "batch"):  # fish 12 bytes, sharks 16, a grid word per cell
        n = case["W"] * case["H"] if app == "wator" else sum(s * s for s in _sides(case))
        return {"bytes": case["steps"] * n * (0.30 * 24 + 0.03 * 32 + 0.33 * 8) + n * (1 + 1 + 12), "flops": 0}
    if app == "traffic":  # a car's road, x, v read, x and v written, its cell's byte read and written
        n = case["R"] * case["L"]
        return {"bytes": case["steps"] * (n * 0.2 * (12 + 8 + 2) + case["R"] * 12) + n * (1 + 4), "flops": 0}
    if app == "sugar":  # an agent's 32 bytes read, 20 written; about 14 cells in sight
        n = case["W"] * case["H"]
        return {"bytes": case["steps"] * n * 0.1 * (32 + 20 + 14 * 4) + n * (1 + 4) + n * 0.1 * (28 + 32), "flops": 0}
    if app == "alloc":  # a reference and a field written, the references read twice, half of both replaced
        return {"bytes": case["n"] * (8 + 4 + 8 + 0.5 * (8 + 4) + 4 + 4 + 8), "flops": 0}
    return {"bytes": case["n"] * case["fill"] / 100 * case["fields"] * 8, "flops": 0}


def _accelerations(x, m, eps2):
    out = torch.empty_like(x)
    for i in range(0, len(x), 1024):
        d = x.unsqueeze(0) - x[i:i + 1024].unsqueeze(1)
        r2 = (d * d).sum(2) + eps2
        out[i:i + 1024] = ((m / (r2 * r2.sqrt())).unsqueeze(2) * d).sum(1)
    return out


def _partners(x, live, r_merge):
    """The lowest other live index within r_merge of each live body, -1 if none."""
    n = len(x)
    out = torch.full((n,), n, dtype=torch.long, device=x.device)
    index = torch.arange(n, device=x.device)
    for i in range(0, n, 1024):
        d = x.unsqueeze(0) - x[i:i + 1024].unsqueeze(1)
        near = ((d * d).sum(2) < r_merge * r_merge) & live & live[i:i + 1024].unsqueeze(1)
        near &= index.unsqueeze(0) != index[i:i + 1024].unsqueeze(1)
        out[i:i + 1024] = torch.where(near, index, n).amin(1)
    return torch.where(out < n, out, -1)


def exact(case, seed):
    if case["app"] != "nbody":
        return None  # whole numbers
    rows = torch.from_numpy(_nbody_rows(case["n"], seed)).cuda().double()
    x, v, m = rows[:, 0:3].clone(), rows[:, 3:6].clone(), rows[:, 6].clone()
    live = torch.ones(len(x), dtype=torch.bool, device="cuda")
    G, eps, dt, r_merge = 1.0, 1e-3, 1e-4, 2e-3
    for _ in range(case["steps"]):
        v += G * _accelerations(x, m, eps * eps) * dt
        x += v * dt
        p = _partners(x, live, r_merge)
        low = torch.arange(len(x), device="cuda")
        low = low[(p > low) & (p[p.clamp(min=0)] == low)]
        high = p[low]
        total = m[low] + m[high]
        for a in (x, v):
            a[low] = (m[low, None] * a[low] + m[high, None] * a[high]) / total[:, None]
            a[high] = 0.0
        m[low], m[high], live[high] = total, 0.0, False
        x[~live], v[~live] = 0.0, 0.0
    return {"position": x, "velocity": v, "mass": m}
