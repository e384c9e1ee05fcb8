// Game of life as an SMMO program (Fig. 6c): three do-alls per generation
// over Cell and Alive objects. Rules: B3/S23 on a torus, Moore neighbourhood.
#include "dsr_apps.h"
#include "dsr_steps.cuh"

namespace {
enum { CELL = 0, ALIVE = 1 };
enum { C_ALIVE = 0, C_COUNT = 1, C_IDX = 2 };
enum { A_X = 0, A_Y = 1 };

struct GolArgs {
    const dsr_ref* cell_ref;  // grid index -> Cell handle
    int32_t W, H;
};

// (i) Cell: number of alive cells among the 8 neighbours.
__device__ __forceinline__ void count_cell(const dsr_dev_heap& H, const GolArgs& a, dsr_ref self) {
    const int idx = *dsr_field<int32_t>(H, CELL, self, C_IDX);
    const int y = idx / a.W, x = idx - y * a.W;
    const int xw = x == 0 ? a.W - 1 : x - 1, xe = x == a.W - 1 ? 0 : x + 1;
    const dsr_ref* mid = a.cell_ref + (idx - x);
    const dsr_ref* up = a.cell_ref + (dsr_u64)(y == 0 ? a.H - 1 : y - 1) * a.W;
    const dsr_ref* down = a.cell_ref + (dsr_u64)(y == a.H - 1 ? 0 : y + 1) * a.W;
    const dsr_ref c[8] = {up[xw], up[x], up[xe], mid[xw], mid[xe], down[xw], down[x], down[xe]};
    int n = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        if (c[k] != DSR_NULL) n += *dsr_field<int32_t>(H, CELL, c[k], C_ALIVE);
    *dsr_field<int32_t>(H, CELL, self, C_COUNT) = n;
}

// (ii) Alive: death when the cell's count is not 2 or 3.
__device__ __forceinline__ void die(const dsr_dev_heap& H, const GolArgs& a, dsr_ref self) {
    const int x = *dsr_field<int32_t>(H, ALIVE, self, A_X);
    const int y = *dsr_field<int32_t>(H, ALIVE, self, A_Y);
    const dsr_ref c = a.cell_ref[y * a.W + x];
    if (c == DSR_NULL) return;
    const int n = *dsr_field<int32_t>(H, CELL, c, C_COUNT);
    if (n != 2 && n != 3) {
        *dsr_field<int32_t>(H, CELL, c, C_ALIVE) = 0;
        dsr_delete(H, self);
    }
}

// (iii) Cell: birth of a dead cell with exactly 3 alive neighbours: true for
// one, which is alive from here on and has the grid index *idx.
__device__ __forceinline__ bool birth(const dsr_dev_heap& H, dsr_ref self, int* idx) {
    int32_t* alive = dsr_field<int32_t>(H, CELL, self, C_ALIVE);
    const int was = *alive, n = *dsr_field<int32_t>(H, CELL, self, C_COUNT);
    if (was || n != 3) return false;
    *alive = 1;
    *idx = *dsr_field<int32_t>(H, CELL, self, C_IDX);
    return true;
}
__device__ __forceinline__ void gol_born(const dsr_dev_heap& H, const GolArgs& a, int idx, dsr_ref r) {
    if (r == DSR_NULL) return;
    *dsr_field<int32_t>(H, ALIVE, r, A_X) = idx % a.W;
    *dsr_field<int32_t>(H, ALIVE, r, A_Y) = idx / a.W;
}

// ---- list do-alls (dsr_parallel_do) ----------------------------------------
struct MCount {
    typedef GolArgs Args;
    static __device__ void run(const dsr_dev_heap& H, int, const Args& a, dsr_ref self) { count_cell(H, a, self); }
};
struct MDie {
    typedef GolArgs Args;
    static __device__ void run(const dsr_dev_heap& H, int, const Args& a, dsr_ref self) { die(H, a, self); }
};
struct MBirth {
    typedef GolArgs Args;
    static __device__ void run(const dsr_dev_heap& H, int, const Args& a, dsr_ref self) {
        int idx;
        if (birth(H, self, &idx)) gol_born(H, a, idx, dsr_new(H, ALIVE));
    }
};

// ---- the plain and the batched generation (dsr_steps.cuh) ------------------
// A: GolArgs (plain form), or GolBatchArgs: heap index h of a group is the
// instance slot, table[h] its view (cell_ref == nullptr: unused slot).
struct GolBatchArgs {
    const GolArgs* table;
};
__device__ __forceinline__ const GolArgs& inst_of(const GolArgs& a, uint32_t) { return a; }
__device__ __forceinline__ const GolArgs& inst_of(const GolBatchArgs& a, uint32_t h) { return a.table[h]; }

struct NoCtx {};
template <class A>
struct GolMethod {
    typedef A Args;
    typedef GolArgs Inst;
    typedef NoCtx Ctx;
    typedef dsr_no_acc Acc;
    enum { kDefers = DSR_NOTHING, kMarks = 0 };
    static __device__ __forceinline__ const GolArgs& inst(const A& a, uint32_t h) { return inst_of(a, h); }
    static __device__ __forceinline__ NoCtx begin(const GolArgs&) { return {}; }
    static __device__ __forceinline__ void flush(const dsr_dev_heap&, const GolArgs&, dsr_no_acc) {}
};
template <class A>
struct DCount : GolMethod<A> {
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap& H, int, const GolArgs& a, NoCtx, dsr_ref self,
                                                   dsr_later&, dsr_no_acc&) {
        count_cell(H, a, self);
        return 0;
    }
};
template <class A>
struct DDie : GolMethod<A> {
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap& H, int, const GolArgs& a, NoCtx, dsr_ref self,
                                                   dsr_later&, dsr_no_acc&) {
        die(H, a, self);
        return 0;
    }
};
template <class A>
struct DBirth : GolMethod<A> {
    enum { kDefers = ALIVE, kDeferBack = 1 };
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap& H, int, const GolArgs&, NoCtx, dsr_ref self,
                                                   dsr_later& later, dsr_no_acc&) {
        int idx;
        if (birth(H, self, &idx)) later.push((dsr_u64)idx);
        return 0;
    }
    static __device__ __forceinline__ void born(const dsr_dev_heap& H, const GolArgs& a, dsr_u64 idx, dsr_ref r) {
        gol_born(H, a, (int)idx, r);
    }
};
// One scan lists both types. A birth and a death never meet: a cell that
// dies has not 3 alive neighbours, and new Alive objects are in no list. They
// share a launch where memory never runs short while no death has given its
// slot back (deaths_may_wait); else the deaths come first.
constexpr dsr_phase kCells{CELL, 0}, kAlive{ALIVE, 1};
// A list of its own for each do-all, of a type and its subtypes.
constexpr dsr_phase kAliveTree{ALIVE, 0};

// Generations of a small board in one launch of one cluster (dsr_steps.cuh).
// No Cell is ever created or deleted after the first list, which so serves
// all generations; the Alive objects are listed while the cells count, which
// leaves them alone: two barriers a generation.
__global__ void __launch_bounds__(DSR_CLUSTER_THREADS, 1)
    k_gol_steps(const __grid_constant__ dsr_dev_heap H, const __grid_constant__ GolArgs a, int n, int apart) {
    constexpr int T = DSR_CLUSTER_THREADS;
    typedef GolArgs A;
    __shared__ dsr_later_smem<T> later;
    __shared__ dsr_list_smem<T> list;
    __shared__ uint32_t len[2];
    const dsr_heap_space S{H, len};
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    const dsr_phase cells{CELL, 0}, alive{ALIVE, 1};
    const unsigned hc = H.span_sh[CELL] - 5, ha = H.span_sh[ALIVE] - 5;
    dsr_clear_sets(H.R_count, first);
    dsr_cluster_barrier();
    // the cells' list length stays in set 0's front word, the Alive objects'
    // take turns in the two back words
    dsr_list<T>(H, CELL, -1, 2u * (unsigned)n, 0, DSR_SET, list);
    dsr_cluster_barrier();
    dsr_set_lengths(H.R_count, DSR_SET, len);
    for (int t = 0; t < n; ++t) {
        const uint32_t set = DSR_SET + 2 * (t & 1), other = DSR_SET + 2 * (~t & 1);
        dsr_list<T>(H, -1, ALIVE, 0, 1, set, list);
        if (first) *(volatile uint32_t*)(H.R_count + other + 1) = 0;
        dsr_run_list<DCount<A>, dsr_heap_space, T>(S, cells, a, hc, false, nullptr);
        dsr_cluster_barrier();
        if (threadIdx.x == 0) len[1] = *(volatile uint32_t*)(H.R_count + set + 1);
        __syncthreads();
        if (apart) {
            dsr_run_list<DDie<A>, dsr_heap_space, T>(S, alive, a, ha, false, nullptr);
            dsr_cluster_barrier();
        }
        dsr_run_list<DBirth<A>, dsr_heap_space, T>(S, cells, a, hc, false, &later);
        if (!apart) dsr_run_list<DDie<A>, dsr_heap_space, T>(S, alive, a, ha, true, nullptr);
        dsr_cluster_barrier();
    }
    dsr_clear_sets(H.R_count, first);
}

// One thread per cell: create the Cell and, where alive, its Alive object.
__global__ void __launch_bounds__(DSR_BULK_THREADS)
    k_gol_init(const __grid_constant__ dsr_dev_heap H, const uint8_t* alive0, dsr_ref* cell_ref, int W, int Hh,
               int rows) {
    __shared__ dsr_bulk_smem<2> sm;
    const int types[2] = {CELL, ALIVE};
    dsr_bulk_create(
        H, (dsr_u64)W * Hh, rows, types, sm, [&](dsr_u64 i) { return alive0[i] ? 3u : 1u; },
        [&](dsr_u64 i, unsigned kind, const dsr_ref (&ref)[2]) {
            cell_ref[i] = ref[0];
            if (ref[0] != DSR_NULL) {
                *dsr_field<int32_t>(H, CELL, ref[0], C_ALIVE) = kind >> 1;
                *dsr_field<int32_t>(H, CELL, ref[0], C_COUNT) = 0;
                *dsr_field<int32_t>(H, CELL, ref[0], C_IDX) = (int32_t)i;
            }
            if (ref[1] != DSR_NULL) {
                *dsr_field<int32_t>(H, ALIVE, ref[1], A_X) = (int32_t)((uint32_t)i % (uint32_t)W);
                *dsr_field<int32_t>(H, ALIVE, ref[1], A_Y) = (int32_t)((uint32_t)i / (uint32_t)W);
            }
        });
}

int launch_init(const dsr_heap* heap, int W, int H, const void* alive0_dev, void* cell_ref_dev, cudaStream_t s) {
    const dsr_u64 n = (dsr_u64)W * H;
    const int rows = dsr__bulk_rows<2>(n, heap->sm_count);
    k_gol_init<<<dsr__bulk_grid(n, rows, heap->sm_count), DSR_BULK_THREADS, 0, s>>>(
        heap->dev, static_cast<const uint8_t*>(alive0_dev), static_cast<dsr_ref*>(cell_ref_dev), W, H, rows);
    return dsr__check_launch("k_gol_init");
}

// Whether the births of a generation find room before its deaths have given
// theirs back, whatever the state of the board: a cell holds an Alive object or
// gets one, never both, so there are at most as many as cells. Of the cells'
// blocks twice as many as full ones are reckoned, as a chunk's objects beyond
// its full blocks may lie in blocks of their own (dsr_bulk.cuh). Other types
// may hold any number of blocks. The default heaps have more than that.
bool deaths_may_wait(const dsr_heap* h, int W, int Hh) {
    const dsr_layout& L = h->layout;
    const dsr_u64 n = (dsr_u64)W * Hh, cc = L.capacity[CELL], ca = L.capacity[ALIVE];
    return L.n_types == 2 && L.n_blocks >= 2 * ((n + cc - 1) / cc) + (n + ca - 1) / ca;
}

const int kCellFields[3] = {4, 4, 4};
const int kAliveFields[2] = {4, 4};

bool heap_matches(const dsr_heap* h) {
    const dsr_layout& L = h->layout;
    if (L.n_types < 2 || L.n_fields[CELL] != 3 || L.n_fields[ALIVE] != 2) return false;
    for (int f = 0; f < 3; ++f)
        if (L.field_bytes[CELL][f] != 4) return false;
    for (int f = 0; f < 2; ++f)
        if (L.field_bytes[ALIVE][f] != 4) return false;
    return true;
}
}  // namespace

struct dsr_gol {
    dsr_heap* heap;
    GolArgs args;
    cudaStream_t capture = nullptr;   // stream the generation is captured on
    cudaGraphExec_t exec = nullptr;   // one generation as a graph
};

extern "C" int dsr_gol_types(dsr_type_desc* out) {
    if (!out) return DSR_E_INVALID;
    out[0] = dsr_type_desc{"Cell", 3, kCellFields};
    out[1] = dsr_type_desc{"Alive", 2, kAliveFields};
    return DSR_OK;
}

extern "C" int dsr_gol_workspace_bytes(int W, int H, size_t* out) {
    if (!out || W < 3 || H < 3 || (int64_t)W * H > (1ll << 31)) return DSR_E_INVALID;
    *out = (size_t)W * H * sizeof(dsr_ref);
    return DSR_OK;
}

extern "C" int dsr_gol_create(dsr_heap* heap, int W, int H, const void* alive0_dev, void* workspace_dev,
                              void* stream, dsr_gol** out) {
    size_t ws;
    if (!heap || !alive0_dev || !workspace_dev || !out || dsr_gol_workspace_bytes(W, H, &ws)) return DSR_E_INVALID;
    if (!heap_matches(heap)) return DSR_E_INVALID;
    dsr_gol* g = new dsr_gol;
    g->heap = heap;
    g->args = GolArgs{static_cast<const dsr_ref*>(workspace_dev), W, H};
    int rc = launch_init(heap, W, H, alive0_dev, workspace_dev, dsr__stream(stream));
    if (rc) {
        delete g;
        return rc;
    }
    *out = g;
    return DSR_OK;
}

static bool has_subtypes(const dsr_heap* h) { return dsr__has_subtypes(h, CELL) || dsr__has_subtypes(h, ALIVE); }

static int issue_generation(dsr_gol* g, cudaStream_t s) {
    typedef GolArgs A;
    if (has_subtypes(g->heap)) {
        dsr__list_tree(g->heap, CELL, 1, s);
        int rc = dsr__step<DCount<A>, dsr_no_method, true>(g->heap, kCells, kCells, g->args, s);
        dsr__list_tree(g->heap, ALIVE, 1, s);
        if (!rc) rc = dsr__step<DDie<A>, dsr_no_method, true>(g->heap, kAliveTree, kAliveTree, g->args, s);
        dsr__list_tree(g->heap, CELL, 1, s);
        if (!rc) rc = dsr__step<DBirth<A>, dsr_no_method, true>(g->heap, kCells, kCells, g->args, s);
        return rc;
    }
    dsr__list_types(g->heap, CELL, ALIVE, 2, 1, s);
    int rc = dsr__step<DCount<A>>(g->heap, kCells, kCells, g->args, s);
    if (deaths_may_wait(g->heap, g->args.W, g->args.H)) {
        if (!rc) rc = dsr__step<DBirth<A>, DDie<A>, true>(g->heap, kCells, kAlive, g->args, s);
        return rc;
    }
    if (!rc) rc = dsr__step<DDie<A>>(g->heap, kAlive, kAlive, g->args, s);
    if (!rc) rc = dsr__step<DBirth<A>, dsr_no_method, true>(g->heap, kCells, kCells, g->args, s);
    return rc;
}

// A generation's launches take a few microseconds each on a board of some
// hundred cells a side, so the generation is captured once into a CUDA graph
// (its kernel arguments never change) and replayed: one launch per generation.
// Heaps up to this many blocks (a board of about 80 x 80 with the default heap)
// run their generations in one cluster: 10 against 17 us a generation at 278
// blocks, 13 and 18 at 580, 23 and 20 at 984.
constexpr dsr_u64 kSmallBlocks = 768;

extern "C" int dsr_gol_step(dsr_gol* g, int n_gen, void* stream) {
    if (!g || n_gen < 0) return DSR_E_INVALID;
    cudaStream_t s = dsr__stream(stream);
    static dsr_per_device fits;
    if (dsr__small_heap(g->heap, kSmallBlocks) && !has_subtypes(g->heap) &&
        dsr__cluster_fits(g->heap, (const void*)k_gol_steps, &fits)) {
        int apart = deaths_may_wait(g->heap, g->args.W, g->args.H) ? 0 : 1;
        for (int i = 0; i < n_gen;) {
            int n = n_gen - i < DSR_CLUSTER_STEPS ? n_gen - i : DSR_CLUSTER_STEPS;
            void* args[] = {&g->heap->dev, &g->args, &n, &apart};
            const int rc = dsr__launch_cluster((const void*)k_gol_steps, args, s);
            if (rc) return rc;
            i += n;
        }
        return DSR_OK;
    }
    if (!g->exec && n_gen > 0) {
        cudaError_t e = g->capture ? cudaSuccess : cudaStreamCreateWithFlags(&g->capture, cudaStreamNonBlocking);
        cudaGraph_t graph = nullptr;
        if (!e) e = cudaStreamBeginCapture(g->capture, cudaStreamCaptureModeThreadLocal);
        if (e) {
            dsr__set_cuda_error(e, "dsr_gol_step capture");
            return DSR_E_CUDA;
        }
        const int rc = issue_generation(g, g->capture);
        e = cudaStreamEndCapture(g->capture, &graph);
        if (rc) {
            if (graph) cudaGraphDestroy(graph);
            return rc;
        }
        if (!e) e = cudaGraphInstantiate(&g->exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e) {
            dsr__set_cuda_error(e, "dsr_gol_step instantiate");
            g->exec = nullptr;
            return DSR_E_CUDA;
        }
    }
    for (int i = 0; i < n_gen; ++i) {
        const cudaError_t e = cudaGraphLaunch(g->exec, s);
        if (e) {
            dsr__set_cuda_error(e, "dsr_gol_step launch");
            return DSR_E_CUDA;
        }
    }
    return DSR_OK;
}

extern "C" int dsr_gol_destroy(dsr_gol* g) {
    if (!g) return DSR_OK;
    if (g->exec) cudaGraphExecDestroy(g->exec);
    if (g->capture) cudaStreamDestroy(g->capture);
    delete g;
    return DSR_OK;
}

// dsr_parallel_do entry for the game-of-life methods. Args: dsr_gol_method_args
// = { const uint64_t* cell_ref_dev; int32_t W, H; }.
int dsr__gol_method(dsr_heap* h, int type, int method, const void* args, size_t bytes, cudaStream_t s,
                    bool with_scan) {
    if (!heap_matches(h) || !args || bytes != sizeof(GolArgs)) return DSR_E_INVALID;
    GolArgs a;
    memcpy(&a, args, sizeof a);
    switch (method) {
        case DSR_METHOD_GOL_COUNT:
            return type == CELL ? dsr__doall<MCount>(h, type, a, s, with_scan) : DSR_E_INVALID;
        case DSR_METHOD_GOL_DIE:
            return type == ALIVE ? dsr__doall<MDie>(h, type, a, s, with_scan) : DSR_E_INVALID;
        case DSR_METHOD_GOL_BIRTH:
            return type == CELL ? dsr__doall<MBirth>(h, type, a, s, with_scan) : DSR_E_INVALID;
        default:
            return DSR_E_INVALID;
    }
}

// ===========================================================================
// batched form: many game-of-life instances in one heap group
// ===========================================================================

namespace {
size_t gol_table_bytes(int n) { return ((size_t)n * sizeof(GolArgs) + 1023) / 1024 * 1024; }
}  // namespace

struct dsr_gol_batch {
    dsr_group* group;
    GolArgs* table_d;
    std::vector<GolArgs> table_h;
    bool table_pooled = false;  // the table came from the group's pool (shared arena)
    cudaStream_t capture;
    cudaGraphExec_t exec = nullptr;
    uint64_t exec_epoch = ~0ull;
};

// The rest of a batch's creation once its group and table exist.
static int finish_gol_batch(dsr_gol_batch* b, int max_instances, void* stream, dsr_gol_batch** out) {
    b->table_h.assign(max_instances, GolArgs{nullptr, 0, 0});
    cudaError_t e = cudaMemsetAsync(b->table_d, 0, gol_table_bytes(max_instances), dsr__stream(stream));
    if (!e) e = cudaStreamCreateWithFlags(&b->capture, cudaStreamNonBlocking);
    if (e) {
        dsr__set_cuda_error(e, "dsr_gol_batch_create");
        if (b->table_pooled) dsr__group_give_bytes(b->group, b->table_d, gol_table_bytes(max_instances));
        dsr_group_destroy(b->group);
        delete b;
        return DSR_E_CUDA;
    }
    *out = b;
    return DSR_OK;
}

extern "C" int dsr_gol_batch_create(void* arena_dev, size_t arena_bytes, int max_instances, const dsr_tuning* tune,
                                    void* stream, dsr_gol_batch** out) {
    if (!arena_dev || !out || max_instances < 1 || (reinterpret_cast<uintptr_t>(arena_dev) & 255)) return DSR_E_INVALID;
    const size_t tb = gol_table_bytes(max_instances);
    if (arena_bytes <= tb) return DSR_E_OOM;
    dsr_type_desc types[2];
    dsr_gol_types(types);
    dsr_gol_batch* b = new dsr_gol_batch;
    int rc = dsr_group_create(types, 2, static_cast<uint8_t*>(arena_dev) + tb, arena_bytes - tb, max_instances, tune,
                              stream, &b->group);
    if (rc) {
        delete b;
        return rc;
    }
    b->table_d = static_cast<GolArgs*>(arena_dev);
    return finish_gol_batch(b, max_instances, stream, out);
}

extern "C" int dsr_gol_batch_create_shared(dsr_group* pool_of, int max_instances, const dsr_tuning* tune,
                                           void* stream, dsr_gol_batch** out) {
    if (!pool_of || !out || max_instances < 1) return DSR_E_INVALID;
    dsr_type_desc types[2];
    dsr_gol_types(types);
    dsr_gol_batch* b = new dsr_gol_batch;
    int rc = dsr_group_create_shared(types, 2, pool_of, max_instances, tune, stream, &b->group);
    if (rc) {
        delete b;
        return rc;
    }
    void* t = nullptr;
    rc = dsr__group_take_bytes(b->group, gol_table_bytes(max_instances), &t);
    if (rc) {
        dsr_group_destroy(b->group);
        delete b;
        return rc;
    }
    b->table_d = static_cast<GolArgs*>(t);
    b->table_pooled = true;
    return finish_gol_batch(b, max_instances, stream, out);
}

extern "C" int dsr_gol_batch_instance_bytes(const dsr_gol_batch* b, int W, int H, uint64_t n_blocks, size_t* out) {
    size_t ws;
    if (!b || !out || dsr_gol_workspace_bytes(W, H, &ws)) return DSR_E_INVALID;
    return dsr_group_heap_bytes(b->group, n_blocks, ws, out);
}

extern "C" int dsr_gol_batch_add(dsr_gol_batch* b, int W, int H, uint64_t n_blocks, const void* alive0_dev,
                                 void* stream, int* inst_out) {
    size_t ws;
    if (!b || !alive0_dev || !inst_out || n_blocks == 0 || dsr_gol_workspace_bytes(W, H, &ws)) return DSR_E_INVALID;
    int slot = -1;
    dsr_heap* heap = nullptr;
    void* extra = nullptr;
    int rc = dsr_group_add_heap(b->group, n_blocks, ws, stream, &slot, &heap, &extra);
    if (rc) return rc;
    cudaStream_t s = dsr__stream(stream);
    rc = launch_init(heap, W, H, alive0_dev, extra, s);
    if (rc) return rc;
    b->table_h[slot] = GolArgs{static_cast<const dsr_ref*>(extra), W, H};
    cudaError_t e = cudaMemcpyAsync(b->table_d + slot, &b->table_h[slot], sizeof(GolArgs), cudaMemcpyHostToDevice, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (e) {
        dsr__set_cuda_error(e, "dsr_gol_batch_add");
        return DSR_E_CUDA;
    }
    *inst_out = slot;
    return DSR_OK;
}

extern "C" int dsr_gol_batch_remove(dsr_gol_batch* b, int inst) {
    if (!b || inst < 0 || inst >= (int)b->table_h.size() || !b->table_h[inst].cell_ref) return DSR_E_INVALID;
    b->table_h[inst] = GolArgs{nullptr, 0, 0};
    cudaError_t e = cudaMemcpy(b->table_d + inst, &b->table_h[inst], sizeof(GolArgs), cudaMemcpyHostToDevice);
    if (e) {
        dsr__set_cuda_error(e, "dsr_gol_batch_remove");
        return DSR_E_CUDA;
    }
    return dsr_group_remove_heap(b->group, inst);
}

// One batched generation (the launches of a plain one), captured into a
// CUDA graph once per set of instances.
static int ensure_gol_graph(dsr_gol_batch* b) {
    if (b->exec_epoch == b->group->epoch) return DSR_OK;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
    cudaGraph_t graph = nullptr;
    cudaError_t e = cudaStreamBeginCapture(b->capture, cudaStreamCaptureModeThreadLocal);
    if (e) {
        dsr__set_cuda_error(e, "dsr_gol_batch_step capture");
        return DSR_E_CUDA;
    }
    GolBatchArgs a{b->table_d};
    typedef GolBatchArgs A;
    dsr__group_list_types(b->group, CELL, ALIVE, 2, 1, b->capture);
    int rc = dsr__group_step<DCount<A>>(b->group, kCells, kCells, a, b->capture);
    bool together = true;
    for (size_t i = 0; i < b->table_h.size(); ++i)
        if (b->table_h[i].cell_ref)
            together = together && deaths_may_wait(b->group->heaps[i], b->table_h[i].W, b->table_h[i].H);
    if (together) {
        if (!rc) rc = dsr__group_step<DBirth<A>, DDie<A>, true>(b->group, kCells, kAlive, a, b->capture);
    } else {
        if (!rc) rc = dsr__group_step<DDie<A>>(b->group, kAlive, kAlive, a, b->capture);
        if (!rc) rc = dsr__group_step<DBirth<A>, dsr_no_method, true>(b->group, kCells, kCells, a, b->capture);
    }
    e = cudaStreamEndCapture(b->capture, &graph);
    if (rc) {
        if (graph) cudaGraphDestroy(graph);
        return rc;
    }
    if (!e) e = cudaGraphInstantiate(&b->exec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (e) {
        dsr__set_cuda_error(e, "dsr_gol_batch_step instantiate");
        b->exec = nullptr;
        return DSR_E_CUDA;
    }
    b->exec_epoch = b->group->epoch;
    return DSR_OK;
}

extern "C" int dsr_gol_batch_prepare(dsr_gol_batch* b) {
    if (!b) return DSR_E_INVALID;
    return ensure_gol_graph(b);
}

extern "C" int dsr_gol_batch_step(dsr_gol_batch* b, int n_gen, void* stream) {
    if (!b || n_gen < 0) return DSR_E_INVALID;
    const int rc = ensure_gol_graph(b);
    if (rc) return rc;
    cudaStream_t s = dsr__stream(stream);
    for (int i = 0; i < n_gen; ++i) {
        cudaError_t e = cudaGraphLaunch(b->exec, s);
        if (e) {
            dsr__set_cuda_error(e, "dsr_gol_batch_step launch");
            return DSR_E_CUDA;
        }
    }
    return DSR_OK;
}

extern "C" int dsr_gol_batch_heap(dsr_gol_batch* b, int inst, dsr_heap** out) {
    if (!b || !out || inst < 0 || inst >= (int)b->table_h.size() || !b->table_h[inst].cell_ref) return DSR_E_INVALID;
    *out = b->group->heaps[inst];
    return DSR_OK;
}

extern "C" int dsr_gol_batch_group(dsr_gol_batch* b, dsr_group** out) {
    if (!b || !out) return DSR_E_INVALID;
    *out = b->group;
    return DSR_OK;
}

extern "C" int dsr_gol_batch_destroy(dsr_gol_batch* b) {
    if (!b) return DSR_E_INVALID;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    cudaStreamDestroy(b->capture);
    if (b->table_pooled) dsr__group_give_bytes(b->group, b->table_d, gol_table_bytes((int)b->table_h.size()));
    dsr_group_destroy(b->group);
    delete b;
    return DSR_OK;
}
