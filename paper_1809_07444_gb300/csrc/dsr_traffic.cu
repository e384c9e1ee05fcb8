// Traffic as an SMMO program (Fig. 6g, the Nagel-Schreckenberg model): R
// single-lane roads of L cells; Car objects move by the model's four rules in
// one do-all per step, Source objects (open roads) admit new cars in a second.
//
// Rules (parallel update; occupancy read at the start of the step):
//   do-all Car:    v1 = min(v + 1, vmax); g = free cells ahead, looking at
//                  most v1 cells ahead (open road: cells past the end are
//                  free; periodic road: wraps); v2 = min(v1, g); with
//                  probability p (draw rand(seed, 5, t, road * L + x))
//                  v3 = max(v2 - 1, 0), else v2; x' = x + v3; an open-road
//                  car with x' >= L leaves (delete this).
//   do-all Source: if cell 0 is free after the cars moved and the draw
//                  rand(seed, 6, t, road) is below alpha, new Car(road, 0,
//                  v_entry); otherwise count an entry blocked by a car.
// Occupancy lives in two byte grids: a step reads `cur` and marks the new
// positions in `next`, which must start empty. A car only moves into free
// cells ahead of it, before the next car, so no two cars mark one cell and
// no car reads a cell another car writes: the do-all needs no atomics. After
// the step `cur` is cleared and the grids swap.
#include "dsr_apps.h"
#include "dsr_steps.cuh"

namespace {
enum { CAR = 0, SOURCE = 1 };
enum { F_ROAD = 0, F_X = 1, F_V = 2 };             // Car
enum { S_ROAD = 0, S_ENTERED = 1, S_BLOCKED = 2 };  // Source
enum { CTR_ENTERED = DSR_CTR_APP0, CTR_LEFT, CTR_MOVED, CTR_VSUM };

struct TrafficArgs {
    uint8_t* cur;   // [R * L] occupancy at the start of the step
    uint8_t* next;  // [R * L] occupancy after the step (zero on entry)
    dsr_traffic_params p;
    dsr_u64 slow_key, enter_key;  // dsr_rand_key of this step's draws (streams 5 and 6)
};

__device__ __forceinline__ int32_t* fld(const dsr_dev_heap& H, int T, dsr_ref r, int f) {
    return dsr_field<int32_t>(H, T, r, f);
}

__device__ __forceinline__ bool draws_below(dsr_u64 r, dsr_u64 thr) { return (r >> 32) < thr; }

// Free cells among the n cells from `cell` on, before the first car: eight
// cells a load. The grid is an array of 8-byte words (its length is a
// multiple of 256), so the words that hold any of these cells are inside it;
// cells read beyond the n are masked out.
__device__ __forceinline__ int32_t free_run(const uint8_t* grid, dsr_u64 cell, int32_t n) {
    int32_t g = 0;
    while (g < n) {
        const dsr_u64 at = cell + (uint32_t)g;
        const dsr_u64* w = reinterpret_cast<const dsr_u64*>(grid) + (at >> 3);
        const unsigned off = (unsigned)at & 7u;
        int32_t k = n - g < 8 ? n - g : 8;
        dsr_u64 v = w[0] >> (8 * off);
        if (off + (unsigned)k > 8u) v |= w[1] << (64 - 8 * off);
        if (k < 8) v &= (1ull << (8 * k)) - 1;
        if (v) return g + ((__ffsll((long long)v) - 1) >> 3);
        g += k;
    }
    return n;
}

struct NoCtx {};
struct TrafficMethod {
    typedef TrafficArgs Args;
    typedef TrafficArgs Inst;
    typedef NoCtx Ctx;
    enum { kDefers = DSR_NOTHING, kMarks = 0 };
    static __device__ __forceinline__ const TrafficArgs& inst(const TrafficArgs& a, uint32_t) { return a; }
    static __device__ __forceinline__ NoCtx begin(const TrafficArgs&) { return {}; }
};

struct Flow {
    unsigned moved, vsum;
};
struct DCar : TrafficMethod {
    typedef Flow Acc;
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap& H, int, const TrafficArgs& a, NoCtx,
                                                   dsr_ref self, dsr_later&, Flow& flow) {
        const int32_t road = *fld(H, CAR, self, F_ROAD), x = *fld(H, CAR, self, F_X), v = *fld(H, CAR, self, F_V);
        const int32_t L = a.p.L;
        const dsr_u64 row = (dsr_u64)(uint32_t)road * (uint32_t)L;
        const int32_t v1 = v + 1 < a.p.vmax ? v + 1 : a.p.vmax;
        // cells past the end of an open road are free; a periodic road wraps
        const int32_t ahead = L - 1 - x < v1 ? L - 1 - x : v1;
        int32_t g = free_run(a.cur, row + (uint32_t)x + 1, ahead);
        if (g == ahead && ahead < v1) g = a.p.periodic ? ahead + free_run(a.cur, row, v1 - ahead) : v1;
        int32_t v3 = g;
        if (draws_below(dsr_splitmix_at(a.slow_key, row + (uint32_t)x), a.p.p_thr)) v3 = v3 > 0 ? v3 - 1 : 0;
        flow.moved += v3 > 0;
        flow.vsum += (unsigned)v3;
        int32_t nx = x + v3;
        if (nx >= L) {
            if (!a.p.periodic) {
                dsr_count_lanes(H.ctr, CTR_LEFT);
                dsr_delete(H, self);
                return 0;
            }
            nx -= L;
        }
        a.next[row + (uint32_t)nx] = 1;
        *fld(H, CAR, self, F_X) = nx;
        *fld(H, CAR, self, F_V) = v3;
        return 0;
    }
    static __device__ __forceinline__ void flush(const dsr_dev_heap& H, const TrafficArgs&, const Flow& f) {
        dsr_flush_count(H, CTR_MOVED, f.moved);
        dsr_flush_count(H, CTR_VSUM, f.vsum);
    }
};

// An entering car is created with the others of its CTA.
struct DSource : TrafficMethod {
    typedef dsr_no_acc Acc;
    enum { kDefers = CAR, kDeferBack = 0 };
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap& H, int, const TrafficArgs& a, NoCtx,
                                                   dsr_ref self, dsr_later& later, dsr_no_acc&) {
        const int32_t road = *fld(H, SOURCE, self, S_ROAD);
        if (a.next[(dsr_u64)(uint32_t)road * (uint32_t)a.p.L]) {
            *fld(H, SOURCE, self, S_BLOCKED) += 1;
            return 0;
        }
        if (draws_below(dsr_splitmix_at(a.enter_key, (dsr_u64)road), a.p.a_thr)) later.push(self);
        return 0;
    }
    static __device__ __forceinline__ void born(const dsr_dev_heap& H, const TrafficArgs& a, dsr_u64 self, dsr_ref c) {
        if (c == DSR_NULL) return;  // out of memory: DSR_ERR_OOM is set
        const int32_t road = *fld(H, SOURCE, self, S_ROAD);
        *fld(H, CAR, c, F_ROAD) = road;
        *fld(H, CAR, c, F_X) = 0;
        *fld(H, CAR, c, F_V) = a.p.v_entry;
        a.next[(dsr_u64)(uint32_t)road * (uint32_t)a.p.L] = 1;
        *fld(H, SOURCE, self, S_ENTERED) += 1;
        dsr_count_lanes(H.ctr, CTR_ENTERED);
    }
    static __device__ __forceinline__ void flush(const dsr_dev_heap&, const TrafficArgs&, dsr_no_acc) {}
};

constexpr dsr_phase kCars{CAR, 0};

// The Source do-all of an open road's step, with the clearing of the old
// occupancy, which nothing reads any more: the few CTAs that have sources
// wait on their chains of accesses while the others write the grid.
template <int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 5 : 1)
    k_traffic_sources_step(const __grid_constant__ dsr_dev_heap H, const __grid_constant__ dsr_phase sources,
                           const __grid_constant__ TrafficArgs a) {
    __shared__ dsr_later_smem<MAXT> later;
    dsr_run_list<DSource, dsr_heap_space, MAXT>(dsr_heap_space{H}, sources, a, H.span_sh[SOURCE] - 5, false, &later);
    uint4* w = reinterpret_cast<uint4*>(a.cur);
    const dsr_u64 n = ((dsr_u64)a.p.R * a.p.L + 255) / 256 * 16;
    for (dsr_u64 i = (dsr_u64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (dsr_u64)gridDim.x * blockDim.x)
        w[i] = make_uint4(0, 0, 0, 0);
    if (blockIdx.x == 0 && threadIdx.x == 0) dsr_end_step(H.R_count);
}

// With the heap's tuning, as the do-alls.
int launch_sources(const dsr_heap* h, const dsr_phase& sources, const TrafficArgs& a, cudaStream_t s) {
    static dsr_grid_cache cache;
    const int threads = h->tune.threads;
    const bool small = threads <= 256;
    const int grid = dsr__tuned_grid(
        h, small ? (const void*)k_traffic_sources_step<256> : (const void*)k_traffic_sources_step<1024>, cache);
    if (small)
        k_traffic_sources_step<256><<<grid, threads, 0, s>>>(h->dev, sources, a);
    else
        k_traffic_sources_step<1024><<<grid, threads, 0, s>>>(h->dev, sources, a);
    return dsr__check_launch("k_traffic_sources_step");
}

// A Car for every cell where v0 >= 0.
__global__ void __launch_bounds__(DSR_BULK_THREADS)
    k_traffic_init(const __grid_constant__ dsr_dev_heap H, const int8_t* v0, uint8_t* cur, dsr_traffic_params p,
                   int rows) {
    __shared__ dsr_bulk_smem<1, true> sm;
    const int types[1] = {CAR};
    const dsr_u64 n = (dsr_u64)p.R * p.L;
    const bool small = n <= 0xFFFFFFFFull;  // 32-bit divisions are several times cheaper than 64-bit ones
    dsr_bulk_create(
        H, n, rows, types, sm, [&](dsr_u64 i) { return v0[i] >= 0 ? 1u : 0u; },
        [&](dsr_u64 i, unsigned, const dsr_ref (&ref)[1]) {
            const dsr_ref c = ref[0];
            if (c == DSR_NULL) return;
            const int v = v0[i];
            const int32_t road = small ? (int32_t)((uint32_t)i / (uint32_t)p.L) : (int32_t)(i / p.L);
            *fld(H, CAR, c, F_ROAD) = road;
            *fld(H, CAR, c, F_X) = (int32_t)(i - (dsr_u64)road * p.L);
            *fld(H, CAR, c, F_V) = v < p.vmax ? v : p.vmax;
            cur[i] = 1;
        });
}

// Open roads: one thread per road, its Source.
__global__ void __launch_bounds__(DSR_BULK_THREADS)
    k_traffic_sources(const __grid_constant__ dsr_dev_heap H, int32_t R, int rows) {
    __shared__ dsr_bulk_smem<1> sm;
    const int types[1] = {SOURCE};
    dsr_bulk_create(
        H, (dsr_u64)R, rows, types, sm, [](dsr_u64) { return 1u; },
        [&](dsr_u64 i, unsigned, const dsr_ref (&ref)[1]) {
            const dsr_ref s = ref[0];
            if (s == DSR_NULL) return;
            *fld(H, SOURCE, s, S_ROAD) = (int32_t)i;
            *fld(H, SOURCE, s, S_ENTERED) = 0;
            *fld(H, SOURCE, s, S_BLOCKED) = 0;
        });
}

const int kCarFields[3] = {4, 4, 4};
const int kSourceFields[3] = {4, 4, 4};

bool heap_matches(const dsr_heap* h) {
    const dsr_layout& L = h->layout;
    if (L.n_types < 2 || L.n_fields[CAR] != 3 || L.n_fields[SOURCE] != 3) return false;
    for (int t = 0; t < 2; ++t)
        for (int f = 0; f < 3; ++f)
            if (L.field_bytes[t][f] != 4) return false;
    return true;
}

bool params_ok(const dsr_traffic_params* p) {
    return p && p->R >= 1 && p->vmax >= 1 && p->vmax <= 127 && p->L > p->vmax && p->v_entry >= 0 &&
           p->v_entry <= p->vmax && (int64_t)p->R * p->L <= (1ll << 40) && p->p_thr <= (1ull << 32) &&
           p->a_thr <= (1ull << 32);
}

size_t grid_bytes(const dsr_traffic_params& p) { return ((size_t)p.R * p.L + 255) / 256 * 256; }
}  // namespace

struct dsr_traffic {
    dsr_heap* heap;
    dsr_traffic_params p;
    uint8_t* grid[2];
    int cur;         // index of the grid holding the current occupancy
    dsr_u64 step;    // steps taken
};

extern "C" int dsr_traffic_types(dsr_type_desc* out) {
    if (!out) return DSR_E_INVALID;
    out[0] = dsr_type_desc{"Car", 3, kCarFields};
    out[1] = dsr_type_desc{"Source", 3, kSourceFields};
    return DSR_OK;
}

extern "C" int dsr_traffic_workspace_bytes(const dsr_traffic_params* p, size_t* out) {
    if (!out || !params_ok(p)) return DSR_E_INVALID;
    *out = 2 * grid_bytes(*p);
    return DSR_OK;
}

extern "C" int dsr_traffic_create(dsr_heap* heap, const dsr_traffic_params* p, const void* v0_dev,
                                  void* workspace_dev, void* stream, dsr_traffic** out) {
    if (!heap || !v0_dev || !workspace_dev || !out || !params_ok(p) || !heap_matches(heap)) return DSR_E_INVALID;
    if (reinterpret_cast<uintptr_t>(workspace_dev) & 255) return DSR_E_INVALID;
    cudaStream_t s = dsr__stream(stream);
    dsr_traffic* t = new dsr_traffic;
    t->heap = heap;
    t->p = *p;
    t->grid[0] = static_cast<uint8_t*>(workspace_dev);
    t->grid[1] = t->grid[0] + grid_bytes(*p);
    t->cur = 0;
    t->step = 0;
    cudaError_t e = cudaMemsetAsync(workspace_dev, 0, 2 * grid_bytes(*p), s);
    if (e) {
        dsr__set_cuda_error(e, "dsr_traffic_create");
        delete t;
        return DSR_E_CUDA;
    }
    const dsr_u64 n = (dsr_u64)p->R * p->L;
    // the sources first: their few blocks are then taken before the cars', which
    // fill whatever is left (after the cars a heap with few blocks to spare,
    // all of them partly filled with cars, had none left for the sources)
    if (!p->periodic) {
        const int srows = dsr__bulk_rows<1>((dsr_u64)p->R, heap->sm_count);
        k_traffic_sources<<<dsr__bulk_grid((dsr_u64)p->R, srows, heap->sm_count), DSR_BULK_THREADS, 0, s>>>(
            heap->dev, p->R, srows);
    }
    const int rows = dsr__bulk_rows<1>(n, heap->sm_count);
    k_traffic_init<<<dsr__bulk_grid(n, rows, heap->sm_count), DSR_BULK_THREADS, 0, s>>>(
        heap->dev, static_cast<const int8_t*>(v0_dev), t->grid[0], *p, rows);
    int rc = dsr__check_launch("k_traffic_init");
    if (rc) {
        delete t;
        return rc;
    }
    *out = t;
    return DSR_OK;
}

extern "C" int dsr_traffic_step(dsr_traffic* t, int n_steps, void* stream) {
    if (!t || n_steps < 0) return DSR_E_INVALID;
    cudaStream_t s = dsr__stream(stream);
    for (int i = 0; i < n_steps; ++i) {
        TrafficArgs a{t->grid[t->cur], t->grid[1 - t->cur], t->p, dsr_rand_key(t->p.seed, 5, t->step),
                      dsr_rand_key(t->p.seed, 6, t->step)};
        const bool open = !t->p.periodic;
        const bool trees = dsr__has_subtypes(t->heap, CAR) || dsr__has_subtypes(t->heap, SOURCE);
        if (trees)
            dsr__list_tree(t->heap, CAR, 1, s);
        else
            dsr__list_types(t->heap, CAR, open ? SOURCE : -1, 1, 1, s);
        int rc = open && !trees ? dsr__step<DCar>(t->heap, kCars, kCars, a, s)
                                : dsr__step<DCar, dsr_no_method, true>(t->heap, kCars, kCars, a, s);
        if (rc) return rc;
        if (open && trees) dsr__list_tree(t->heap, SOURCE, 1, s);
        if (open) {
            rc = launch_sources(t->heap, dsr_phase{SOURCE, trees ? 0 : 1}, a, s);
            if (rc) return rc;
        } else {
            cudaError_t e = cudaMemsetAsync(t->grid[t->cur], 0, grid_bytes(t->p), s);  // the next step's `next`
            if (e) {
                dsr__set_cuda_error(e, "dsr_traffic_step");
                return DSR_E_CUDA;
            }
        }
        t->cur = 1 - t->cur;
        t->step += 1;
    }
    return DSR_OK;
}

extern "C" int dsr_traffic_occupancy(const dsr_traffic* t, const void** grid_dev) {
    if (!t || !grid_dev) return DSR_E_INVALID;
    *grid_dev = t->grid[t->cur];
    return DSR_OK;
}

extern "C" int dsr_traffic_destroy(dsr_traffic* t) {
    delete t;
    return DSR_OK;
}
