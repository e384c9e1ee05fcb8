// Sugarscape as an SMMO program (Fig. 6f; Epstein and Axtell's movement rule
// M, growback rule G_alpha and replacement rule R): Agent objects on a
// W x H torus of sugar cells, four do-alls per step.
//
//   A1 choose:  the candidate cell with the most sugar among the agent's own
//               cell and the free cells up to `vision` away in the order N,
//               E, S, W; then the nearest; then (r >> 32) mod k with
//               r = rand(seed, 12, t, own cell). Another cell is claimed
//               (atomicMin of the own cell index).
//   A2 move:    the winner of a claim moves (and resets the claim); every
//               agent harvests its cell, pays its metabolism, ages, and is
//               marked dead when its sugar is below 0 or its age reached
//               max_age.
//   A3 claim:   a dead agent draws c = (rand(seed, 13, t, own) >> 32) mod
//               (W * H) and claims c if no agent occupies it.
//   A4 replace: a dead agent creates a new agent (age 0, attributes drawn
//               from streams 8..11 keyed on the new cell) at c if it won c,
//               else in its own cell, and deletes itself.
// Sugar grows back lazily: a cell keeps the step of its last harvest h, and
// its sugar at the start of step t is min(cap, alpha * (t - h)) (cap if
// never harvested), which equals applying G_alpha at the end of every step,
// without a pass over all cells. A cell is one 32-bit word: bit 31 set
// while an agent (alive or dead) is on it, bits 28-30 its capacity, bits
// 0-27 its last harvest step + 1 (0: never), so that the choice reads one
// word per cell in sight. Steps are limited to 2^28 - 2.
#include <climits>

#include "dsr_apps.h"
#include "dsr_steps.cuh"

namespace {
enum { AGENT = 0 };
enum { F_X, F_Y, F_SUGAR, F_METAB, F_VISION, F_AGE, F_MAXAGE, F_DEAD, NF };
enum { EV_MOVES, EV_STARVED, EV_AGED, EV_AWAY, EV_HARVEST, N_EV };
constexpr uint32_t NO_CLAIM = 0xFFFFFFFFu;
constexpr uint32_t OCC = 0x80000000u, CAP_SHIFT = 28, STEP_MASK = 0x0FFFFFFFu;

struct SugarWs {
    uint32_t* cell;      // [n] occupancy bit, capacity, last harvest step + 1
    uint32_t* claim;     // [n] A1 claims (lowest own cell wins), NO_CLAIM
    uint32_t* claim2;    // [n] A3 claims
    uint32_t* intent;    // [heap slots] A1 target of each agent slot
    dsr_u64 n_slots;
    dsr_u64* events;     // [DSR_CTR_SLOTS][N_EV] cumulative, one row per SM slot
};

enum { K_ENDOW, K_METAB, K_VISION, K_AGE, K_TIE, K_PLACE, N_KEYS };  // streams 8 .. 13

struct SugarArgs {
    SugarWs ws;
    dsr_sugarscape_params p;
    int32_t step;
    dsr_u64 key[N_KEYS];  // dsr_rand_key of this step's draws
};

__device__ __forceinline__ int32_t* fld(const dsr_dev_heap& H, dsr_ref r, int f) {
    return dsr_field<int32_t>(H, AGENT, r, f);
}

// Sugar of a cell word at the start of the step: min(cap, alpha * d) after d
// steps of growback; cap if never harvested. Capacities are below 8, so d and
// alpha count up to 8 only, and 32 bits hold their product.
__device__ __forceinline__ int32_t sugar_of(const SugarArgs& a, uint32_t st) {
    const int32_t cap = (int32_t)((st >> CAP_SHIFT) & 7u);
    const int32_t h1 = (int32_t)(st & STEP_MASK);
    const int32_t d = h1 ? min(a.step + 1 - h1, 8) : 8;
    return min(cap, min(a.p.alpha, 8) * d);
}

__device__ __forceinline__ int32_t draw(dsr_u64 key, int64_t c, int32_t lo, int32_t hi) {
    const uint32_t r = (uint32_t)(dsr_splitmix_at(key, (dsr_u64)c) >> 32);
    const uint32_t n = (uint32_t)hi - (uint32_t)lo + 1u;
    return (int32_t)((uint32_t)lo + (n < 0x80000000u ? r % n : r));
}

struct NoCtx {};
struct SugarMethod {
    typedef SugarArgs Args;
    typedef SugarArgs Inst;
    typedef NoCtx Ctx;
    typedef dsr_no_acc Acc;
    enum { kDefers = DSR_NOTHING, kMarks = 0 };
    static __device__ __forceinline__ const SugarArgs& inst(const SugarArgs& a, uint32_t) { return a; }
    static __device__ __forceinline__ NoCtx begin(const SugarArgs&) { return {}; }
    static __device__ __forceinline__ void flush(const dsr_dev_heap&, const SugarArgs&, dsr_no_acc) {}
};

// Add the sum over the calling warp (whole) to event k, on the row of the
// warp's SM (rows spread the atomics over many addresses).
__device__ __forceinline__ void flush_event(const SugarArgs& a, int k, unsigned v) {
    v = __reduce_add_sync(0xFFFFFFFFu, v);
    if (v && dsr_lane() == 0) {
        unsigned smid;
        asm("mov.u32 %0, %%smid;" : "=r"(smid));
        atomicAdd(a.ws.events + (smid % DSR_CTR_SLOTS) * N_EV + k, (dsr_u64)v);
    }
}

struct DChoose : SugarMethod {
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap& H, int, const SugarArgs& a, NoCtx, dsr_ref self,
                                                   dsr_later&, dsr_no_acc&) {
        const int32_t x = *fld(H, self, F_X), y = *fld(H, self, F_Y), vision = *fld(H, self, F_VISION);
        const int32_t W = a.p.W, Hh = a.p.H;
        const uint32_t own = (uint32_t)y * (uint32_t)W + (uint32_t)x, n = (uint32_t)W * (uint32_t)Hh;
        const uint32_t* cell = a.ws.cell;
        int32_t best = sugar_of(a, cell[own]), best_d = 0;
        unsigned dirs = 0;  // directions (bit 0 N, 1 E, 2 S, 3 W) of the candidates at distance best_d
        for (int32_t d = 1; d <= vision; ++d) {
            const uint32_t rows = (uint32_t)d * (uint32_t)W;
            const uint32_t cn = y < d ? own + (n - rows) : own - rows, cs = y + d >= Hh ? own - (n - rows) : own + rows;
            const uint32_t ce = x + d >= W ? own + (uint32_t)(d - W) : own + (uint32_t)d;
            const uint32_t cw = x < d ? own + (uint32_t)(W - d) : own - (uint32_t)d;
            const uint32_t st[4] = {cell[cn], cell[ce], cell[cs], cell[cw]};
            int32_t v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = (int32_t)st[k] < 0 ? -1 : sugar_of(a, st[k]);  // OCC is the sign bit
            const int32_t m = max(max(v[0], v[1]), max(v[2], v[3]));
            if (m > best) {
                best = m;
                best_d = d;
                dirs = (v[0] == m ? 1u : 0u) | (v[1] == m ? 2u : 0u) | (v[2] == m ? 4u : 0u) | (v[3] == m ? 8u : 0u);
            }
        }
        uint32_t t = own;
        if (best_d > 0) {
            const unsigned k = (unsigned)__popc(dirs);
            unsigned m = dirs, pick = 0;
            if (k > 1) pick = dsr_mod_upto4((uint32_t)(dsr_splitmix_at(a.key[K_TIE], own) >> 32), k);
            if (pick > 0) m &= m - 1;
            if (pick > 1) m &= m - 1;
            if (pick > 2) m &= m - 1;
            const int dir = __ffs(m) - 1;
            const int32_t d = best_d;
            const uint32_t rows = (uint32_t)d * (uint32_t)W;
            if (dir == 0) t = y < d ? own + (n - rows) : own - rows;
            if (dir == 1) t = x + d >= W ? own + (uint32_t)(d - W) : own + (uint32_t)d;
            if (dir == 2) t = y + d >= Hh ? own - (n - rows) : own + rows;
            if (dir == 3) t = x < d ? own + (uint32_t)(W - d) : own - (uint32_t)d;
        }
        if (dsr_check(self < a.ws.n_slots, H.err, H.dbg, 8, self)) a.ws.intent[self] = t;
        if (t != own) atomicMin(a.ws.claim + t, own);
        return 0;
    }
};

struct Events {
    unsigned moves, starved, aged, harvest;
};
// Returns 1 for an agent that dies: the list then holds the dead, for the
// two do-alls that replace them.
struct DMove : SugarMethod {
    typedef Events Acc;
    enum { kMarks = 1 };
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap& H, int, const SugarArgs& a, NoCtx, dsr_ref self,
                                                   dsr_later&, Events& ev) {
        if (!dsr_check(self < a.ws.n_slots, H.err, H.dbg, 8, self)) return 0;
        const int32_t x = *fld(H, self, F_X), y = *fld(H, self, F_Y);
        const uint32_t t = a.ws.intent[self];
        const uint32_t own = (uint32_t)y * (uint32_t)a.p.W + (uint32_t)x;
        uint32_t c = own;
        // the cells are read after the claim is known, and only by those who
        // write them: loading both cells of every agent together with its
        // claim made a step 26 us slower (1.68 M agents), as lines fetched for
        // a later store were gone from L1 by then
        if (t != own && a.ws.claim[t] == own) {
            a.ws.claim[t] = NO_CLAIM;  // only the winner matches, so the reset cannot make a loser win
            a.ws.cell[own] &= ~OCC;  // this agent is the only writer of both cells in this do-all
            a.ws.cell[t] |= OCC;
            *fld(H, self, F_X) = (int32_t)(t % (uint32_t)a.p.W);
            *fld(H, self, F_Y) = (int32_t)(t / (uint32_t)a.p.W);
            c = t;
            ++ev.moves;
        }
        const uint32_t st = a.ws.cell[c];
        const int32_t sugar0 = *fld(H, self, F_SUGAR), metab = *fld(H, self, F_METAB);
        const int32_t age = *fld(H, self, F_AGE) + 1, max_age = *fld(H, self, F_MAXAGE);
        const int32_t got = sugar_of(a, st);
        a.ws.cell[c] = (st & ~STEP_MASK) | (uint32_t)(a.step + 1);
        const int32_t sugar = sugar0 + got - metab;
        *fld(H, self, F_SUGAR) = sugar;
        *fld(H, self, F_AGE) = age;
        const unsigned starved = sugar < 0, aged = !starved && age >= max_age;
        if (starved || aged) *fld(H, self, F_DEAD) = 1;
        ev.starved += starved;
        ev.aged += aged;
        ev.harvest += (unsigned)got;
        return starved | aged;
    }
    static __device__ __forceinline__ void flush(const dsr_dev_heap&, const SugarArgs& a, const Events& ev) {
        flush_event(a, EV_MOVES, ev.moves);
        flush_event(a, EV_STARVED, ev.starved);
        flush_event(a, EV_AGED, ev.aged);
        flush_event(a, EV_HARVEST, ev.harvest);
    }
};

__device__ __forceinline__ uint32_t replacement_cell(const SugarArgs& a, uint32_t own) {
    return (uint32_t)(dsr_splitmix_at(a.key[K_PLACE], own) >> 32) % ((uint32_t)a.p.W * (uint32_t)a.p.H);
}

// A few agents in a hundred die in a step, one or two of a warp's 32: the
// dead of a CTA are gathered first and handled by full warps.
struct DReplaceClaim : SugarMethod {
    enum { kDefers = DSR_WORK };
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap&, int, const SugarArgs&, NoCtx, dsr_ref self,
                                                   dsr_later& later, dsr_no_acc&) {
        later.push(self);
        return 0;
    }
    static __device__ __forceinline__ void later(const dsr_dev_heap& H, const SugarArgs& a, NoCtx, dsr_u64 self,
                                                 dsr_no_acc&) {
        const uint32_t own = (uint32_t)*fld(H, self, F_Y) * (uint32_t)a.p.W + (uint32_t)*fld(H, self, F_X);
        const uint32_t c = replacement_cell(a, own);
        if (!(a.ws.cell[c] & OCC)) atomicMin(a.ws.claim2 + c, own);
    }
};

struct DReplace : SugarMethod {
    typedef unsigned Acc;  // replacements placed away from the dead agent's cell
    enum { kDefers = DSR_WORK };
    static __device__ __forceinline__ unsigned run(const dsr_dev_heap&, int, const SugarArgs&, NoCtx, dsr_ref self,
                                                   dsr_later& later, unsigned&) {
        later.push(self);
        return 0;
    }
    static __device__ __forceinline__ void later(const dsr_dev_heap& H, const SugarArgs& a, NoCtx, dsr_u64 self,
                                                 unsigned& away) {
        const uint32_t own = (uint32_t)*fld(H, self, F_Y) * (uint32_t)a.p.W + (uint32_t)*fld(H, self, F_X);
        const uint32_t c = replacement_cell(a, own);
        uint32_t at = own;
        if (a.ws.claim2[c] == own) {
            a.ws.claim2[c] = NO_CLAIM;
            a.ws.cell[own] &= ~OCC;
            a.ws.cell[c] |= OCC;
            at = c;
            ++away;
        }
        dsr_delete(H, self);  // first, so that the new agent may take the slot
        const dsr_ref r = dsr_new(H, AGENT, self);  // tried first: the block just given a free slot
        if (r == DSR_NULL) return;  // out of memory: DSR_ERR_OOM is set
        *fld(H, r, F_X) = (int32_t)(at % (uint32_t)a.p.W);
        *fld(H, r, F_Y) = (int32_t)(at / (uint32_t)a.p.W);
        *fld(H, r, F_SUGAR) = draw(a.key[K_ENDOW], at, a.p.endow_lo, a.p.endow_hi);
        *fld(H, r, F_METAB) = draw(a.key[K_METAB], at, a.p.metab_lo, a.p.metab_hi);
        *fld(H, r, F_VISION) = draw(a.key[K_VISION], at, a.p.vision_lo, a.p.vision_hi);
        *fld(H, r, F_AGE) = 0;
        *fld(H, r, F_MAXAGE) = draw(a.key[K_AGE], at, a.p.age_lo, a.p.age_hi);
        *fld(H, r, F_DEAD) = 0;
    }
    static __device__ __forceinline__ void flush(const dsr_dev_heap&, const SugarArgs& a, unsigned away) {
        flush_event(a, EV_AWAY, away);
    }
};
constexpr dsr_phase kAgents{AGENT, 0};

// One thread per initial agent (agents0[i] = x, y, sugar, metabolism,
// vision, age, max_age; distinct cells).
__global__ void __launch_bounds__(DSR_BULK_THREADS)
    k_sugar_init(const __grid_constant__ dsr_dev_heap H, const int32_t* agents0, int64_t n_agents, SugarWs ws,
                 int32_t W, int rows) {
    __shared__ dsr_bulk_smem<1> sm;
    const int types[1] = {AGENT};
    dsr_bulk_create(
        H, (dsr_u64)n_agents, rows, types, sm, [](dsr_u64) { return 1u; },
        [&](dsr_u64 i, unsigned, const dsr_ref (&ref)[1]) {
            const dsr_ref r = ref[0];
            if (r == DSR_NULL) return;
            const int32_t* src = agents0 + 7 * i;
            for (int f = 0; f < 7; ++f) *fld(H, r, f) = src[f];
            *fld(H, r, F_DEAD) = 0;
            ws.cell[(int64_t)src[1] * W + src[0]] |= OCC;
        });
}

// Cells from the capacities: unoccupied, never harvested. Four cells a thread
// and round: 16-byte stores.
__global__ void __launch_bounds__(256) k_sugar_fill(uint32_t* cell, const uint8_t* cap, int64_t n) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool words = (reinterpret_cast<uintptr_t>(cap) & 3) == 0;
    const int64_t n4 = words ? n / 4 : 0;
    for (int64_t i = tid; i < n4; i += stride) {
        const uchar4 c = reinterpret_cast<const uchar4*>(cap)[i];
        reinterpret_cast<uint4*>(cell)[i] = make_uint4((c.x & 7u) << CAP_SHIFT, (c.y & 7u) << CAP_SHIFT,
                                                       (c.z & 7u) << CAP_SHIFT, (c.w & 7u) << CAP_SHIFT);
    }
    for (int64_t i = 4 * n4 + tid; i < n; i += stride) cell[i] = (uint32_t)(cap[i] & 7u) << CAP_SHIFT;
}

__global__ void __launch_bounds__(256) k_sugar_read(const __grid_constant__ SugarArgs a, int32_t* out) {
    const int64_t n = (int64_t)a.p.W * a.p.H;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool words = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    const int64_t n4 = words ? n / 4 : 0;
    for (int64_t i = tid; i < n4; i += stride) {
        const uint4 c = reinterpret_cast<const uint4*>(a.ws.cell)[i];
        reinterpret_cast<int4*>(out)[i] = make_int4(sugar_of(a, c.x), sugar_of(a, c.y), sugar_of(a, c.z), sugar_of(a, c.w));
    }
    for (int64_t i = 4 * n4 + tid; i < n; i += stride) out[i] = sugar_of(a, a.ws.cell[i]);
}

const int kAgentFields[NF] = {4, 4, 4, 4, 4, 4, 4, 4};

bool heap_matches(const dsr_heap* h) {
    const dsr_layout& L = h->layout;
    if (L.n_types < 1 || L.n_fields[AGENT] != NF) return false;
    for (int f = 0; f < NF; ++f)
        if (L.field_bytes[AGENT][f] != 4) return false;
    return true;
}

bool params_ok(const dsr_sugarscape_params* p) {
    return p && p->alpha >= 1 && p->vision_lo >= 1 && p->vision_hi >= p->vision_lo && p->vision_hi <= 64 &&
           p->W >= 2 * p->vision_hi + 1 && p->H >= 2 * p->vision_hi + 1 && (int64_t)p->W * p->H < (1ll << 31) &&
           p->metab_hi >= p->metab_lo && p->endow_hi >= p->endow_lo && p->age_lo >= 1 && p->age_hi >= p->age_lo;
}

size_t r256(size_t x) { return (x + 255) / 256 * 256; }

size_t ws_bytes(const dsr_sugarscape_params& p, dsr_u64 slots) {
    const size_t n = (size_t)p.W * p.H;
    return 3 * r256(n * 4) + r256(slots * 4) + r256(DSR_CTR_SLOTS * N_EV * 8);
}

SugarWs carve(void* base, const dsr_sugarscape_params& p, dsr_u64 slots) {
    const size_t n = (size_t)p.W * p.H;
    uint8_t* q = static_cast<uint8_t*>(base);
    SugarWs w;
    w.cell = reinterpret_cast<uint32_t*>(q);
    q += r256(n * 4);
    w.claim = reinterpret_cast<uint32_t*>(q);
    q += r256(n * 4);
    w.claim2 = reinterpret_cast<uint32_t*>(q);
    q += r256(n * 4);
    w.intent = reinterpret_cast<uint32_t*>(q);
    q += r256(slots * 4);
    w.events = reinterpret_cast<dsr_u64*>(q);
    w.n_slots = slots;
    return w;
}
}  // namespace

struct dsr_sugarscape {
    dsr_heap* heap;
    SugarArgs args;
};

extern "C" int dsr_sugarscape_types(dsr_type_desc* out) {
    if (!out) return DSR_E_INVALID;
    out[0] = dsr_type_desc{"Agent", NF, kAgentFields};
    return DSR_OK;
}

extern "C" int dsr_sugarscape_workspace_bytes(const dsr_heap* heap, const dsr_sugarscape_params* p, size_t* out) {
    if (!heap || !out || !params_ok(p)) return DSR_E_INVALID;
    *out = ws_bytes(*p, heap->layout.n_blocks * 64);
    return DSR_OK;
}

extern "C" int dsr_sugarscape_create(dsr_heap* heap, const dsr_sugarscape_params* p, const void* cap_dev,
                                     const void* agents0_dev, int64_t n_agents, void* workspace_dev, void* stream,
                                     dsr_sugarscape** out) {
    if (!heap || !cap_dev || (n_agents && !agents0_dev) || n_agents < 0 || !workspace_dev || !out || !params_ok(p) ||
        !heap_matches(heap))
        return DSR_E_INVALID;
    if (reinterpret_cast<uintptr_t>(workspace_dev) & 255) return DSR_E_INVALID;
    cudaStream_t s = dsr__stream(stream);
    const dsr_u64 slots = heap->layout.n_blocks * 64;
    const int64_t n = (int64_t)p->W * p->H;
    dsr_sugarscape* g = new dsr_sugarscape;
    g->heap = heap;
    g->args.ws = carve(workspace_dev, *p, slots);
    g->args.p = *p;
    g->args.step = 0;
    SugarWs& w = g->args.ws;
    cudaError_t e = cudaMemsetAsync(w.claim, 0xFF, (size_t)n * 4, s);
    if (!e) e = cudaMemsetAsync(w.claim2, 0xFF, (size_t)n * 4, s);
    if (!e) e = cudaMemsetAsync(w.events, 0, DSR_CTR_SLOTS * N_EV * 8, s);
    if (e) {
        dsr__set_cuda_error(e, "dsr_sugarscape_create");
        delete g;
        return DSR_E_CUDA;
    }
    const int ctas = heap->sm_count * 8;
    k_sugar_fill<<<ctas, 256, 0, s>>>(w.cell, static_cast<const uint8_t*>(cap_dev), n);
    if (n_agents) {
        const int rows = dsr__bulk_rows<1>((dsr_u64)n_agents, heap->sm_count);
        k_sugar_init<<<dsr__bulk_grid((dsr_u64)n_agents, rows, heap->sm_count), DSR_BULK_THREADS, 0, s>>>(
            heap->dev, static_cast<const int32_t*>(agents0_dev), n_agents, w, p->W, rows);
    }
    const int rc = dsr__check_launch("k_sugar_init");
    if (rc) {
        delete g;
        return rc;
    }
    *out = g;
    return DSR_OK;
}

extern "C" int dsr_sugarscape_step(dsr_sugarscape* g, int n_steps, void* stream) {
    if (!g || n_steps < 0 || (int64_t)g->args.step + n_steps > (int64_t)STEP_MASK - 1) return DSR_E_INVALID;
    cudaStream_t s = dsr__stream(stream);
    for (int i = 0; i < n_steps; ++i) {
        // One scan lists the agents for A1 and A2; A2 leaves the dead in the
        // list for A3 and A4. (All four count as visits of every agent.)
        SugarArgs& a = g->args;
        for (int k = 0; k < N_KEYS; ++k) a.key[k] = dsr_rand_key(a.p.seed, 8 + k, (dsr_u64)a.step);
        if (dsr__has_subtypes(g->heap, AGENT))
            dsr__list_tree(g->heap, AGENT, 4, s);
        else
            dsr__list_types(g->heap, AGENT, -1, 4, 0, s);
        int rc = dsr__step<DChoose>(g->heap, kAgents, kAgents, a, s);
        if (!rc) rc = dsr__step<DMove>(g->heap, kAgents, kAgents, a, s);
        if (!rc) rc = dsr__step<DReplaceClaim>(g->heap, kAgents, kAgents, a, s);
        if (!rc) rc = dsr__step<DReplace, dsr_no_method, true>(g->heap, kAgents, kAgents, a, s);
        if (rc) return rc;
        g->args.step += 1;
    }
    return DSR_OK;
}

extern "C" int dsr_sugarscape_events(dsr_sugarscape* g, void* stream, uint64_t* out) {
    if (!g || !out) return DSR_E_INVALID;
    cudaStream_t s = dsr__stream(stream);
    static thread_local dsr_u64 rows[DSR_CTR_SLOTS * N_EV];
    cudaError_t e = cudaMemcpyAsync(rows, g->args.ws.events, sizeof rows, cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (e) {
        dsr__set_cuda_error(e, "dsr_sugarscape_events");
        return DSR_E_CUDA;
    }
    for (int k = 0; k < N_EV; ++k) {
        out[k] = 0;
        for (int r = 0; r < DSR_CTR_SLOTS; ++r) out[k] += rows[r * N_EV + k];
    }
    return DSR_OK;
}

extern "C" int dsr_sugarscape_sugar(dsr_sugarscape* g, void* out_dev, void* stream) {
    if (!g || !out_dev) return DSR_E_INVALID;
    k_sugar_read<<<g->heap->sm_count * 8, 256, 0, dsr__stream(stream)>>>(g->args, static_cast<int32_t*>(out_dev));
    return dsr__check_launch("k_sugar_read");
}

extern "C" int dsr_sugarscape_destroy(dsr_sugarscape* g) {
    delete g;
    return DSR_OK;
}
