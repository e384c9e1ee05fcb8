// The do-alls of the applications' steps.
//
// dsr_parallel_do lists the allocated blocks of one type in one kernel and
// runs one method over the list in a second. A step of an application is a
// fixed sequence of do-alls over two types, and it knows which of them leave
// the live set of a type alone. So a step lists both types in one scan (type
// A's blocks from the front of H.R_bid / H.R_mask, type B's from the back:
// together at most M entries), and every do-all of the step runs over those
// lists. A method that deletes objects replaces its entry's mask by the
// survivors (kMarks) where a later do-all of the step visits them. Two
// do-alls that do not depend on each other share a launch.
//
// A warp takes every W-th (block, 32 slots) item. Its 32 lanes load the
// entries of its next 32 items at once and hand them out by shuffle, so the
// list costs one round trip per 32 items and warp, not one per item.
//
// Deferred work. A method may put off an object's creation: it pushes a
// word, and the CTA later creates all pending objects together and calls
// M::born for each. Births come from the few lanes of a warp whose object
// breeds; together they are whole blocks' worth, which are claimed many at a
// time and born full (dsr_claim_full). That is done while few blocks of the
// type have free slots; else births fill the holes at once through dsr_new,
// lane group by lane group, as in any other method, so that fragmentation
// stays as it is there. "Few": less than one block in DSR_BULK_HOLES, by a
// sample of 32 leaf words of active[T] and allocated[T] when the do-all
// starts. Work that few objects have (a dead agent's replacement) can be
// deferred in the same way without a creation: full warps then do it.
//
// A method is a type with
//   Args; Inst; Ctx; Acc
//   static Inst inst(const Args&, uint32_t heap)         the instance of a heap
//   static Ctx begin(const Inst&)                        once per do-all (plain) or item (group)
//   static unsigned run(H, T, const Inst&, const Ctx&, dsr_ref self, dsr_later&, Acc&)
//   kDefers: DSR_NOTHING, DSR_WORK (M::later(H, I, ctx, word, acc) for each
//     pushed word) or the type created (M::born(H, I, ctx, word, ref, acc))
//   kMarks: 1 if run's result (0 or 1) replaces the slot's bit of the list entry
//   static void flush(H, const Inst&, const Acc&)        by every whole warp at
//     the end: event counts gathered in Acc go to memory
#pragma once

#include <type_traits>

#include "dsr_bulk.cuh"
#include "dsr_group.cuh"

#ifndef DSR_BULK_HOLES
#define DSR_BULK_HOLES 8
#endif
constexpr int DSR_PENDING = 2048;  // deferred words of a CTA at a time
constexpr int DSR_LIST_BACK = 2;   // R_count[2] counts the entries at the back of the list

enum { DSR_NOTHING = -1, DSR_WORK = -2 };
struct dsr_no_acc {};
struct dsr_no_method {};

// The list a do-all runs over: type T's entries, at the front or the back.
struct dsr_phase {
    int type;
    int back;
};

struct dsr_later_smem {
    dsr_u64 pending[DSR_PENDING];
    uint32_t block[DSR_PENDING / 16];
    uint32_t np, nb;
    int few;
};

// push() may be called by any lanes of a warp.
struct dsr_later {
    dsr_later_smem* sm;
    bool on;  // creations are deferred
    __device__ __forceinline__ void push(dsr_u64 word) {
        const unsigned act = __activemask();
        const unsigned lane = dsr_lane();
        const int leader = __ffs(act) - 1;
        uint32_t at = 0;
        if ((int)lane == leader) at = atomicAdd(&sm->np, (uint32_t)__popc(act));
        at = __shfl_sync(act, at, leader);
        sm->pending[at + __popc(act & ((1u << lane) - 1))] = word;
    }
};

// Whether fewer than one in DSR_BULK_HOLES of the allocated blocks of T has a
// free slot, by a sample. Called by a whole warp.
__device__ __forceinline__ bool dsr_few_holes(const dsr_dev_heap& H, int T, unsigned hint) {
    const uint32_t at = __umulhi(dsr_hash32(hint + dsr_lane() * 0x9E3779B9u), H.active_bm[T].nwords[0]);
    const unsigned active = __popcll(dsr_ld_relaxed(H.active_bm[T].lvl[0] + at));
    const unsigned alloc = __popcll(dsr_ld_relaxed(H.alloc_bm[T].lvl[0] + at));
    return DSR_BULK_HOLES * __reduce_add_sync(0xFFFFFFFFu, active) <= __reduce_add_sync(0xFFFFFFFFu, alloc);
}

// The deferred work of a CTA. Called by the whole CTA, after a barrier.
template <class M>
__device__ __forceinline__ void dsr_do_pending(const dsr_dev_heap& H, const typename M::Inst& I,
                                               const typename M::Ctx& ctx, typename M::Acc& acc, dsr_later_smem& sm,
                                               unsigned hint) {
    const uint32_t np = sm.np;
    if constexpr (M::kDefers >= 0) {
        constexpr int T = M::kDefers;
        const uint32_t cap = H.cap[T];
        if (threadIdx.x < 32) {
            uint32_t nb = 0;
            if (np >= cap && cap >= 16) nb = dsr_claim_full(H, T, np / cap, hint, sm.block);
            if (threadIdx.x == 0) {
                sm.nb = nb;
                if (nb) dsr_count(H.ctr, DSR_CTR_ALLOCS, (dsr_u64)nb * cap);
            }
        }
        __syncthreads();
        const uint32_t full = sm.nb * cap;
        for (uint32_t p0 = threadIdx.x & ~31u; p0 < np; p0 += blockDim.x) {
            __syncwarp();
            const uint32_t p = p0 + (threadIdx.x & 31);
            if (p < np) {
                const dsr_ref r = p < full ? ((dsr_ref)sm.block[p / cap] << 6) | (p % cap) : dsr_new(H, T);
                M::born(H, I, ctx, sm.pending[p], r, acc);
            }
        }
    } else {
        for (uint32_t p0 = threadIdx.x & ~31u; p0 < np; p0 += blockDim.x) {
            __syncwarp();
            const uint32_t p = p0 + (threadIdx.x & 31);
            if (p < np) M::later(H, I, ctx, sm.pending[p], acc);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) sm.np = 0;
    __syncthreads();
}

// Add the sum over the calling warp (whole) of v to event counter k.
__device__ __forceinline__ void dsr_flush_count(const dsr_dev_heap& H, unsigned k, unsigned v) {
    v = __reduce_add_sync(0xFFFFFFFFu, v);
    if (dsr_lane() == 0 && v) dsr_count(H.ctr, k, v);
}

// A do-all over one list of a heap; called by the whole grid. `turn`: the
// warps take items from the other end, so that those with the fewest items of
// a do-all before this one in the same launch get the first of this one's.
template <class M>
__device__ __forceinline__ void dsr_run_list(const dsr_dev_heap& H, const dsr_phase& ph, const typename M::Args& a,
                                             bool turn, dsr_later_smem* sm) {
    const unsigned lane = threadIdx.x & 31;
    const int T = ph.type;
    const unsigned hsh = H.span_sh[T] - 5;  // log2 of the 32-slot items of a block
    const uint32_t W = gridDim.x * (blockDim.x >> 5);
    const uint32_t w0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const uint32_t w = turn ? W - 1 - w0 : w0;
    // 32 bits hold the items of any heap: a block of more than 32 slots has
    // at least 256 bytes, a smaller one 128 and one item
    const uint32_t items = *(volatile uint32_t*)(H.R_count + (ph.back ? DSR_LIST_BACK : 0)) << hsh;
    const typename M::Inst& I = M::inst(a, 0);
    const typename M::Ctx ctx = M::begin(I);
    typename M::Acc acc{};
    dsr_later later{sm, true};
    if constexpr (M::kDefers >= 0) {
        if (threadIdx.x < 32) {
            const bool few = dsr_few_holes(H, M::kDefers, blockIdx.x);
            if (threadIdx.x == 0) {
                sm->few = few;
                sm->np = 0;
            }
        }
        __syncthreads();
        later.on = sm->few != 0;
    } else if constexpr (M::kDefers == DSR_WORK) {
        if (threadIdx.x == 0) sm->np = 0;
        __syncthreads();
    }
    // with deferral, CTAs meet after so many items of every warp that the
    // pending words cannot overflow
    const uint32_t burst = M::kDefers == DSR_NOTHING ? 32u : DSR_PENDING / 2 / blockDim.x;
    for (uint32_t base = 0; base < items; base += 32 * W) {  // uniform over the grid
        // lane k holds the warp's k-th item from here
        const uint32_t mine = base + lane * W + w;
        uint32_t bid = 0, live = 0, half = 0;
        uint32_t at = 0;
        if (mine < items) {
            const uint32_t e = mine >> hsh;
            half = mine & ((1u << hsh) - 1);
            at = ph.back ? (uint32_t)H.M - 1 - e : e;
            bid = H.R_bid[at];
            live = reinterpret_cast<const uint32_t*>(H.R_mask + at)[half];
        }
        for (uint32_t k0 = 0; k0 < 32; k0 += burst) {
            if (base + k0 * W >= items) break;  // uniform over the grid
            for (uint32_t k = k0; k < k0 + burst && k < 32; ++k) {
                // reconverge: lanes that drifted apart in a method would
                // otherwise miss each other at warp-wide steps
                __syncwarp();
                const uint32_t m = __shfl_sync(0xFFFFFFFFu, live, k);
                if (!m) continue;
                const uint32_t b = __shfl_sync(0xFFFFFFFFu, bid, k);
                const uint32_t hf = __shfl_sync(0xFFFFFFFFu, half, k);
                unsigned mark = 0;
                if ((m >> lane) & 1u) mark = M::run(H, T, I, ctx, ((dsr_u64)b << 6) | (32 * hf + lane), later, acc);
                if (M::kMarks) {
                    mark = __ballot_sync(0xFFFFFFFFu, mark);
                    if (lane == k) reinterpret_cast<uint32_t*>(H.R_mask + at)[half] = mark;
                }
            }
            if constexpr (M::kDefers != DSR_NOTHING) {
                // the last thread to arrive sees every push: all decide alike
                if (__syncthreads_or(*(volatile uint32_t*)&sm->np > DSR_PENDING / 2)) dsr_do_pending<M>(H, I, ctx, acc, *sm, dsr_hash32(blockIdx.x + k0));
            }
        }
    }
    if constexpr (M::kDefers != DSR_NOTHING) {
        __syncthreads();
        if (sm->np) dsr_do_pending<M>(H, I, ctx, acc, *sm, dsr_hash32(blockIdx.x * 0x9E3779B1u));
        __syncthreads();
    }
    __syncwarp();
    M::flush(H, I, acc);
}

// End of a step's last do-all: true in every thread of the last CTA.
__device__ __forceinline__ bool dsr_last_cta(uint32_t* done) {
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
        if (last) *(volatile uint32_t*)done = 0;
        __threadfence();
    }
    __syncthreads();
    return last;
}

// One do-all, or two that do not depend on each other. END: the last of the
// step (its last CTA empties the lists). F: a type whose finish(H, args) that
// CTA's first thread runs.
template <class M1, class M2, bool END, class F, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 6 : 1)
    dsr_step_kernel(const __grid_constant__ dsr_dev_heap H, const __grid_constant__ dsr_phase p1,
                    const __grid_constant__ dsr_phase p2, const __grid_constant__ typename M1::Args a) {
    constexpr bool two = !std::is_same<M2, dsr_no_method>::value;
    constexpr int defers = M1::kDefers;
    dsr_later_smem* sm = nullptr;
    if constexpr (defers != DSR_NOTHING) {
        __shared__ dsr_later_smem later;
        sm = &later;
    }
    dsr_run_list<M1>(H, p1, a, false, sm);
    if constexpr (two) {
        static_assert(M2::kDefers == DSR_NOTHING || defers != DSR_NOTHING, "M2 uses M1's shared memory");
        dsr_run_list<M2>(H, p2, a, true, sm);
    }
    if constexpr (END) {
        if (dsr_last_cta(H.R_done) && threadIdx.x == 0) {
            *(volatile uint32_t*)H.R_count = 0;
            *(volatile uint32_t*)(H.R_count + DSR_LIST_BACK) = 0;
            if constexpr (!std::is_same<F, dsr_no_method>::value) F::finish(H, a);
        }
    }
}

// Queue one launch of a step.
template <class M1, class M2 = dsr_no_method, bool END = false, class F = dsr_no_method>
int dsr__step(dsr_heap* h, const dsr_phase& p1, const dsr_phase& p2, const typename M1::Args& a, cudaStream_t s) {
    const int threads = h->tune.threads;
    const bool small = threads <= 256;
    const void* k = small ? (const void*)dsr_step_kernel<M1, M2, END, F, 256>
                          : (const void*)dsr_step_kernel<M1, M2, END, F, 1024>;
    static int grid_cache[17] = {0};  // as in dsr__doall
    int grid;
    if (h->tune.ctas_per_sm > 0) {
        grid = dsr__persistent_grid(h, k, threads);
    } else {
        int& cached = grid_cache[threads / 64];
        if (cached == 0) cached = dsr__persistent_grid(h, k, threads);
        grid = cached;
    }
    const dsr_u64 most = (h->dev.M * 64 + threads - 1) / threads;
    if ((dsr_u64)grid > most) grid = (int)most;
    if (grid < 1) grid = 1;
    if (small)
        dsr_step_kernel<M1, M2, END, F, 256><<<grid, threads, 0, s>>>(h->dev, p1, p2, a);
    else
        dsr_step_kernel<M1, M2, END, F, 1024><<<grid, threads, 0, s>>>(h->dev, p1, p2, a);
    return dsr__check_launch("dsr_step_kernel");
}

// Queue the listing of type A (front) and, unless -1, type B (back). mult:
// visits counted per listed object.
void dsr__list_types(const dsr_heap* h, int type_a, int type_b, unsigned mult_a, unsigned mult_b, cudaStream_t s);

// ---- heap groups -------------------------------------------------------------
// The same over the heaps of a group: G.R_heap / R_bid / R_mask hold the
// entries of all heaps, type A's from the front and type B's from the back.
constexpr int DSR_GROUP_LIST_BACK = 32;  // index from G.R_count of the back's count

template <class M>
__device__ __forceinline__ void dsr_run_group_list(const dsr_group_dev& G, const dsr_phase& ph,
                                                   const typename M::Args& a, unsigned hsh, bool turn) {
    const unsigned lane = threadIdx.x & 31;
    const int T = ph.type;
    const uint32_t W = gridDim.x * (blockDim.x >> 5);
    const uint32_t w0 = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const uint32_t w = turn ? W - 1 - w0 : w0;
    const uint32_t items = *(volatile uint32_t*)(G.R_count + (ph.back ? DSR_GROUP_LIST_BACK : 0)) << hsh;
    dsr_later later{nullptr, false};
    for (uint32_t base = 0; base < items; base += 32 * W) {
        const uint32_t mine = base + lane * W + w;
        uint32_t bid = 0, live = 0, half = 0, heap = 0;
        uint32_t at = 0;
        if (mine < items) {
            const uint32_t e = mine >> hsh;
            half = mine & ((1u << hsh) - 1);
            at = ph.back ? (uint32_t)G.R_cap - 1 - e : e;
            heap = G.R_heap[at];
            bid = G.R_bid[at];
            live = reinterpret_cast<const uint32_t*>(G.R_mask + at)[half];
        }
        for (uint32_t k = 0; k < 32; ++k) {
            if (base + k * W >= items) break;
            __syncwarp();
            const uint32_t m = __shfl_sync(0xFFFFFFFFu, live, k);
            if (!m) continue;
            const uint32_t b = __shfl_sync(0xFFFFFFFFu, bid, k);
            const uint32_t h = __shfl_sync(0xFFFFFFFFu, heap, k);
            const uint32_t hf = __shfl_sync(0xFFFFFFFFu, half, k);
            if (!dsr_check(h < G.n_slots, G.err, G.dbg, 3, h) || !dsr_check(b < G.heaps[h].M, G.err, G.dbg, 4, b)) continue;
            const dsr_dev_heap& H = G.heaps[h];
            const typename M::Inst& I = M::inst(a, h);
            const typename M::Ctx ctx = M::begin(I);
            typename M::Acc acc{};
            unsigned mark = 0;
            if ((m >> lane) & 1u) mark = M::run(H, T, I, ctx, ((dsr_u64)b << 6) | (32 * hf + lane), later, acc);
            __syncwarp();
            if (M::kMarks) {
                mark = __ballot_sync(0xFFFFFFFFu, mark);
                if (lane == k) reinterpret_cast<uint32_t*>(G.R_mask + at)[half] = mark;
            }
            M::flush(H, I, acc);
        }
    }
}

template <class M1, class M2, bool END, class F, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 6 : 1)
    dsr_group_step_kernel(const __grid_constant__ dsr_group_dev G, const __grid_constant__ dsr_phase p1,
                          const __grid_constant__ dsr_phase p2, const __grid_constant__ typename M1::Args a,
                          unsigned hsh1, unsigned hsh2) {
    dsr_run_group_list<M1>(G, p1, a, hsh1, false);
    if constexpr (!std::is_same<M2, dsr_no_method>::value) dsr_run_group_list<M2>(G, p2, a, hsh2, true);
    if constexpr (END) {
        if (dsr_last_cta(G.R_done)) {
            if (threadIdx.x == 0) {
                *(volatile uint32_t*)G.R_count = 0;
                *(volatile uint32_t*)(G.R_count + DSR_GROUP_LIST_BACK) = 0;
            }
            if constexpr (!std::is_same<F, dsr_no_method>::value) F::finish_group(G, a);
        }
    }
}

template <class M1, class M2 = dsr_no_method, bool END = false, class F = dsr_no_method>
int dsr__group_step(dsr_group* g, const dsr_phase& p1, const dsr_phase& p2, const typename M1::Args& a,
                    cudaStream_t s) {
    const int threads = g->tune.threads > 0 ? g->tune.threads : 256;
    const unsigned h1 = dsr__group_span(g, p1.type) - 5, h2 = dsr__group_span(g, p2.type) - 5;
    if (threads <= 256) {
        const int grid = dsr__group_grid(g, (const void*)dsr_group_step_kernel<M1, M2, END, F, 256>, threads);
        dsr_group_step_kernel<M1, M2, END, F, 256><<<grid, threads, 0, s>>>(g->dev, p1, p2, a, h1, h2);
    } else {
        const int grid = dsr__group_grid(g, (const void*)dsr_group_step_kernel<M1, M2, END, F, 1024>, threads);
        dsr_group_step_kernel<M1, M2, END, F, 1024><<<grid, threads, 0, s>>>(g->dev, p1, p2, a, h1, h2);
    }
    return dsr__check_launch("dsr_group_step_kernel");
}

void dsr__group_list_types(const dsr_group* g, int type_a, int type_b, unsigned mult_a, unsigned mult_b,
                           cudaStream_t s);
