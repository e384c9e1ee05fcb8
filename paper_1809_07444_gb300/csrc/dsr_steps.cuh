// The do-alls of the applications' steps.
//
// dsr_parallel_do lists the allocated blocks of one type in one kernel and
// runs one method over the list in a second. A step of an application is a
// fixed sequence of do-alls over two types, and it knows which of them leave
// the live set of a type alone. So a step lists both types in one scan (type
// A's blocks from the front of R_bid / R_mask, type B's from the back:
// together at most as many entries as there are blocks), and every do-all of
// the step runs over those lists. A method that deletes objects replaces its
// entry's mask by the survivors (kMarks) where a later do-all of the step
// visits them. Two do-alls that do not depend on each other share a launch.
//
// A warp takes every W-th (block, 32 slots) item of the list, so that at any
// time the grid works on neighbouring entries; a CTA of a group do-all that
// creates takes one stretch, which lies in one or two heaps. A warp's 32 lanes
// load the entries of its next 32 items at once and hand them out by shuffle,
// so the list costs one round trip per 32 items and warp, not one per item.
//
// Deferred work. A method may put off an object's creation: it pushes a
// word, and the CTA later creates all pending objects together and calls
// M::born for each. Births come from the few lanes of a warp whose object
// breeds, and a search by their leader is a chain of five dependent accesses
// that the rest of the warp waits for, in competition with all other leaders.
// The list says where the free slots of the created type are: each CTA has a
// stretch of that type's blocks as well, whose holes are its own to fill, one
// block per thread, with one atomic each and no search. Only when they are
// full are whole blocks claimed (dsr_claim_full). A remainder goes to another
// CTA's partly filled block, if two searches find one; else a block is opened
// for it if it fills half of it or if the CTA has at least DSR_OPEN_SHARE blocks
// already (so that few are partly filled), or it goes through dsr_new. Work that
// few objects have (a dead agent's replacement) can be deferred in the same
// way without a creation: full warps then do it.
//
// A method is a type with
//   Args; Inst; Ctx; Acc
//   static Inst inst(const Args&, uint32_t heap)         the instance of a heap
//   static Ctx begin(const Inst&)                        once per do-all (plain) or item (group)
//   static unsigned run(H, T, const Inst&, const Ctx&, dsr_ref self, dsr_later&, Acc&)
//   kDefers: DSR_NOTHING, DSR_WORK (M::later(H, I, ctx, word, acc) for each
//     pushed word; not in groups) or the type created (M::born(H, I, ctx,
//     word, ref); words of 32 bits in groups); kDeferBack: whether that type
//     is listed at the back
//   kMarks: 1 if run's result (0 or 1) replaces the slot's bit of the list entry
//   static void flush(H, const Inst&, const Acc&)        by a whole warp: event
//     counts gathered in Acc go to memory
//
// Subtypes. A do-all over a type visits the objects of its subtypes as well
// (dsr_heap_set_bases), whose blocks the two-type scan does not list, and one
// of the two types may be a subtype of the other. The steps of a heap with
// such types (dsr__has_subtypes) go do-all by do-all, as dsr_parallel_do would:
// dsr__list_tree lists one type with its subtypes, and END follows where the
// live set has changed. A kDefers method then finds no list of the type it
// creates, or one with blocks of subtypes, which dsr_take gives back.
#pragma once

#include <type_traits>

#include "dsr_bulk.cuh"
#include "dsr_group.cuh"
#include "dsr_per_device.h"

// Words from R_count that the lists use. Their lengths live in two sets of
// (front, back) words, which steps use in turn: the scan of a step adds to one
// set, whose words are zero then, and the step's last do-all clears the other
// for the next. DSR_TURN counts the steps; the scan copies it to DSR_TURN_NOW,
// where the step's do-alls read which set is theirs, and the last do-all
// advances it. No kernel writes a word that another of its CTAs reads, so a
// step ends without a rendezvous of its last kernel's CTAs (a fence and an
// atomic that each waited for, 2 to 3 us a step). R_count[0], the length of
// dsr_doall_scan's list, stays zero.
constexpr uint32_t DSR_SET = 8;  // front of set 0; + 1: back; + 2, + 3: set 1
constexpr uint32_t DSR_TURN = 12, DSR_TURN_NOW = 13;
#ifndef DSR_OPEN_SHARE
#define DSR_OPEN_SHARE 16
#endif

enum { DSR_NOTHING = -1, DSR_WORK = -2 };
struct dsr_no_acc {};
struct dsr_no_method {};

// The list a do-all runs over: type T's entries, at the front or the back.
struct dsr_phase {
    int type;
    int back;
};

// Deferred words of a CTA at a time: two from every thread at least.
template <int MAXT>
struct dsr_later_smem {
    enum { PENDING = MAXT > 512 ? 2 * MAXT : 1024 };
    dsr_u64 pending[PENDING];
    dsr_ref ref[PENDING];
    uint16_t index[PENDING];  // groups: the pending words of the heap being served
    uint32_t block[PENDING / 16];
    uint32_t holes[MAXT / 32];  // per warp
    uint32_t np, nb, next, n_open, heap;
    dsr_ref open;  // the first slot of the block opened for the remainder
};

// push() may be called by any lanes of a warp.
struct dsr_later {
    uint32_t* np;
    dsr_u64* pending;
    dsr_u64 tag;  // groups: heap index << 32
    __device__ __forceinline__ void push(dsr_u64 word) {
        const unsigned act = __activemask();
        const unsigned lane = dsr_lane();
        const int leader = __ffs(act) - 1;
        uint32_t at = 0;
        if ((int)lane == leader) at = atomicAdd(np, (uint32_t)__popc(act));
        at = __shfl_sync(act, at, leader);
        pending[at + __popc(act & ((1u << lane) - 1))] = word | tag;
    }
};

// The length of this step's front or back list. Called by whole warps: five
// lanes read the words, one request a warp (read by all lanes word by word,
// the sector they are in had 36,000 requests from a full grid to answer: 20 us
// a kernel; read by one warp for the CTA, with a barrier, the car do-all of
// 6.7 M cars took 82 us instead of 63: its warps then march in step).
__device__ __forceinline__ uint32_t dsr_list_length(const uint32_t* R_count, int back) {
    const unsigned lane = dsr_lane();
    uint32_t v = 0;
    if (lane < 5) v = *(const volatile uint32_t*)(R_count + (lane < 4 ? DSR_SET + lane : DSR_TURN_NOW));
    const unsigned turn = __shfl_sync(0xFFFFFFFFu, v, 4);
    return __shfl_sync(0xFFFFFFFFu, v, 2 * (turn & 1) + (unsigned)back);
}
// The scan's part: the first word of the step's set, read by the threads that
// add to it, and the copy of the turn.
__device__ __forceinline__ uint32_t dsr_begin_step(uint32_t* R_count) {
    uint32_t turn = 0;
    if (threadIdx.x < 2) turn = *(volatile uint32_t*)(R_count + DSR_TURN);
    if (blockIdx.x == 0 && threadIdx.x == 0) *(volatile uint32_t*)(R_count + DSR_TURN_NOW) = turn;
    return DSR_SET + 2 * (turn & 1);
}
// By one thread of a step's last do-all, at any time.
__device__ __forceinline__ void dsr_end_step(uint32_t* R_count) {
    volatile uint32_t* w = R_count;
    const uint32_t next = w[DSR_TURN_NOW] + 1;
    w[DSR_SET + 2 * (next & 1)] = 0;
    w[DSR_SET + 2 * (next & 1) + 1] = 0;
    w[DSR_TURN] = next;
}

// The list of a heap, or of all heaps of a group.
struct dsr_heap_space {
    static constexpr bool kGroup = false;
    const dsr_dev_heap& H;
    const uint32_t* len = nullptr;  // the lists' lengths, in shared memory (small heaps), or by the turn
    __device__ __forceinline__ const dsr_dev_heap& heap(uint32_t) const { return H; }
    __device__ __forceinline__ uint32_t count(int back) const { return len ? len[back] : dsr_list_length(H.R_count, back); }
    __device__ __forceinline__ uint32_t at(uint32_t e, int back) const { return back ? (uint32_t)H.M - 1 - e : e; }
    __device__ __forceinline__ uint32_t heap_of(uint32_t) const { return 0; }
    __device__ __forceinline__ uint32_t bid(uint32_t at) const { return H.R_bid[at]; }
    __device__ __forceinline__ dsr_u64* mask(uint32_t at) const { return H.R_mask + at; }
    __device__ __forceinline__ bool ok(uint32_t, uint32_t b) const { return dsr_check(b < H.M, H.err, H.dbg, 10, b); }
};
struct dsr_group_space {
    static constexpr bool kGroup = true;
    const dsr_group_dev& G;
    __device__ __forceinline__ const dsr_dev_heap& heap(uint32_t h) const { return G.heaps[h]; }
    __device__ __forceinline__ uint32_t count(int back) const { return dsr_list_length(G.R_count, back); }
    __device__ __forceinline__ uint32_t at(uint32_t e, int back) const { return back ? (uint32_t)G.R_cap - 1 - e : e; }
    __device__ __forceinline__ uint32_t heap_of(uint32_t at) const { return G.R_heap[at]; }
    __device__ __forceinline__ uint32_t bid(uint32_t at) const { return G.R_bid[at]; }
    __device__ __forceinline__ dsr_u64* mask(uint32_t at) const { return G.R_mask + at; }
    __device__ __forceinline__ bool ok(uint32_t h, uint32_t b) const {
        return dsr_check(h < G.n_slots, G.err, G.dbg, 3, h) && dsr_check(b < G.heaps[h].M, G.err, G.dbg, 4, b);
    }
};

// Take up to k of the free slots `snap` of block b, the first ones at or after
// slot rot, for objects of type T; returns those obtained (an earlier taker's
// are missing). As in dsr_reserve: while slots of the block are held its type
// is fixed, and it may not be T, if the block was emptied and reused.
__device__ __forceinline__ dsr_u64 dsr_take(const dsr_dev_heap& H, int T, dsr_u64 b, dsr_u64 snap, int k, unsigned rot) {
    if (!snap) return 0;
    const dsr_u64 take = dsr_rotl(dsr_lowest_bits(dsr_rotr(snap, rot), k), rot);
    const dsr_u64 prev = dsr_atom_and_acquire(H.obj + b, ~take);
    const dsr_u64 got = prev & take;
    if (!got) return 0;
    const int T2 = dsr_block_type(H, b);
    if (!(prev & ~take)) dsr_hb_clear(H.active_bm[T2], b, true, H.err);
    if (T2 == T) return got;
    dsr_release(H, T2, b, got);
    return 0;
}
__device__ __forceinline__ void dsr_keep(dsr_ref* refs, uint32_t at, dsr_u64 b, dsr_u64 slots) {
    for (; slots; slots &= slots - 1) refs[at++] = (b << 6) | (dsr_ref)(__ffsll((long long)slots) - 1);
}

// Create the pending objects of a CTA. Called by the whole CTA, after a
// barrier.
template <class M, class Space, int MAXT>
__device__ __forceinline__ void dsr_create_pending(const Space& S, const typename M::Args& a, uint32_t cta,
                                                   uint32_t ctas, dsr_later_smem<MAXT>& sm, unsigned hint) {
    constexpr int T = M::kDefers;
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const uint32_t np = sm.np;
    // the CTA's stretch of the created type's blocks, one per thread (read
    // here and not kept: the method's loop has no registers to spare)
    const dsr_u64 blocks = S.count(M::kDeferBack);
    const uint32_t b0 = (uint32_t)(blocks * cta / ctas);
    const uint32_t share = (uint32_t)(blocks * (cta + 1) / ctas) - b0;
    uint32_t my_bid = 0, my_heap = 0xFFFFFFFFu;
    dsr_u64 my_free = 0;
    if (threadIdx.x < share) {
        const uint32_t at = S.at(b0 + threadIdx.x, M::kDeferBack);
        my_heap = S.heap_of(at);
        my_bid = S.bid(at);
        my_free = dsr_ld_relaxed(S.heap(my_heap).obj + my_bid);
    }
    for (;;) {  // one round per heap that has pending words (one round for a single heap)
        uint32_t n = np, hp = 0;
        if constexpr (Space::kGroup) {
            if (threadIdx.x == 0) {
                sm.heap = 0xFFFFFFFFu;
                sm.next = 0;
            }
            __syncthreads();
            for (uint32_t p = threadIdx.x; p < np; p += blockDim.x) atomicMin(&sm.heap, (uint32_t)(sm.pending[p] >> 32));
            __syncthreads();
            hp = sm.heap;
            if (hp == 0xFFFFFFFFu) break;
            for (uint32_t p = threadIdx.x; p < np; p += blockDim.x)
                if ((uint32_t)(sm.pending[p] >> 32) == hp) sm.index[atomicAdd(&sm.next, 1u)] = (uint16_t)p;
            __syncthreads();
            n = sm.next;
            __syncthreads();  // read before it is used again
        }
        const dsr_dev_heap& H = S.heap(hp);
        const uint32_t cap = H.cap[T];
        // the CTA's holes, in thread order
        const bool have = my_free && my_heap == hp;
        uint32_t in_warp;
        uint32_t before = dsr_warp_prefix(have ? (uint32_t)__popcll(my_free) : 0u, &in_warp);
        const unsigned own = __ballot_sync(0xFFFFFFFFu, my_heap == hp);  // blocks of this heap
        if (lane == 0) sm.holes[warp] = in_warp | ((uint32_t)__popc(own) << 16);
        if (threadIdx.x == 0) {
            sm.next = 0;
            sm.nb = 0;
            sm.n_open = 0;
        }
        __syncthreads();
        uint32_t holes = 0, own_blocks = 0;
        for (unsigned w = 0; w < warps; ++w) {
            if (w == warp) before += holes;
            holes += sm.holes[w] & 0xFFFFu;
            own_blocks += sm.holes[w] >> 16;
        }
        const uint32_t from_holes = n < holes ? n : holes;
        const uint32_t rest = n - from_holes;
        // beyond the holes: whole blocks, claimed by the first warp, and the
        // remainder, placed by the last
        if (warp == 0 && rest >= cap && cap >= 16) {
            const uint32_t nb = dsr_claim_full(H, T, rest / cap, hint, sm.block);
            if (lane == 0) {
                sm.nb = nb;
                if (nb) dsr_count(H.ctr, DSR_CTR_ALLOCS, (dsr_u64)nb * cap);
            }
        }
        const uint32_t rem = cap >= 16 ? rest % cap : rest < DSR_OPEN_SHARE ? rest : 0;
        if (warp == warps - 1 && lane == 0 && rem && !*(volatile uint32_t*)H.inject) {
            uint32_t left = rem;
            for (unsigned t = 0; t < 2 && left; ++t) {
                const unsigned h = dsr_hash32(hint ^ (t + 1) * 0x5bd1e995u);
                const long long b = dsr_hb_find(H.active_bm[T], h);
                if (b < 0) break;
                const dsr_u64 got = dsr_take(H, T, (dsr_u64)b, dsr_ld_relaxed(H.obj + b), (int)left, h >> 26);
                const uint32_t n = (uint32_t)__popcll(got);
                if (n) dsr_keep(sm.ref, atomicAdd(&sm.next, n), (dsr_u64)b, got);
                left -= n;
            }
            if (left != rem) dsr_count(H.ctr, DSR_CTR_ALLOCS, rem - left);
            if (left && (own_blocks >= DSR_OPEN_SHARE || 2 * left >= cap)) {
                const dsr_grab g = dsr_init_block(H, T, (int)left, hint ^ 0x5bd1e995u);
                if (!g.status) {
                    sm.open = g.bid << 6;  // its lowest slots: `left`, or all of a block with fewer
                    sm.n_open = (uint32_t)__popcll(g.bits);
                    dsr_count(H.ctr, DSR_CTR_ALLOCS, sm.n_open);
                }
            }
        }
        __syncwarp();
        // the holes, one block per thread; an earlier taker's slots are missing from `got`
        dsr_u64 got = 0;
        if (have && before < from_holes) {
            got = dsr_take(H, T, my_bid, my_free, (int)(from_holes - before), 0);
        }
        __syncwarp();
        uint32_t served;
        uint32_t r = dsr_warp_prefix((uint32_t)__popcll(got), &served), base = 0;
        if (lane == 0 && served) {
            base = atomicAdd(&sm.next, served);
            dsr_count(H.ctr, DSR_CTR_ALLOCS, (dsr_u64)served);
        }
        r += __shfl_sync(0xFFFFFFFFu, base, 0);
        dsr_keep(sm.ref, r, my_bid, got);
        __syncthreads();
        const uint32_t s0 = sm.next, s1 = s0 + sm.nb * cap, s2 = s1 + sm.n_open;
        const typename M::Inst& I = M::inst(a, hp);
        for (uint32_t q0 = threadIdx.x & ~31u; q0 < n; q0 += blockDim.x) {
            __syncwarp();
            const uint32_t q = q0 + lane;
            if (q < n) {
                dsr_ref r;
                if (q < s0)
                    r = sm.ref[q];
                else if (q < s1)
                    r = ((dsr_ref)sm.block[(q - s0) / cap] << 6) | ((q - s0) % cap);
                else if (q < s2)
                    r = sm.open + (q - s1);
                else
                    r = dsr_new(H, T);
                const uint32_t p = Space::kGroup ? sm.index[q] : q;
                const dsr_u64 word = sm.pending[p];
                if (Space::kGroup) sm.pending[p] = ~0ull;
                M::born(H, I, Space::kGroup ? (dsr_u64)(uint32_t)word : word, r);
            }
        }
        __syncthreads();
        if (!Space::kGroup) break;
    }
    if (threadIdx.x == 0) sm.np = 0;
    __syncthreads();
}

// Add the sum over the calling warp (whole) of v to event counter k.
__device__ __forceinline__ void dsr_flush_count(const dsr_dev_heap& H, unsigned k, unsigned v) {
    v = __reduce_add_sync(0xFFFFFFFFu, v);
    if (dsr_lane() == 0 && v) dsr_count(H.ctr, k, v);
}

// M::later for every pending word of a DSR_WORK method, by full warps. Called by the whole CTA, after a barrier.
template <class M, int MAXT>
__device__ __forceinline__ void dsr_work_pending(const dsr_dev_heap& H, const typename M::Inst& I,
                                                 const typename M::Ctx& ctx, typename M::Acc& acc,
                                                 dsr_later_smem<MAXT>& sm) {
    const uint32_t np = sm.np;
    for (uint32_t p0 = threadIdx.x & ~31u; p0 < np; p0 += blockDim.x) {
        __syncwarp();
        const uint32_t p = p0 + (threadIdx.x & 31);
        if (p < np) M::later(H, I, ctx, sm.pending[p], acc);
    }
    __syncthreads();
    if (threadIdx.x == 0) sm.np = 0;
    __syncthreads();
}

// A do-all over one list; called by the whole grid. hsh: log2 of the 32-slot
// items of a listed block. `turn`: the CTAs take the stretches in reverse
// order, so that those with the most work in a do-all before this one in the
// same launch do not have the most again.
template <class M, class Space, int MAXT>
__device__ __forceinline__ void dsr_run_list(const Space& S, const dsr_phase& ph, const typename M::Args& a,
                                             unsigned hsh, bool turn, dsr_later_smem<MAXT>* sm) {
    const unsigned lane = threadIdx.x & 31, warps = blockDim.x >> 5, warp = threadIdx.x >> 5;
    const int T = ph.type;
    const uint32_t cta = turn ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const dsr_u64 items = (dsr_u64)S.count(ph.back) << hsh;
    // the CTA's stretch: below 2^32 items in all, as a block of more than 32
    // slots has at least 256 bytes, and one with fewer is one item. Few items
    // go to few CTAs, one to a warp: what a CTA defers is then worth a block.
    const dsr_u64 wanted = (items + warps - 1) / warps;
    const uint32_t ctas = wanted < gridDim.x ? (uint32_t)wanted : gridDim.x;
    // Group do-alls that create take a stretch of items per CTA, so that a
    // CTA's births belong to one or two heaps. All others take every
    // (ctas * warps)-th item per warp: the grid is then at one place of the
    // list, and of the instances' grids, at a time (256 wa-tor instances, 46.6 M
    // cells, several times what L2 holds: with stretches the fish-choice
    // kernel took 1389 us, with every n-th item 629).
    constexpr bool kStretch = Space::kGroup && M::kDefers != DSR_NOTHING;
    const uint32_t end = kStretch ? (uint32_t)(cta < ctas ? items * (cta + 1) / ctas : 0) : (uint32_t)items;
    const uint32_t stride = kStretch ? warps : ctas * warps;
    const uint32_t cta0 = cta >= ctas ? end : kStretch ? (uint32_t)(items * cta / ctas) : cta * warps;
    dsr_later later{nullptr, nullptr, 0};
    if constexpr (M::kDefers != DSR_NOTHING) {
        later.np = &sm->np;
        later.pending = sm->pending;
        if (threadIdx.x == 0) sm->np = 0;
        __syncthreads();
    }
    // with deferral, CTAs meet after so many items of every warp that the
    // pending words cannot overflow
    constexpr uint32_t kHalf = dsr_later_smem<MAXT>::PENDING / 2;
    const uint32_t burst = M::kDefers == DSR_NOTHING ? 32u : kHalf / blockDim.x;
    typename M::Acc acc{};
    typename M::Ctx ctx{};
    if (!Space::kGroup) ctx = M::begin(M::inst(a, 0));
    for (uint32_t base = cta0; base < end; base += 32 * stride) {  // uniform over the CTA
        // lane k holds the warp's k-th item from here
        const uint32_t item = base + lane * stride + warp;
        uint32_t bid = 0, live = 0, half = 0, at = 0, heap = 0;
        if (item < end) {
            half = item & ((1u << hsh) - 1);
            at = S.at(item >> hsh, ph.back);
            heap = S.heap_of(at);
            bid = S.bid(at);
            live = reinterpret_cast<const uint32_t*>(S.mask(at))[half];
        }
        for (uint32_t k0 = 0; k0 < 32; k0 += burst) {
            if (base + k0 * stride >= end) break;  // uniform over the CTA
            for (uint32_t k = k0; k < k0 + burst && k < 32; ++k) {
                // reconverge: lanes that drifted apart in a method would
                // otherwise miss each other at warp-wide steps
                __syncwarp();
                const uint32_t m = __shfl_sync(0xFFFFFFFFu, live, k);
                if (!m) continue;
                const uint32_t b = __shfl_sync(0xFFFFFFFFu, bid, k);
                const uint32_t hf = __shfl_sync(0xFFFFFFFFu, half, k);
                const uint32_t h = Space::kGroup ? __shfl_sync(0xFFFFFFFFu, heap, k) : 0u;
                if (!S.ok(h, b)) continue;
                const dsr_dev_heap& H = S.heap(h);
                const typename M::Inst& I = M::inst(a, h);
                if (Space::kGroup) {
                    ctx = M::begin(I);
                    later.tag = (dsr_u64)h << 32;
                }
                unsigned mark = 0;
                if ((m >> lane) & 1u) mark = M::run(H, T, I, ctx, ((dsr_u64)b << 6) | (32 * hf + lane), later, acc);
                if (Space::kGroup || M::kMarks) __syncwarp();
                if (M::kMarks) {
                    mark = __ballot_sync(0xFFFFFFFFu, mark);
                    if (lane == k) reinterpret_cast<uint32_t*>(S.mask(at))[half] = mark;
                }
                if (Space::kGroup) {
                    M::flush(H, I, acc);
                    acc = typename M::Acc{};
                }
            }
            if constexpr (M::kDefers != DSR_NOTHING) {
                // the last to push reads the count after its own push, so a
                // count above the half is seen by one at least: all decide alike
                if (__syncthreads_or(*(volatile uint32_t*)&sm->np > kHalf)) {
                    if constexpr (M::kDefers >= 0)
                        dsr_create_pending<M, Space, MAXT>(S, a, cta, ctas, *sm, dsr_hash32(cta + k0 * 0x85EBCA77u));
                    else
                        dsr_work_pending<M, MAXT>(S.heap(0), M::inst(a, 0), ctx, acc, *sm);
                }
            }
        }
    }
    if constexpr (M::kDefers != DSR_NOTHING) {
        __syncthreads();
        if (sm->np) {
            if constexpr (M::kDefers >= 0)
                dsr_create_pending<M, Space, MAXT>(S, a, cta, ctas, *sm, dsr_hash32(cta * 0x9E3779B1u));
            else
                dsr_work_pending<M, MAXT>(S.heap(0), M::inst(a, 0), ctx, acc, *sm);
        }
        __syncthreads();
    }
    if (!Space::kGroup) {
        __syncwarp();
        M::flush(S.heap(0), M::inst(a, 0), acc);
    }
}

// The lists of a step: type A's allocated blocks at the front (ta is -1: none),
// type B's (tb is -1: none) at the back, with a snapshot of their occupied
// slots; mult: visits counted per listed object. One thread per block id and
// round of the CTAs cta, cta + ctas ..: a CTA forms the prefix sums of its
// warps' counts and reserves its runs with one atomic each (`set`: the first
// word of the lengths, needed in threads 0 and 1). A block has one
// type, so a thread takes part in one list at most; its bitmap words and its
// object bitmap load together.
template <int MAXT>
struct dsr_list_smem {
    unsigned n[2][MAXT / 32];
    unsigned base[2];
};
template <int MAXT>
__device__ __forceinline__ void dsr_list(const dsr_dev_heap& H, int ta, int tb, unsigned mult_a, unsigned mult_b,
                                         uint32_t set, dsr_list_smem<MAXT>& sm) {
    const dsr_u64 M = H.M;
    constexpr unsigned warps = MAXT / 32;  // the CTA has MAXT threads
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned fsh = H.free_bm.shift, flo = (1u << fsh) - 1;
    dsr_u64 objs = 0;
    for (dsr_u64 base = (dsr_u64)blockIdx.x * blockDim.x; base < M; base += (dsr_u64)gridDim.x * blockDim.x) {
        const dsr_u64 b = base + threadIdx.x;
        bool in_a = false, in_b = false;
        dsr_u64 obj = 0;
        if (b < M) {
            const dsr_u64 wa = ta >= 0 ? H.alloc_bm[ta].lvl[0][b >> fsh] : 0ull;
            const dsr_u64 wb = tb >= 0 ? H.alloc_bm[tb].lvl[0][b >> fsh] : 0ull;
            obj = H.obj[b];
            in_a = (wa >> (b & flo)) & 1ull;
            in_b = (wb >> (b & flo)) & 1ull;
        }
        const unsigned ba = __ballot_sync(0xFFFFFFFFu, in_a), bb = __ballot_sync(0xFFFFFFFFu, in_b);
        if (lane == 0) sm.n[0][warp] = __popc(ba), sm.n[1][warp] = __popc(bb);
        __syncthreads();
        if (threadIdx.x < 2) {
            unsigned total = 0;
#pragma unroll
            for (unsigned w = 0; w < warps; ++w) {
                const unsigned n = sm.n[threadIdx.x][w];
                sm.n[threadIdx.x][w] = total;
                total += n;
            }
            sm.base[threadIdx.x] = total ? atomicAdd(H.R_count + set + threadIdx.x, total) : 0;
        }
        __syncthreads();
        if (in_a || in_b) {
            const int l = in_a ? 0 : 1;
            const dsr_u64 live = H.valid[in_a ? ta : tb] & ~obj;
            const dsr_u64 k = sm.base[l] + sm.n[l][warp] + __popc((in_a ? ba : bb) & ((1u << lane) - 1));
            const dsr_u64 at = in_a ? k : M - 1 - k;
            H.R_bid[at] = (uint32_t)b;
            H.R_mask[at] = live;
            objs += (dsr_u64)__popcll(live) * (in_a ? mult_a : mult_b);
        }
        __syncthreads();
    }
    for (int o = 16; o; o >>= 1) objs += __shfl_xor_sync(0xFFFFFFFFu, objs, o);
    if (lane == 0 && objs) dsr_count(H.ctr, DSR_CTR_VISITS, objs);
}

// ---- small heaps: whole steps in one launch ----------------------------------
// On a small heap a do-all is a few microseconds of launch and dependent
// accesses, on a handful of SMs: one thread-block cluster runs the do-alls of
// many steps one after the other, with the cluster's hardware barrier between
// them instead of a kernel boundary.
constexpr int DSR_CLUSTER = 16;           // CTAs (a non-portable size)
constexpr int DSR_CLUSTER_THREADS = 512;
constexpr int DSR_CLUSTER_STEPS = 256;    // per launch

// The lengths in set `set` (its front's word), after a barrier.
__device__ __forceinline__ void dsr_set_lengths(const uint32_t* R_count, uint32_t set, uint32_t* len) {
    if (threadIdx.x < 2) len[threadIdx.x] = *(const volatile uint32_t*)(R_count + set + threadIdx.x);
    __syncthreads();
}
__device__ __forceinline__ void dsr_clear_set(uint32_t* R_count, uint32_t set) {
    volatile uint32_t* w = R_count;
    w[set] = 0;
    w[set + 1] = 0;
}
// The first thing a cluster's kernel does (`first`: one thread of the grid):
// both sets are zero behind the next cluster barrier. A step of the general
// form leaves its own set's lengths for the step after it to clear, and a heap
// can take both forms in turn (timed wa-tor steps are general ones).
__device__ __forceinline__ void dsr_clear_sets(uint32_t* R_count, bool first) {
    if (first) {
        dsr_clear_set(R_count, DSR_SET);
        dsr_clear_set(R_count, DSR_SET + 2);
    }
}

// All writes of the cluster's threads before it are visible to all of them after it.
__device__ __forceinline__ void dsr_cluster_barrier() {
    __syncthreads();
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Whether `kernel` can run as one cluster of DSR_CLUSTER CTAs on the heap's
// device, which its first use there also allows it to. known: the kernel's own.
bool dsr__cluster_fits(const dsr_heap* h, const void* kernel, dsr_per_device* known);
// Queue it with the given arguments.
int dsr__launch_cluster(const void* kernel, void** args, cudaStream_t s);
// Small heaps of the default tuning (a caller that sets threads or CTAs gets
// the kernels it set them for).
inline bool dsr__small_heap(const dsr_heap* h, dsr_u64 blocks) {
    return h->dev.M <= blocks && h->tune.threads == 256 && h->tune.ctas_per_sm <= 0;
}

// One do-all, or two that do not depend on each other. Five CTAs of 256 threads
// per SM (48 registers; sugarscape 1914 -> 1854, life 1500 x 1000 1632 -> 1565 us
// a pass against six, whose 40 registers spill); the group form, whose methods
// wait longer for their heap's view, has six (7440 against 7524). END: the last of the
// step. F: a type whose finish(H, args) one thread then runs (finish_group:
// the threads of one CTA), at any time during the do-all.
template <class M1, class M2, bool END, class F, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 5 : 1)
    dsr_step_kernel(const __grid_constant__ dsr_dev_heap H, const __grid_constant__ dsr_phase p1,
                    const __grid_constant__ dsr_phase p2, const __grid_constant__ typename M1::Args a) {
    dsr_later_smem<MAXT>* sm = nullptr;
    if constexpr (M1::kDefers != DSR_NOTHING) {
        __shared__ dsr_later_smem<MAXT> later;
        sm = &later;
    }
    const dsr_heap_space S{H};
    dsr_run_list<M1, dsr_heap_space, MAXT>(S, p1, a, H.span_sh[p1.type] - 5, false, sm);
    if constexpr (!std::is_same<M2, dsr_no_method>::value) {
        static_assert(M2::kDefers == DSR_NOTHING, "only the first do-all of a launch defers");
        dsr_run_list<M2, dsr_heap_space, MAXT>(S, p2, a, H.span_sh[p2.type] - 5, true, nullptr);
    }
    if constexpr (END) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            dsr_end_step(H.R_count);
            if constexpr (!std::is_same<F, dsr_no_method>::value) F::finish(H, a);
        }
    }
}

template <class M1, class M2, bool END, class F, int MAXT>
__global__ void __launch_bounds__(MAXT, MAXT == 256 ? 6 : 1)
    dsr_group_step_kernel(const __grid_constant__ dsr_group_dev G, const __grid_constant__ dsr_phase p1,
                          const __grid_constant__ dsr_phase p2, const __grid_constant__ typename M1::Args a,
                          unsigned hsh1, unsigned hsh2) {
    static_assert(M1::kDefers != DSR_WORK, "group do-alls defer creations only");
    dsr_later_smem<MAXT>* sm = nullptr;
    if constexpr (M1::kDefers != DSR_NOTHING) {
        __shared__ dsr_later_smem<MAXT> later;
        sm = &later;
    }
    const dsr_group_space S{G};
    dsr_run_list<M1, dsr_group_space, MAXT>(S, p1, a, hsh1, false, sm);
    if constexpr (!std::is_same<M2, dsr_no_method>::value) {
        static_assert(M2::kDefers == DSR_NOTHING, "only the first do-all of a launch defers");
        dsr_run_list<M2, dsr_group_space, MAXT>(S, p2, a, hsh2, true, nullptr);
    }
    if constexpr (END) {
        if (blockIdx.x == 0) {
            if (threadIdx.x == 0) dsr_end_step(G.R_count);
            if constexpr (!std::is_same<F, dsr_no_method>::value) F::finish_group(G, a);
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
    static dsr_grid_cache cache;
    int grid = dsr__tuned_grid(h, k, cache);
    const dsr_u64 most = (h->dev.M * 64 + threads - 1) / threads;
    if ((dsr_u64)grid > most) grid = (int)most;
    if (grid < 1) grid = 1;
    if (small)
        dsr_step_kernel<M1, M2, END, F, 256><<<grid, threads, 0, s>>>(h->dev, p1, p2, a);
    else
        dsr_step_kernel<M1, M2, END, F, 1024><<<grid, threads, 0, s>>>(h->dev, p1, p2, a);
    return dsr__check_launch("dsr_step_kernel");
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

// Queue the listing of type A (front) and, unless -1, type B (back). mult:
// visits counted per listed object.
void dsr__list_types(const dsr_heap* h, int type_a, int type_b, unsigned mult_a, unsigned mult_b, cudaStream_t s);
// The same for one type and its subtypes, at the front.
void dsr__list_tree(const dsr_heap* h, int type, unsigned mult, cudaStream_t s);
inline bool dsr__has_subtypes(const dsr_heap* h, int type) { return h->dev.sub[type] != (1u << type); }
void dsr__group_list_types(const dsr_group* g, int type_a, int type_b, unsigned mult_a, unsigned mult_b,
                           cudaStream_t s);
