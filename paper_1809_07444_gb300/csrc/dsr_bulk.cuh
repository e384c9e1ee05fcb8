// Bulk creation of objects by whole CTAs: the kernels that place an
// application's initial state.
//
// dsr_new serves the requests of one warp at a time. A kernel in which every
// thread creates an object then has thousands of leaders opening blocks and
// searching for the ones the others opened, and is bound by those searches
// (throttled slow paths, empty descents, back-off), not by the objects: on a
// GB300, 6.7 M cars took 1730 us, 8192 bodies 131 us. Here a CTA first counts
// the objects of a chunk of its elements, claims whole blocks for them from
// the free bitmap, many with one atomic on a leaf word, and hands the slots
// out by a prefix sum. Blocks claimed this way are born full: their object
// bitmap stays 0 as it was and active[T] is not touched. What does not fill
// a block goes through dsr_new, in whole-warp groups, and so shares blocks
// with the other chunks' remainders.
// Objects of consecutive elements get consecutive slots, so their fields are
// written coalesced, and later do-alls find neighbours in the same block.
// Measured (us, dsr_new per thread -> this): 8192 x 4096 traffic cells with
// 6.7 M cars 1730 -> 161, 1500 x 1000 life cells 761 -> 52, 1.68 M sugarscape
// agents 434 -> 45, 2048 x 2048 wa-tor 302 -> 74, 4097 bodies 131 -> 13.
#pragma once

#include "dsr_internal.cuh"

constexpr int DSR_BULK_THREADS = 256;
constexpr int DSR_BULK_WARPS = DSR_BULK_THREADS / 32;
template <int NT>
constexpr int dsr_bulk_rows_max = 32 / NT;  // elements per thread and chunk at most: their kinds fill one word
constexpr int DSR_BULK_BLOCKS = 256;        // blocks claimed per type and chunk at most
constexpr int DSR_BULK_REST = 64;           // objects of a chunk beyond its full blocks (a block has at most 64 slots)

template <int NT, bool SPARSE = false>
struct dsr_bulk_smem {
    uint32_t before[NT][dsr_bulk_rows_max<NT> * DSR_BULK_WARPS];  // objects of the chunk before each (row, warp)
    uint32_t total[NT];
    uint32_t n_blocks[NT];
    uint32_t block[NT][DSR_BULK_BLOCKS];
    dsr_ref rest[NT][DSR_BULK_REST];
    uint16_t order[SPARSE ? dsr_bulk_rows_max<NT> * DSR_BULK_THREADS : 1];  // of object `rank`: its element in the chunk
};

// Claim up to `want` free blocks as full blocks of type T (every slot taken
// by the caller) and write their ids to out; called by a whole warp. Returns
// how many it got, the same in every lane: fewer than `want` when the free
// bitmap runs out or failures are being injected. The claim is the one of
// dsr_hb_clear with several bits of a leaf at once; like there, the call that
// leaves the leaf empty clears the nested bit. A free block's object bitmap
// is 0, which is also a full block's, so publishing one needs its type byte
// only, before the allocated[T] bit.
__device__ inline uint32_t dsr_claim_full(const dsr_dev_heap& H, int T, uint32_t want, unsigned hint, uint32_t* out) {
    const unsigned lane = dsr_lane();
    const unsigned sh = H.free_bm.shift;
    uint32_t n = 0;
    if (H.inject && *(volatile uint32_t*)H.inject != 0) return 0;
    for (unsigned a = 0; n < want && a < DSR_FIND_CAP; ++a) {
        dsr_u64 got = 0;
        long long leaf = -1;
        if (lane == 0) {
            const long long b = dsr_hb_find(H.free_bm, hint + a * 0x9E3779B9u);
            if (b >= 0) {
                leaf = b >> sh;
                dsr_u64* w = H.free_bm.lvl[0] + leaf;
                const dsr_u64 take = dsr_lowest_bits(dsr_ld_relaxed(w), (int)(want - n));
                if (take) {
                    const dsr_u64 prev = atomicAnd(w, ~take);
                    got = prev & take;
                    if (got && !(prev & ~take)) dsr_hb_clear_t<0>(H.free_bm, (dsr_u64)leaf, true, H.err, 1);
                }
            } else if (dsr_ld_relaxed(H.free_bm.lvl[H.free_bm.n_levels - 1]) == 0) {
                leaf = -2;  // nothing free
            } else {
                dsr_backoff(a);
            }
        }
        got = __shfl_sync(0xFFFFFFFFu, got, 0);
        leaf = __shfl_sync(0xFFFFFFFFu, leaf, 0);
        if (leaf == -2) break;
        if (!got) continue;
        const uint32_t k = (uint32_t)__popcll(got);
        for (uint32_t j = lane; j < k; j += 32) {
            const uint32_t b = ((uint32_t)leaf << sh) + (uint32_t)dsr_nth_bit(got, (int)j);
            H.btype[b] = (uint8_t)T;
            out[n + j] = b;
        }
        __threadfence();
        __syncwarp();
        if (lane == 0) {
            dsr_u64* w = H.alloc_bm[T].lvl[0] + leaf;
            dsr_u64 todo = got;
            for (unsigned tries = 0; todo; ++tries) {
                const dsr_u64 prev = atomicOr(w, todo);
                if (prev == 0) dsr_hb_set_t<0>(H.alloc_bm[T], (dsr_u64)leaf, true, H.err, 1);
                todo &= prev;  // a bit whose earlier owner has yet to clear it
                if (todo && tries >= DSR_SPIN_CAP) {
                    atomicOr(H.err, DSR_ERR_RETRY);
                    break;
                }
                if (todo) dsr_backoff(tries);
            }
            dsr_count(H.ctr, DSR_CTR_BLOCKS, k);
        }
        n += k;
    }
    __syncwarp();
    return n;
}

// Exclusive prefix sum of v over the calling warp (whole); *total: its sum.
__device__ __forceinline__ uint32_t dsr_warp_prefix(uint32_t v, uint32_t* total) {
    const unsigned lane = dsr_lane();
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += y;
    }
    *total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    return incl - v;
}

// Elements 0 .. n - 1, `rows` (1 .. dsr_bulk_rows_max<NT>) x 256 of them a chunk, one
// chunk per CTA and round. kind(i): bit k set if element i creates an object
// of types[k]. make(i, kind, refs): runs once for every element; refs[k] is
// the object for bit k (DSR_NULL if the bit is clear or memory ran out).
// SPARSE (one type): make runs for the elements that create an object only,
// and 32 of those at a time: the CTA lists them by rank first. With one cell
// in five holding a car a warp otherwise goes through make for six of its
// lanes (traffic's initial state, 33.5 M cells: 270 -> 161 us).
// Called by all 256 threads of every CTA of the grid.
template <int NT, bool SPARSE, class Kind, class Make>
__device__ __forceinline__ void dsr_bulk_create(const dsr_dev_heap& H, dsr_u64 n, int rows, const int (&types)[NT],
                                                dsr_bulk_smem<NT, SPARSE>& sm, Kind kind, Make make) {
    static_assert(!SPARSE || NT == 1, "a list of one type's objects");
    const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1;
    const dsr_u64 chunk = (dsr_u64)rows * DSR_BULK_THREADS;
    for (dsr_u64 base = blockIdx.x * chunk; base < n; base += gridDim.x * chunk) {
        unsigned kinds = 0;
        for (int r0 = 0; r0 < rows; r0 += 8) {  // eight elements of a thread are loaded at a time
            unsigned m[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const dsr_u64 i = base + (r0 + q) * DSR_BULK_THREADS + threadIdx.x;
                m[q] = r0 + q < rows && i < n ? kind(i) : 0u;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (r0 + q >= rows) break;
                kinds |= m[q] << (NT * (r0 + q));
#pragma unroll
                for (int k = 0; k < NT; ++k) {
                    const unsigned b = __ballot_sync(0xFFFFFFFFu, (m[q] >> k) & 1u);
                    if (lane == 0) sm.before[k][(r0 + q) * DSR_BULK_WARPS + warp] = __popc(b);
                }
            }
        }
        __syncthreads();
        if (warp < NT) {
            // exclusive prefix sum over the (row, warp) counts, some of them a lane
            constexpr int PER = dsr_bulk_rows_max<NT> * DSR_BULK_WARPS / 32;
            uint32_t* c = sm.before[warp];
            const int m = rows * DSR_BULK_WARPS;
            uint32_t v[PER], sum = 0;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int at = PER * (int)lane + q;
                v[q] = at < m ? c[at] : 0u;
                sum += v[q];
            }
            uint32_t total;
            uint32_t at = dsr_warp_prefix(sum, &total);
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                if (PER * (int)lane + q < m) c[PER * (int)lane + q] = at;
                at += v[q];
            }
            const int T = types[warp];
            uint32_t want = total / H.cap[T];
            if (want > DSR_BULK_BLOCKS) want = DSR_BULK_BLOCKS;
            const unsigned hint = dsr_hash32((unsigned)(base / chunk) * 0x9E3779B1u + warp);
            const uint32_t nb = want ? dsr_claim_full(H, T, want, hint, sm.block[warp]) : 0u;
            if (lane == 0) {
                sm.total[warp] = total;
                sm.n_blocks[warp] = nb;
                if (nb) dsr_count(H.ctr, DSR_CTR_ALLOCS, (dsr_u64)nb * H.cap[T]);
            }
        }
        __syncthreads();
        // the objects beyond the full blocks: two warps per type
        if (warp < 2 * NT) {
            const int k = (int)warp >> 1;
            const uint32_t at = (warp & 1) * 32 + lane;
            const uint32_t full = sm.n_blocks[k] * H.cap[types[k]];
            if (full + at < sm.total[k]) sm.rest[k][at] = dsr_new(H, types[k]);
        }
        if constexpr (SPARSE) {
            for (int r = 0; r < rows; ++r) {
                const bool set = (kinds >> r) & 1u;
                const unsigned b = __ballot_sync(0xFFFFFFFFu, set);
                if (set)
                    sm.order[sm.before[0][r * DSR_BULK_WARPS + warp] + __popc(b & below)] =
                        (uint16_t)(r * DSR_BULK_THREADS + threadIdx.x);
            }
            __syncthreads();
            const uint32_t total = sm.total[0], cap = H.cap[types[0]], full = sm.n_blocks[0] * cap;
            for (uint32_t at = warp * 32; at < total; at += DSR_BULK_THREADS) {
                const uint32_t rank = at + lane;
                if (rank < total) {
                    dsr_ref ref[1];
                    if (rank < full)
                        ref[0] = ((dsr_ref)sm.block[0][rank / cap] << 6) | (rank % cap);
                    else if (rank - full < DSR_BULK_REST)
                        ref[0] = sm.rest[0][rank - full];
                    else
                        ref[0] = dsr_new(H, types[0]);  // the free bitmap gave fewer blocks than asked for
                    make(base + sm.order[rank], 1u, ref);
                }
                __syncwarp();  // whole-warp groups for dsr_new
            }
            __syncthreads();  // the tables are reused by the next chunk
            continue;
        }
        __syncthreads();
        for (int r = 0; r < rows; ++r) {
            __syncwarp();  // whole-warp groups for dsr_new
            const dsr_u64 i = base + r * DSR_BULK_THREADS + threadIdx.x;
            const unsigned m = kinds >> (NT * r);
            dsr_ref refs[NT];
#pragma unroll
            for (int k = 0; k < NT; ++k) {
                refs[k] = DSR_NULL;
                const unsigned b = __ballot_sync(0xFFFFFFFFu, (m >> k) & 1u);
                if ((m >> k) & 1u) {
                    const uint32_t rank = sm.before[k][r * DSR_BULK_WARPS + warp] + __popc(b & below);
                    const uint32_t cap = H.cap[types[k]], full = sm.n_blocks[k] * cap;
                    if (rank < full)
                        refs[k] = ((dsr_ref)sm.block[k][rank / cap] << 6) | (rank % cap);
                    else if (rank - full < DSR_BULK_REST)
                        refs[k] = sm.rest[k][rank - full];
                    else
                        refs[k] = dsr_new(H, types[k]);  // the free bitmap gave fewer blocks than asked for
                }
                __syncwarp();
            }
            if (i < n) make(i, m & ((1u << NT) - 1), refs);
        }
        __syncthreads();  // the tables are reused by the next chunk
    }
}

// Rows of a chunk for n elements of which each may create objects of NT
// types: enough chunks for about four CTAs on every SM, and as many elements a
// chunk as that allows, so that few of a chunk's objects fall outside its full
// blocks.
template <int NT>
inline int dsr__bulk_rows(dsr_u64 n, int sm_count) {
    const dsr_u64 r = n / ((dsr_u64)DSR_BULK_THREADS * 4 * (dsr_u64)sm_count);
    return r < 1 ? 1 : (r > (dsr_u64)dsr_bulk_rows_max<NT> ? dsr_bulk_rows_max<NT> : (int)r);
}
inline unsigned dsr__bulk_grid(dsr_u64 n, int rows, int sm_count) {
    const dsr_u64 c = (n + (dsr_u64)rows * DSR_BULK_THREADS - 1) / ((dsr_u64)rows * DSR_BULK_THREADS);
    const dsr_u64 cap = (dsr_u64)sm_count * 8;
    return (unsigned)(c < 1 ? 1 : (c < cap ? c : cap));
}
