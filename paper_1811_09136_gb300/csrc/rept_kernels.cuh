// Kernels of one REPT batch, in launch order:
//   k_classify  colour every edge (all hash groups), find the edges some
//               processor keeps, count new table entries per node, list the
//               touched nodes                                  (Alg. 1 "if h(u,v)==i")
//   k_plan      size the touched nodes' tables for their new entry counts and
//               reserve pool space for the ones that must be re-allocated
//   k_commit    move re-allocated tables (rehash), publish the new counts
//   k_insert    insert each kept edge (nbr, stream index) into both
//               endpoints' tables                              (Alg. 1 E^(i) <- E^(i) + {(u,v)})
//   k_units, k_order
//               group the edges that can close wedges by their larger endpoint
//               (those with a short smaller list stay as they are)
//   k_intersect for every edge t = (s, l), s the endpoint with fewer entries:
//               scan s's list, let through the entries that a filter of l's list
//               holds (short lists: whose colours may agree), look those up in
//               l's table, and count the wedges whose two edges both arrived
//               before t and carry the same kept colour; tally tau^(i), tau_u,
//               tau_v, tau_w
//                                                               (Alg. 1 UpdateTriangleCNT)
// Counting after inserting is exact because every entry carries its stream
// index and k_intersect only accepts entries with index < t: the state seen by
// edge t is exactly the sequential algorithm's state before t.
#pragma once

#include <type_traits>

#include "rept_common.cuh"

namespace rept {
// Internal linkage: every translation unit of the library that launches these kernels gets its own copy.
namespace {

__device__ __forceinline__ uint32_t* block_at(uint2* pool, unsigned long long off_quads) {
    return reinterpret_cast<uint32_t*>(pool) + 8ull * off_quads;
}
__device__ __forceinline__ const uint32_t* block_at(const uint2* pool, unsigned long long off_quads) {
    return reinterpret_cast<const uint32_t*>(pool) + 8ull * off_quads;
}

// A node's table of 2^lg slots at `table` holds 2^lg neighbour ids (keys; probed a 4-key, 16-byte
// bucket at a time) and, per id, its stream index (and colour word), laid out as key_word and eidx_of
// say.  Insert (nbr, eidx, cw): claim a key slot with a 32-bit CAS, then store the rest.
// Returns false only if the table has no empty slot left (impossible while cnt <= capacity / 2).
// Lookups read whole 4-key buckets, so where a key sits inside its bucket does not matter: an insert
// tries the slots of a bucket starting from one chosen by other bits of the key, so that keys sharing
// a home bucket seldom contend for the same slot, and moves to the next bucket only when all four are
// taken.
// The slot of its home bucket, whose ids are q, that an insert of nbr tries first: an empty one if there
// is one.
__device__ __forceinline__ uint32_t empty_slot(const uint4& q, uint32_t nbr) {
    const uint32_t start = (nbr * 0x85EBCA6Bu) >> 30;
    const uint32_t empty = (q.x == kEmptyId ? 1u : 0u) | (q.y == kEmptyId ? 2u : 0u) | (q.z == kEmptyId ? 4u : 0u) |
                           (q.w == kEmptyId ? 8u : 0u);
    const uint32_t from = (empty | (empty << 4)) >> start;  // bit i: slot start + i
    return empty ? (start + (uint32_t)__ffs((int)from) - 1u) & 3u : start;
}

__device__ __forceinline__ void table_store(uint32_t* table, uint32_t lg, uint32_t h, uint32_t eidx, uint32_t cw,
                                            uint32_t colours) {
    uint32_t* at = eidx_of(table, h, lg, colours);
    if (colours == kColMulti) *reinterpret_cast<uint2*>(at) = make_uint2(eidx, cw);
    else *at = eidx;
}

__device__ __forceinline__ bool table_insert(uint32_t* table, uint32_t lg, uint32_t nbr, uint32_t eidx, uint32_t cw,
                                             uint32_t colours) {
    const uint32_t mask = (1u << lg) - 1u;
    const uint32_t start = (nbr * 0x85EBCA6Bu) >> 30;
    uint32_t b = home_slot(nbr, lg);
    for (uint32_t probe = 0; probe <= mask; probe += 4u) {
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) {
            const uint32_t h = b + ((start + i) & 3u);
            if (atomicCAS(table + key_word(h, colours), kEmptyId, nbr) == kEmptyId) {
                table_store(table, lg, h, eidx, cw, colours);
                return true;
            }
        }
        b = (b + 4u) & mask;
    }
    return false;
}

// First statement of every kernel of a single stream's batch.  Each but k_classify is launched as the programmatic
// dependent of the one before it on its stream: its blocks may be set up while that one's last blocks still
// run, and wait here until it (and so all that it waited for) has ended and its writes are visible.
__device__ __forceinline__ void follow_previous() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Has an earlier step failed?  The answer is the same for the whole block (another block may be setting
// the status meanwhile), so that its threads meet at the same barriers.
__device__ __forceinline__ bool block_failed(const Ctrl* c) {
    __shared__ unsigned s_status;
    __syncthreads();
    if (threadIdx.x == 0) s_status = c->status;
    __syncthreads();
    return s_status != 0u;
}

// Scratch that lives in another step's memory: per edge, its places among the batch's new entries of its
// two endpoints (k_classify to k_insert, where the units go later); per touched node, the batch's new
// entries (k_plan to k_commit, where the work records go later).
__device__ __forceinline__ uint2* edge_ranks(const StreamDev& d) { return reinterpret_cast<uint2*>(d.units); }
__device__ __forceinline__ uint32_t* touched_adds(const StreamDev& d) { return reinterpret_cast<uint32_t*>(d.rec); }

__device__ __forceinline__ void k_classify_body(const StreamDev& d, const BatchDev& b, const Grid g) {
    // the previous batch's work lists are consumed
    if (g.bx == 0 && threadIdx.x < kBins) {
        d.ctrl->bin_next[threadIdx.x] = 0ull;
        d.ctrl->bin_count[threadIdx.x] = threadIdx.x == kBinSmall ? (b.n + b.chunk - 1u) / b.chunk : 0ull;
    }
    if (g.bx == 0 && threadIdx.x == 0) {
        d.ctrl->n_pairs = 0ull;
        d.ctrl->n_groups = 0ull;
        d.ctrl->n_items = 0ull;
    }
    if (block_failed(d.ctrl)) return;
    __shared__ BlockReserve<uint32_t> part[2];
    uint32_t turn = 0;
    const unsigned long long stride = (unsigned long long)g.nbx * blockDim.x;
    for (unsigned long long base = (unsigned long long)g.bx * blockDim.x; base < b.n; base += stride) {
        const unsigned long long e = base + threadIdx.x;
        const bool valid = e < b.n;
        uint32_t u = 0, v = 0;
        if (valid) { u = b.src[e]; v = b.dst[e]; }
        const bool in_range = u < d.n_nodes && v < d.n_nodes;
        if (valid && !in_range) atomicOr(&d.ctrl->status, kStRange);
        const bool kept = valid && in_range && u != v && kept_by_any(d, u, v);
        bool first_u = false, first_v = false;
        if (kept) {  // the edge's places among the batch's new entries of u and v, for k_insert
            const uint32_t ru = atomicAdd(&d.cnt_add[u], 1u), rv = atomicAdd(&d.cnt_add[v], 1u);
            first_u = ru == 0u;
            first_v = rv == 0u;
            edge_ranks(d)[e] = make_uint2(ru, rv);
        }
        unsigned long long o = block_reserve(part[turn], &d.ctrl->n_touched, (first_u ? 1u : 0u) + (first_v ? 1u : 0u));
        if (first_u) d.touched[o++] = u;
        if (first_v) d.touched[o] = v;
        turn ^= 1u;
    }
}

// AGAIN: the batch's new entries have been taken by an earlier pass (the blocks' layout has changed since).
template <bool AGAIN = false>
__device__ __forceinline__ void k_plan_body(const StreamDev& d, const Grid g) {
    if (block_failed(d.ctrl)) return;
    // (whole block sizes: those of a few hundred large hubs together pass 2^32 quads)
    __shared__ BlockReserve<unsigned long long> part[2];
    uint32_t turn = 0;
    const unsigned long long n_t = d.ctrl->n_touched;
    const unsigned long long stride = (unsigned long long)g.nbx * blockDim.x;
    for (unsigned long long base = (unsigned long long)g.bx * blockDim.x; base < n_t; base += stride) {
        const unsigned long long i = base + threadIdx.x;
        const bool valid = i < n_t;
        uint32_t need = 0;
        if (valid) {
            const uint32_t x = d.touched[i];
            const uint32_t cnt = d.meta[x].y, add = AGAIN ? touched_adds(d)[i] : d.cnt_add[x];
            if (!AGAIN) {
                d.cnt_add[x] = 0u;  // zero again for the next batch
                touched_adds(d)[i] = add;
            }
            const uint32_t lg_old = table_lg(cnt), lg_new = table_lg(cnt + add);
            if (lg_new != lg_old) need = block_quads(lg_new, d.colours);
        }
        const unsigned long long rel = block_reserve(part[turn], &d.ctrl->need_quads, need);
        if (valid) d.grow_rel[i] = need ? (uint32_t)rel : kNoGrow;
        turn ^= 1u;
    }
}

// REPT_DEBUG_BOUNDS: the block with a table of 2^lg slots at `off_quads` lies inside the pool.
__device__ __forceinline__ bool block_fits(const StreamDev& d, unsigned site, unsigned long long off_quads,
                                          uint32_t lg) {
    return REPT_CHECK(d.ctrl, site, off_quads + block_quads(lg, d.colours) - 1ull, d.pool_quads);
}

// Copy n entries' words from one 16-byte aligned array to another (whole quads: the arrays' capacities
// are multiples of four words), lanes `rank` of `width`.
__device__ __forceinline__ void copy_words(uint32_t* to, const uint32_t* from, uint32_t n, uint32_t rank, uint32_t width) {
    for (uint32_t q = rank; q < (n + 3u) / 4u; q += width)
        reinterpret_cast<uint4*>(to)[q] = reinterpret_cast<const uint4*>(from)[q];
}

// Copy the list of cnt_old entries from the block at `from` (table of 2^lg_old slots) to the new one.
__device__ __forceinline__ void move_list(uint32_t* to, const uint32_t* from, uint32_t cnt_old, uint32_t lg_old,
                                          uint32_t lg_new, uint32_t colours, uint32_t rank, uint32_t width) {
    copy_words(list_of(to, lg_new, colours), list_of(from, lg_old, colours), cnt_old, rank, width);
    if (colours == kColWords) copy_words(cw_of(to, lg_new), cw_of(from, lg_old), cnt_old, rank, width);
    if (colours == kColNone || colours == kColMulti)
        copy_words(aux_of(to, lg_new, colours), aux_of(from, lg_old, colours),
                   colours == kColMulti ? 2u * cnt_old : cnt_old, rank, width);
}

// Call put(id, eidx, j) for every entry of the block at `from`: from its table (interleaved tables, whose
// lists hold no stream indices; j unused) or from its list, whose entry j it is.
template <class Put>
__device__ __forceinline__ void each_entry(const uint32_t* from, uint32_t cnt, uint32_t lg, uint32_t colours, uint32_t rank,
                                           uint32_t width, Put&& put) {
    if (interleaved(colours)) {
        if (cnt == 0u) return;
        const uint4* quads = reinterpret_cast<const uint4*>(from);
        for (uint32_t b = rank; b < (1u << lg) / 4u; b += width) {
            const uint4 id = quads[2u * b], t = quads[2u * b + 1u];
            if (id.x != kEmptyId) put(id.x, t.x, 0u);
            if (id.y != kEmptyId) put(id.y, t.y, 0u);
            if (id.z != kEmptyId) put(id.z, t.z, 0u);
            if (id.w != kEmptyId) put(id.w, t.w, 0u);
        }
    } else {
        const uint32_t *ids = list_of(from, lg, colours), *aux = aux_of(from, lg, colours);
        const uint32_t step = colours == kColMulti ? 2u : 1u;
        for (uint32_t j = rank; j < cnt; j += width) put(ids[j], aux[j * step], j);
    }
}

// Move a node's block of cnt_old entries at `from` into its new block at `to`, whose table keys are
// empty: copy the list and insert each entry into the new table.  Lanes `rank` of `width` share the work.
__device__ __forceinline__ bool move_block(uint32_t* to, const uint32_t* from, uint32_t cnt_old, uint32_t lg_new,
                                           uint32_t colours, uint32_t rank, uint32_t width) {
    const uint32_t lg_old = table_lg(cnt_old);
    move_list(to, from, cnt_old, lg_old, lg_new, colours, rank, width);
    bool ok = true;
    const uint32_t* aux = aux_of(from, lg_old, colours);
    each_entry(from, cnt_old, lg_old, colours, rank, width, [&](uint32_t id, uint32_t eidx, uint32_t j) {
        ok &= table_insert(to, lg_new, id, eidx, colours == kColMulti ? aux[2u * j + 1u] : 0u, colours);
    });
    return ok;
}

// Set every key of the new table of 2^lg slots at `table` to empty (lanes `rank` of `width`).  The
// pool is not cleared between streams: a block's table gets its empty keys when the block is handed
// out, from here or from the shared-memory builds, which write the whole table.  (Stream indices are
// read only beside a matching key, so they need no initial value.)
__device__ __forceinline__ void init_table_keys(uint32_t* table, uint32_t lg, uint32_t colours, uint32_t rank,
                                                uint32_t width) {
    uint4* quads = reinterpret_cast<uint4*>(table);
    const uint4 empty = make_uint4(kEmptyId, kEmptyId, kEmptyId, kEmptyId);
    for (uint32_t b = rank; b < (1u << lg) / 4u; b += width) quads[interleaved(colours) ? 2u * b : b] = empty;
}

// New tables of at most kMoveSlots slots are rebuilt in shared memory by a warp (k_rehash_big), those
// of at most kBlockMoveSlots by a thread block (k_rehash_huge); larger ones are built in place, each by
// kGiantPieces thread blocks, for a table that one block moves is longer under way than the rest of a
// batch's moves together.  Commit and moves, one block for each table against so: R-MAT scale 20 1.73 and
// 1.62 ms (15 batches), 1.5M edges in batches of 65,536 1.19 and 0.92 ms, 2M edges with hubs of 170,000 0.86
// and 0.41 ms (with the limit at 16,384 slots 1.60, 0.95 and 0.44; at 32,768 1.60, 1.04 and 0.50).
constexpr uint32_t kMoveSlots = 512;
constexpr uint32_t kBlockMoveSlots = 8192;
constexpr uint32_t kGiantPieces = 16;
constexpr uint32_t kHugeSmemWords = kBlockMoveSlots / 2u;  // a 16-bit word per slot

// move_block with the new table built in shared memory (keys and, per key, its stream index or with
// kColMulti its list position; 2^lg_new slots, the same placement rule as table_insert) and then written
// out with coalesced stores, by the lanes `rank` of `width` of one warp.  The new block is the caller's alone
// until the batch's inserts run.  Parts of a warp may each move a node at the same time; an inactive part
// takes part in the barriers only.
__device__ __forceinline__ bool move_block_smem(uint32_t* to, const uint32_t* from, uint32_t cnt_old, uint32_t lg_new,
                                                uint32_t colours, uint32_t* s_keys, uint32_t* s_aux, uint32_t rank,
                                                uint32_t width, bool active = true) {
    const uint32_t cap = active ? 1u << lg_new : 0u, mask = cap - 1u;
    for (uint32_t q = rank; q < cap; q += width) s_keys[q] = kEmptyId;
    __syncwarp();
    const uint32_t lg_old = table_lg(cnt_old);
    move_list(to, from, cnt_old, lg_old, lg_new, colours, rank, width);
    bool ok = true;
    each_entry(from, cnt_old, lg_old, colours, rank, width, [&](uint32_t key, uint32_t eidx, uint32_t j) {
        const uint32_t start = (key * 0x85EBCA6Bu) >> 30;
        uint32_t b = home_slot(key, lg_new);
        bool placed = false;
        for (uint32_t probe = 0; probe <= mask && !placed; probe += 4u) {
            for (uint32_t i = 0; i < 4u && !placed; ++i) {
                const uint32_t h = b + ((start + i) & 3u);
                if (atomicCAS(&s_keys[h], kEmptyId, key) == kEmptyId) {
                    s_aux[h] = colours == kColMulti ? j : eidx;
                    placed = true;
                }
            }
            b = (b + 4u) & mask;
        }
        ok &= placed;
    });
    __syncwarp();
    uint4* quads = reinterpret_cast<uint4*>(to);
    for (uint32_t b = rank; b < cap / 4u; b += width) {
        const uint4 id = reinterpret_cast<const uint4*>(s_keys)[b], t = reinterpret_cast<const uint4*>(s_aux)[b];
        if (interleaved(colours)) {
            quads[2u * b] = id;
            quads[2u * b + 1u] = t;
        } else {
            quads[b] = id;
            if (colours == kColNone) quads[cap / 4u + b] = t;
        }
    }
    if (colours == kColMulti) {  // the pairs of the keys' entries, from the old list
        const uint2* pairs = reinterpret_cast<const uint2*>(aux_of(from, lg_old, colours));
        uint2* out = reinterpret_cast<uint2*>(to + cap);
        for (uint32_t q = rank; q < cap; q += width)
            if (s_keys[q] != kEmptyId) out[q] = pairs[s_aux[q]];
    }
    return ok;
}

// Publish the new entry counts of the touched nodes and move the blocks that were re-allocated: those
// with new tables of at most kPartSlots slots here, eight at a time by four lanes each (a thread per node
// with global compare-and-swaps paid their latency once per entry); the others are left to k_rehash_big
// (a warp each, new tables of at most kMoveSlots slots) or k_rehash_huge (a thread block each).  49 batches
// of 4,096 edges: the three kernels took 2.1 ms with a thread per node, 1.8 ms so.
// `smem`: kCommitSmemWords words.
constexpr uint32_t kPartSlots = 64u, kPartLanes = 4u;
constexpr uint32_t kCommitSmemWords = 2u * (256u / kPartLanes) * kPartSlots;
__device__ __forceinline__ void k_commit_body(const StreamDev& d, const Grid g, uint32_t* smem) {
    const unsigned status = d.ctrl->status;
    const unsigned long long n_t = d.ctrl->n_touched;
    const unsigned long long need = d.ctrl->need_quads, top = d.ctrl->pool_top;
    const bool bad = status != 0u || top + need > d.pool_quads;
    if (status == 0u && bad && g.bx == 0 && threadIdx.x == 0) atomicOr(&d.ctrl->status, kStCapacity);
    if (bad) return;
    const unsigned lane = threadIdx.x & 31u, part = lane / kPartLanes, rank = lane % kPartLanes;
    uint32_t* s_keys = smem + (threadIdx.x / kPartLanes) * 2u * kPartSlots;
    uint32_t* s_aux = s_keys + kPartSlots;
    const unsigned long long stride = (unsigned long long)g.nbx * blockDim.x;
    for (unsigned long long base = (unsigned long long)g.bx * blockDim.x + threadIdx.x - lane; base < n_t;
         base += stride) {
        const unsigned long long i = base + lane;
        bool move = false, defer = false, huge = false;
        uint32_t off_old = 0, cnt_old = 0, off_new = 0, lg_new = 0;
        if (i < n_t) {
            const uint32_t x = d.touched[i];
            const uint4 m = d.meta[x];
            const uint32_t cnt_new = m.y + touched_adds(d)[i];
            const uint32_t rel = d.grow_rel[i];
            if (rel == kNoGrow) {
                d.meta[x].y = cnt_new;
            } else {
                lg_new = table_lg(cnt_new);
                off_old = m.x;
                cnt_old = m.y;
                off_new = (uint32_t)(top + rel);
                move = (1u << lg_new) <= kPartSlots;
                defer = !move && (1u << lg_new) <= kMoveSlots;
                huge = !move && !defer;
                if (move) d.meta[x] = make_uint4(off_new, cnt_new, 0u, 0u);
                if (!(block_fits(d, 10, off_old, table_lg(cnt_old)) && block_fits(d, 11, off_new, lg_new))) move = false;
            }
        }
        const unsigned movers = __ballot_sync(0xFFFFFFFFu, move);
        const uint32_t n_move = __popc(movers);
        for (uint32_t r = 0; r < n_move; r += 32u / kPartLanes) {
            const bool active = r + part < n_move;
            uint32_t from = 0;  // the lane of the part's node: the (r + part)-th mover
#pragma unroll
            for (uint32_t step = 16u; step; step >>= 1)
                if ((uint32_t)__popc(movers & ((1u << (from + step)) - 1u)) <= r + part) from += step;
            const uint32_t oo = __shfl_sync(0xFFFFFFFFu, off_old, from), co = __shfl_sync(0xFFFFFFFFu, cnt_old, from),
                           on = __shfl_sync(0xFFFFFFFFu, off_new, from), ln = __shfl_sync(0xFFFFFFFFu, lg_new, from);
            if (!move_block_smem(block_at(d.pool, on), block_at(d.pool, oo), active ? co : 0u, ln, d.colours, s_keys,
                                        s_aux, rank, kPartLanes, active))
                atomicOr(&d.ctrl->status, kStInternal);
            __syncwarp();
        }
        const unsigned long long o = warp_reserve_one(&d.ctrl->n_big, defer);
        if (defer) d.big[o] = (uint32_t)i;
        if (huge && (1u << lg_new) > kBlockMoveSlots) {
            // listed in the memory that the batch's larger endpoints and their edges use later; what does not
            // fit there (batches of a few edges) is moved by one block
            const uint32_t k = atomicAdd(&d.ctrl->n_giant, 1u);
            if (k < d.unit_cap) {
                d.glist[k] = (uint32_t)i;
                d.order[k] = 0u;  // pieces that are done
                huge = false;
            }
        }
        const unsigned long long h = warp_reserve_one(&d.ctrl->n_huge, huge);
        if (huge) d.big[d.big_cap - 1 - h] = (uint32_t)i;
    }
}

// The move of the i-th touched node's block.
struct Move {
    uint32_t x, cnt_old, cnt_new, lg_new, off_new;
    uint32_t *to, *from;
    bool fits;
};
__device__ __forceinline__ Move move_of(const StreamDev& d, uint32_t i, unsigned long long top) {
    Move mv;
    mv.x = d.touched[i];
    const uint4 m = d.meta[mv.x];
    const unsigned long long off = top + d.grow_rel[i];
    mv.cnt_old = m.y;
    mv.cnt_new = m.y + touched_adds(d)[i];
    mv.lg_new = table_lg(mv.cnt_new);
    mv.off_new = (uint32_t)off;
    mv.fits = block_fits(d, 10, m.x, table_lg(m.y)) && block_fits(d, 11, off, mv.lg_new);
    mv.to = block_at(d.pool, off);
    mv.from = block_at(d.pool, m.x);
    return mv;
}
// Nodes listed for moves in pieces.
__device__ __forceinline__ unsigned long long n_giants(const StreamDev& d) {
    return min((unsigned long long)d.ctrl->n_giant, (unsigned long long)d.unit_cap);
}

// Move the blocks listed by k_commit whose new table has at most kMoveSlots slots: one warp per node.
// `smem`: a key and a stream-index table of kMoveSlots slots for each of the block's warps (kMoveSmemWords
// words for 8).
constexpr uint32_t kMoveSmemWords = 2u * 8u * kMoveSlots;
__device__ __forceinline__ void k_rehash_big_body(const StreamDev& d, const Grid g, uint32_t* smem) {
    const unsigned long long n_big = d.ctrl->n_big, top = d.ctrl->pool_top;
    // the tables that k_rehash_huge builds in place start with empty keys
    for (unsigned long long p = g.bx; p < n_giants(d) * kGiantPieces; p += g.nbx) {
        const Move mv = move_of(d, d.glist[p / kGiantPieces], top);
        if (mv.fits)
            init_table_keys(mv.to, mv.lg_new, d.colours, (uint32_t)(p % kGiantPieces) * blockDim.x + threadIdx.x,
                            kGiantPieces * blockDim.x);
    }
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    const unsigned long long warps = ((unsigned long long)g.nbx * blockDim.x) >> 5;
    for (unsigned long long k = ((unsigned long long)g.bx * blockDim.x + threadIdx.x) >> 5; k < n_big;
         k += warps) {
        const Move mv = move_of(d, d.big[k], top);
        bool ok = true;
        if (mv.fits && REPT_CHECK(d.ctrl, 14, wid, 32u))
            ok = move_block_smem(mv.to, mv.from, mv.cnt_old, mv.lg_new, d.colours, smem + wid * 2u * kMoveSlots,
                                 smem + (wid * 2u + 1u) * kMoveSlots, lane, 32u);
        if (!ok) atomicOr(&d.ctrl->status, kStInternal);
        __syncwarp();
        if (lane == 0) d.meta[mv.x] = make_uint4(mv.off_new, mv.cnt_new, 0u, 0u);
    }
}

// move_block by one thread block, for tables of at most kBlockMoveSlots slots: the new table is laid out in
// shared memory as one 16-bit number per slot, 1 + where its entry stands in the old block (table slot or
// list position), and then written out bucket by bucket.  Built in place instead, with a global
// compare-and-swap per entry, the moves of R-MAT scale 20 took 1.02 ms, so 0.85 ms.
__device__ __forceinline__ bool move_block_index(uint32_t* to, const uint32_t* from, uint32_t cnt_old, uint32_t lg_new,
                                                 uint32_t colours, uint16_t* s_at) {
    const uint32_t cap = 1u << lg_new, mask = cap - 1u, lg_old = table_lg(cnt_old), rank = threadIdx.x, width = blockDim.x;
    const bool inter = interleaved(colours);
    for (uint32_t q = rank; q < cap / 8u; q += width) reinterpret_cast<uint4*>(s_at)[q] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    move_list(to, from, cnt_old, lg_old, lg_new, colours, rank, width);
    bool ok = true;
    auto place = [&](uint32_t key, uint32_t at) {
        const uint32_t start = (key * 0x85EBCA6Bu) >> 30;
        uint32_t b = home_slot(key, lg_new);
        for (uint32_t probe = 0; probe <= mask; probe += 4u) {
            for (uint32_t i = 0; i < 4u; ++i)
                if (atomicCAS(reinterpret_cast<unsigned short*>(s_at) + b + ((start + i) & 3u), (unsigned short)0,
                              (unsigned short)(at + 1u)) == 0)
                    return;
            b = (b + 4u) & mask;
        }
        ok = false;
    };
    const uint32_t* ids = list_of(from, lg_old, colours);
    const uint32_t* aux = aux_of(from, lg_old, colours);
    if (inter) {
        for (uint32_t h = rank; cnt_old && h < (1u << lg_old); h += width) {
            const uint32_t id = from[key_word(h, colours)];
            if (id != kEmptyId) place(id, h);
        }
    } else {
        for (uint32_t j = rank; j < cnt_old; j += width) place(ids[j], j);
    }
    __syncthreads();
    for (uint32_t b = rank; b < cap / 4u; b += width) {
        uint32_t id[4], t[4], cw[4];
        const uint2 at4 = reinterpret_cast<const uint2*>(s_at)[b];
#pragma unroll
        for (uint32_t i = 0; i < 4u; ++i) {
            const uint32_t at = ((i < 2u ? at4.x : at4.y) >> (16u * (i & 1u))) & 0xFFFFu;
            id[i] = kEmptyId;
            t[i] = cw[i] = 0u;
            if (at) {
                const uint32_t j = at - 1u;
                id[i] = inter ? from[key_word(j, colours)] : ids[j];
                t[i] = inter ? *eidx_of(from, j, lg_old, colours) : colours == kColMulti ? aux[2u * j] : aux[j];
                if (colours == kColMulti) cw[i] = aux[2u * j + 1u];
            }
        }
        uint4* out = reinterpret_cast<uint4*>(to);
        out[inter ? 2u * b : b] = make_uint4(id[0], id[1], id[2], id[3]);
        if (inter) {
            out[2u * b + 1u] = make_uint4(t[0], t[1], t[2], t[3]);
        } else if (colours == kColNone) {
            out[cap / 4u + b] = make_uint4(t[0], t[1], t[2], t[3]);
        } else {
            out[cap / 4u + 2u * b] = make_uint4(t[0], cw[0], t[1], cw[1]);
            out[cap / 4u + 2u * b + 1u] = make_uint4(t[2], cw[2], t[3], cw[3]);
        }
    }
    return ok;
}

// Move the blocks listed by k_commit whose new table has more than kMoveSlots slots: thread blocks
// claim pieces of the largest, then one node at a time, and build tables of at most kBlockMoveSlots slots in
// shared memory (`smem`: as many 16-bit words), larger ones in place.
__device__ __forceinline__ void k_rehash_huge_body(const StreamDev& d, const Grid g, uint32_t* smem) {
    __shared__ unsigned long long s_k;
    __shared__ int s_bad;
    const unsigned long long pieces = n_giants(d) * kGiantPieces;
    const unsigned long long n_work = pieces + d.ctrl->n_huge, top = d.ctrl->pool_top;
    for (;;) {
        if (threadIdx.x == 0) {
            s_k = atomicAdd(&d.ctrl->huge_next, 1ull);
            s_bad = 0;
        }
        __syncthreads();
        const unsigned long long k = s_k;
        if (k >= n_work) break;
        const uint32_t giant = (uint32_t)(k / kGiantPieces);
        const Move mv = move_of(d, k < pieces ? d.glist[giant] : d.big[d.big_cap - 1 - (k - pieces)], top);
        bool ok = true;
        if (mv.fits && k < pieces) {  // (uniform over the block)
            ok = move_block(mv.to, mv.from, mv.cnt_old, mv.lg_new, d.colours,
                            (uint32_t)(k % kGiantPieces) * blockDim.x + threadIdx.x, kGiantPieces * blockDim.x);
        } else if (mv.fits && (1u << mv.lg_new) <= kBlockMoveSlots) {
            ok = move_block_index(mv.to, mv.from, mv.cnt_old, mv.lg_new, d.colours, reinterpret_cast<uint16_t*>(smem));
        } else if (mv.fits) {  // built in place: empty keys first
            init_table_keys(mv.to, mv.lg_new, d.colours, threadIdx.x, blockDim.x);
            __syncthreads();
            ok = move_block(mv.to, mv.from, mv.cnt_old, mv.lg_new, d.colours, threadIdx.x, blockDim.x);
        }
        if (!ok) s_bad = 1;
        __syncthreads();
        if (threadIdx.x == 0) {
            if (s_bad) atomicOr(&d.ctrl->status, kStInternal);
            // the record changes when every piece has read it
            if (k >= pieces || atomicAdd(&d.order[giant], 1u) == kGiantPieces - 1u)
                d.meta[mv.x] = make_uint4(mv.off_new, mv.cnt_new, 0u, 0u);
        }
        __syncthreads();
    }
}

__device__ __forceinline__ void k_insert_body(const StreamDev& d, const BatchDev& b, const Grid g) {
    Ctrl* ct = d.ctrl;
    const bool failed = block_failed(ct);
    if (g.bx == 0 && threadIdx.x == 0) {
        // the batch's table space is now in use; reset the per-batch counters
        if (!failed) ct->pool_top += ct->need_quads;
        ct->need_quads = 0;
        ct->n_touched = 0;
        ct->n_big = 0;
        ct->n_huge = 0;
        ct->n_giant = 0;
        ct->huge_next = 0;
    }
    if (failed) return;
    __shared__ BlockReserve<uint32_t> part[2];
    uint32_t turn = 0;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned long long stride = (unsigned long long)g.nbx * blockDim.x;
    unsigned long long n_loops = 0, n_kept = 0;  // this lane's tallies, added once per warp at the end
    for (unsigned long long base = (unsigned long long)g.bx * blockDim.x; base < b.n; base += stride) {
        const unsigned long long e = base + threadIdx.x;
        const bool valid = e < b.n;
        uint32_t u = 0, v = 0;
        if (valid) { u = b.src[e]; v = b.dst[e]; }
        const bool loop = valid && u == v;
        // with stored colours the edge's colours decide whether it is kept and ride with its entries (in
        // the list entries' top bits or in a word per entry): the same hashes serve both
        uint32_t cj = 0u, cw = 0u;
        bool kept;
        if (d.colours == kColInEntry) {
            uint32_t i;
            const uint32_t j = colour_of(u, v, d.seed, d.fm);
            kept = processor_of(d, 0u, j, i);
            cj = j << kIdBits;
        } else if (d.colours != kColNone) {
            cw = colour_word(d, u, v, kept);
        } else {
            kept = kept_by_any(d, u, v);
        }
        kept = kept && valid && u != v;
        uint32_t mark = kNoWork;
        bool lead = false;  // the first grouped edge seen with its larger endpoint
        if (valid && u != v) {
            // list positions: the batch's new entries of a node fill its list from the end.  The two
            // records, then the first CAS of each table insert are issued before any result is used, so
            // that their round trips overlap.
            const uint2 rank = kept ? edge_ranks(d)[e] : make_uint2(0u, 0u);
            const uint4 mu = d.meta[u], mv = d.meta[v];
            if (kept && block_fits(d, 1, mu.x, table_lg(mu.y)) && block_fits(d, 1, mv.x, table_lg(mv.y))) {
                const uint32_t t = (uint32_t)(b.t0 + e);
                const uint32_t lu = table_lg(mu.y), lv = table_lg(mv.y);
                uint32_t *tu = block_at(d.pool, mu.x), *tv = block_at(d.pool, mv.x);
                const uint32_t col = d.colours;
                // the home buckets are read before the compare-and-swaps: a bucket that is not in L2 is
                // then fetched by a load, of which many more can be waiting than atomics (R-MAT scale 20,
                // 15.7M edges: 3.2 ms without, 2.5 ms with)
                const uint32_t bu = home_slot(v, lu), bv = home_slot(u, lv);
                const uint4 qu = __ldcg(reinterpret_cast<const uint4*>(tu) + key_quad(bu, col)),
                            qv = __ldcg(reinterpret_cast<const uint4*>(tv) + key_quad(bv, col));
                const uint32_t hu = bu + empty_slot(qu, v), hv = bv + empty_slot(qv, u);
                const uint32_t cu = atomicCAS(tu + key_word(hu, col), kEmptyId, v);
                const uint32_t cv = atomicCAS(tv + key_word(hv, col), kEmptyId, u);
                bool ok = true;
                if (cu == kEmptyId) table_store(tu, lu, hu, t, cw, col);
                else ok = table_insert(tu, lu, v, t, cw, col);
                if (cv == kEmptyId) table_store(tv, lv, hv, t, cw, col);
                else ok &= table_insert(tv, lv, u, t, cw, col);
                if (!ok) atomicOr(&ct->status, kStInternal);
                const uint32_t pu = mu.y - 1u - rank.x, pv = mv.y - 1u - rank.y;
                if (REPT_CHECK(ct, 2, pu, list_slots(lu)) && REPT_CHECK(ct, 2, pv, list_slots(lv))) {
                    list_of(tu, lu, col)[pu] = v | cj;
                    list_of(tv, lv, col)[pv] = u | cj;
                    if (col == kColWords) {
                        cw_of(tu, lu)[pu] = cw;
                        cw_of(tv, lv)[pv] = cw;
                    } else if (col == kColNone) {
                        aux_of(tu, lu, col)[pu] = t;
                        aux_of(tv, lv, col)[pv] = t;
                    } else if (col == kColMulti) {
                        reinterpret_cast<uint2*>(aux_of(tu, lu, col))[pu] = make_uint2(t, cw);
                        reinterpret_cast<uint2*>(aux_of(tv, lv, col))[pv] = make_uint2(t, cw);
                    }
                }
                if (d.edge_ends) d.edge_ends[t] = make_uint2(u, v);
            }
            // an edge can close wedges only if both endpoints have stored edges
            if (mu.y != 0u && mv.y != 0u) {
                const bool u_small = mu.y <= mv.y;
                const uint4 ms = u_small ? mu : mv, ml = u_small ? mv : mu;
                WorkItem it;
                it.s = u_small ? u : v;
                it.l = u_small ? v : u;
                it.off_s = ms.x;
                it.off_l = ml.x;
                it.t = (uint32_t)(b.t0 + e);
                it.lgs = table_lg(ms.y) | (table_lg(ml.y) << 8);
                it.cnt_s = ms.y;
                it.cnt_l = ml.y;
                d.rec[e] = it;
                mark = kSmallEdge;
                if (ms.y > b.small_max) {
                    mark = it.l;
                    lead = atomicAdd(&d.meta[it.l].w, 1u) == 0u;
                }
            }
        }
        if (valid) d.mark[e] = mark;
        const unsigned long long o = block_reserve(part[turn], &ct->n_groups, lead ? 1u : 0u);
        if (lead) d.glist[o] = mark;
        turn ^= 1u;
        n_loops += loop ? 1ull : 0ull;
        n_kept += kept ? 1ull : 0ull;
    }
    for (int o = 16; o > 0; o >>= 1) {
        n_loops += __shfl_down_sync(0xFFFFFFFFu, n_loops, o);
        n_kept += __shfl_down_sync(0xFFFFFFFFu, n_kept, o);
    }
    if (lane == 0) {
        if (n_loops) atomicAdd(&ct->self_loops, n_loops);
        if (n_kept) atomicAdd(&ct->stored, n_kept);
    }
}

// Place the grouped edges: every larger endpoint l gets a run of order[] for its edges (its record's
// cursor starts there), cut into units.  Runs and units are handed out in no particular order.
__device__ __forceinline__ void k_units_body(const StreamDev& d, const BatchDev& b, const Grid g) {
    Ctrl* ct = d.ctrl;
    if (ct->status) return;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned long long n_g = ct->n_groups;
    const unsigned long long stride = (unsigned long long)g.nbx * blockDim.x;
    for (unsigned long long base = (unsigned long long)g.bx * blockDim.x + threadIdx.x - lane; base < n_g;
         base += stride) {
        const unsigned long long i = base + lane;
        uint32_t l = 0, count = 0;
        uint32_t per = 1;
        int kind = kBinWarp;
        if (i < n_g) {
            l = d.glist[i];
            const uint4 m = d.meta[l];
            count = m.w;
            kind = m.y > kBigUnitNodes ? kBinBig : m.y > kWarpUnitNodes ? kBinBlock : kBinWarp;
            // (an edge's smaller list is no longer than the larger: at most kWarpUnitEntries per warp unit)
            per = kind == kBinWarp ? min(max(kWarpUnitEntries / m.y, 1u), kWarpUnitItems) : b.unit_edges;
        }
        const uint32_t first = (uint32_t)warp_reserve(&ct->n_items, count);
        if (i < n_g) d.meta[l].w = first;
        const uint32_t n_u = (count + per - 1u) / per;
        const unsigned long long uw = warp_reserve(&ct->bin_count[kBinWarp], kind == kBinWarp ? n_u : 0u);
        unsigned long long at = d.unit_cap - 1ull - uw;
        if (__any_sync(0xFFFFFFFFu, kind != kBinWarp)) {
            const unsigned long long ub = warp_reserve(&ct->bin_count[kBinBlock], kind == kBinBlock ? n_u : 0u);
            const unsigned long long ug = warp_reserve(&ct->bin_count[kBinBig], kind == kBinBig ? n_u : 0u);
            if (kind == kBinBlock) at = d.unit_cap + ub;
            else if (kind == kBinBig) at = ug;
        }
        for (uint32_t k = 0; k < n_u; ++k) {
            if (!REPT_CHECK(ct, 15, at, 2ull * d.unit_cap)) break;
            d.units[at] = Unit{first + k * per, min(per, count - k * per)};
            at += kind == kBinWarp ? -1ll : 1ll;
        }
    }
}

// Write each grouped edge to its place in order[].
__device__ __forceinline__ void k_order_body(const StreamDev& d, const BatchDev& b, const Grid g) {
    if (d.ctrl->status) return;
    const unsigned long long stride = (unsigned long long)g.nbx * blockDim.x;
    for (unsigned long long e = (unsigned long long)g.bx * blockDim.x + threadIdx.x; e < b.n; e += stride) {
        const uint32_t l = d.mark[e];
        if (l >= kSmallEdge) continue;
        const uint32_t pos = atomicAdd(&d.meta[l].w, 1u);
        if (REPT_CHECK(d.ctrl, 16, pos, d.unit_cap)) d.order[pos] = (uint32_t)e;
    }
}

// Look neighbour w up in the table of 2^lg slots at `table` (lg >= 2): read 4-key buckets from w's
// home bucket on until w or an empty key shows up.  Returns w's slot, or kEmptyId when w is absent;
// `slots` receives the number of keys read.
__device__ __forceinline__ uint32_t table_slot(const uint32_t* table, uint32_t lg, uint32_t w,
                                               uint32_t& slots, uint32_t colours) {
    const uint32_t mask = (1u << lg) - 1u;
    const uint4* buckets = reinterpret_cast<const uint4*>(table);
    uint32_t h = home_slot(w, lg);
    for (uint32_t probe = 0; probe <= mask; probe += 4u) {  // h: the first slot of a bucket
        const uint4 k4 = buckets[key_quad(h, colours)];
        slots = probe + 4u;
        if (k4.x == w) return h;
        if (k4.y == w) return h + 1u;
        if (k4.z == w) return h + 2u;
        if (k4.w == w) return h + 3u;
        if (k4.x == kEmptyId || k4.y == kEmptyId || k4.z == kEmptyId || k4.w == kEmptyId) return kEmptyId;
        h = (h + 4u) & mask;
    }
    return kEmptyId;
}

// w's stream index in that table, or kEmptyId.
__device__ __forceinline__ uint32_t table_find(const uint32_t* table, uint32_t lg, uint32_t w,
                                               uint32_t& slots, uint32_t colours) {
    const uint32_t h = table_slot(table, lg, w, slots, colours);
    return h == kEmptyId ? kEmptyId : *eidx_of(table, h, lg, colours);
}

// REPT_FLAG_CHECK_DUPS: before the batch is applied, flag an edge that repeats an earlier stored
// edge (found in its endpoint's table) or another edge of the same batch (found in a set of the
// batch's edge keys, built in the work-record scratch, which is free at this point and was filled
// with ~0 by the host).  `mask` + 1 is the set's capacity, a power of two at least twice the batch.
__global__ void k_check_dups(StreamDev d, BatchDev b, unsigned long long mask) {
    if (d.ctrl->status) return;
    unsigned long long* set = reinterpret_cast<unsigned long long*>(d.rec);
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    bool dup = false;
    for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < b.n; e += stride) {
        const uint32_t u = b.src[e], v = b.dst[e];
        if (u == v || u >= d.n_nodes || v >= d.n_nodes) continue;
        const uint4 mu = d.meta[u];
        uint32_t ns;
        if (mu.y != 0u && table_find(block_at(d.pool, mu.x), table_lg(mu.y), v, ns, d.colours) != kEmptyId) dup = true;
        const unsigned long long key = ((unsigned long long)(u < v ? u : v) << 32) | (u < v ? v : u);
        unsigned long long h = splitmix64(key) & mask;
        for (unsigned long long probe = 0; probe <= mask; ++probe) {
            const unsigned long long old = atomicCAS(set + h, ~0ull, key);
            if (old == ~0ull) break;
            if (old == key) { dup = true; break; }
            h = (h + 1u) & mask;
        }
    }
    if (dup) atomicOr(&d.ctrl->status, kStDuplicate);
}

// Work counters of k_intersect<true>, kept per lane in registers.
struct Work {
    unsigned long long entries = 0, slots = 0, probes = 0, pslots = 0, wedges = 0, counted = 0;
};

// Wedge (s, w), (l, w), both edges older than the arriving edge (s, l): count it for every hash group
// whose colour of the two edges agrees and names a kept processor, and add the number of such groups
// to tau_s, tau_l and tau_w (Algorithm 1's local updates, one wedge at a time).
// Algorithm 2's pair counters: one more closed wedge through stored edge t in group k this batch.
__device__ __forceinline__ void pair_event(const StreamDev& d, uint32_t t, uint32_t k) {
    const unsigned long long idx = (unsigned long long)t * d.groups + k;
    if (atomicAdd(&d.pair_evt[idx], 1u) == 0u) d.pair_list[atomicAdd(&d.ctrl->n_pairs, 1ull)] = (uint32_t)idx;
}

// kColAny: the colour storage is read from each stream's descriptor (groups).
constexpr int kColAny = 8;
template <int MODE>
__device__ __forceinline__ uint32_t colours_of(const StreamDev& d) {
    return MODE == kColAny ? d.colours : (uint32_t)MODE;
}

// Where closed wedges are tallied: a single stream's blocks keep tau^(i) in shared memory, as a low and a
// high 32-bit half (processor i: words 2i, 2i + 1; 64-bit shared atomics are compare-and-swap loops); a
// group's go straight to global memory (half == nullptr).
__device__ __forceinline__ void tally(const StreamDev& d, uint32_t* half, uint32_t i) {
    if (half == nullptr) atomicAdd(&d.proc[i], 1ull);
    else if (atomicAdd(&half[2u * i], 1u) == 0xFFFFFFFFu) atomicAdd(&half[2u * i + 1u], 1u);
}

// Processor i counted the wedge (s, w), (l, w): its own tau_v^(i), when kept.
__device__ __forceinline__ void count_local_proc(const StreamDev& d, uint32_t i, uint32_t s, uint32_t l, uint32_t w) {
    unsigned long long* lp = d.local_proc + (unsigned long long)i * d.n_nodes;
    atomicAdd(&lp[s], 1ull);
    atomicAdd(&lp[l], 1ull);
    atomicAdd(&lp[w], 1ull);
}

// `found` groups counted it for the local sums, `found2` for Algorithm 2's partial group.
__device__ __forceinline__ void count_locals(const StreamDev& d, uint32_t found, uint32_t found2, uint32_t s, uint32_t l,
                                             uint32_t w) {
    if (found) {
        atomicAdd(&d.local[w], (unsigned long long)found);
        atomicAdd(&d.local[s], (unsigned long long)found);
        atomicAdd(&d.local[l], (unsigned long long)found);
    }
    if (found2) {
        atomicAdd(&d.local2[w], (unsigned long long)found2);
        atomicAdd(&d.local2[s], (unsigned long long)found2);
        atomicAdd(&d.local2[l], (unsigned long long)found2);
    }
}

// The wedge's colours from the hashes.  Single-group streams with colours in their entries form both
// colours, which keeps registers low; the others decide each group's agreement from the two hash values'
// difference (same_colour: one remainder only when they agree).
template <int MODE>
__device__ __forceinline__ uint32_t count_wedge(const StreamDev& d, uint32_t* half, uint32_t s, uint32_t l, uint32_t w) {
    if (!REPT_CHECK(d.ctrl, 9, max(w, max(s, l)), d.n_nodes)) return 0u;
    uint32_t found = 0, found2 = 0;
    uint32_t t_sw = kEmptyId, t_lw = kEmptyId;
    for (uint32_t k = d.kbeg; k < d.kend; ++k) {
        uint32_t js, i;
        bool agree;
        if (MODE != (int)kColInEntry) {
            agree = same_colour(s, l, w, group_seed(d.seed, k), d.fm, js) && processor_of(d, k, js, i);
        } else {
            const uint64_t sk = group_seed(d.seed, k);
            js = colour_of(s, w, sk, d.fm);
            agree = processor_of(d, k, js, i) && colour_of(l, w, sk, d.fm) == js;
        }
        if (agree) {
            tally(d, half, i);
            if (d.local2 && k >= d.c1) ++found2; else ++found;
            if (d.local_proc) count_local_proc(d, i, s, l, w);
            if (d.pair_tau) {
                if (t_sw == kEmptyId) {  // the wedge's two stream indices, looked up once
                    uint32_t ns;
                    const uint4 ms = d.meta[s], ml = d.meta[l];
                    t_sw = table_find(block_at(d.pool, ms.x), table_lg(ms.y), w, ns, kColNone);
                    t_lw = table_find(block_at(d.pool, ml.x), table_lg(ml.y), w, ns, kColNone);
                }
                pair_event(d, t_sw, k);
                pair_event(d, t_lw, k);
            }
        }
    }
    count_locals(d, found, found2, s, l, w);
    return found + found2;
}

// The groups in which two edges with the stored colour words cs, cl (kColMulti) have the same colour: bit
// (k + 1) cbits - 1 for group k, found for all groups at once (a field of cs ^ cl is zero); where a group
// keeps one colour only, the groups that keep both edges.
__device__ __forceinline__ uint32_t agreeing_groups(const StreamDev& d, uint32_t cs, uint32_t cl) {
    if (d.keep == 1u) return cs & cl;
    const uint32_t x = cs ^ cl, low = ~d.ctop;
    return ~(((x & low) + low) | x) & d.ctop;
}

// Count the wedge (s, w), (l, w) in those groups, where a processor keeps the colour (cs, of {s, w}).
__device__ __forceinline__ uint32_t count_groups(const StreamDev& d, uint32_t* half, uint32_t s, uint32_t l, uint32_t w,
                                                 uint32_t groups, uint32_t cs) {
    if (!REPT_CHECK(d.ctrl, 9, max(w, max(s, l)), d.n_nodes)) return 0u;
    uint32_t found = 0, found2 = 0;
    uint32_t t_sw = kEmptyId, t_lw = kEmptyId;
    for (; groups; groups &= groups - 1u) {
        const uint32_t top = (uint32_t)__ffs((int)groups), k = top / d.cbits - 1u;
        uint32_t i;
        const uint32_t js = d.keep == 1u ? 0u : (cs >> (top - d.cbits)) & d.cmask;
        if (!processor_of(d, k, js, i)) continue;
        tally(d, half, i);
        if (d.local2 && k >= d.c1) ++found2; else ++found;
        if (d.local_proc) count_local_proc(d, i, s, l, w);
        if (d.pair_tau) {
            if (t_sw == kEmptyId) {  // the wedge's two stream indices, looked up once
                uint32_t ns;
                const uint4 ms = d.meta[s], ml = d.meta[l];
                t_sw = table_find(block_at(d.pool, ms.x), table_lg(ms.y), w, ns, kColMulti);
                t_lw = table_find(block_at(d.pool, ml.x), table_lg(ml.y), w, ns, kColMulti);
            }
            pair_event(d, t_sw, k);
            pair_event(d, t_lw, k);
        }
    }
    count_locals(d, found, found2, s, l, w);
    return found + found2;
}

// ---------------------------------------------------------------------------------------------
// The intersection.  An edge t = (s, l) closes the wedges {s, w}, {l, w} of entries w that both lists
// hold.  Few entries of s's list do (with the same colour in both, about 0.1 % on the R-MAT streams), so
// the work is to reject the others cheaply.  A filter of l's list is built in shared memory -- a Bloom
// filter of two bits per entry, both in one 32-bit word, keyed by the entry's id and stored colour --
// and the lists of l's grouped edges are scanned against it: nine instructions and one shared-memory
// read per entry, where hashing the larger endpoint's edge for its colour takes 58.  Grouping by l makes
// one filter serve all edges of l (R-MAT scale 20, late batches: 14 to 26 times as many entries are
// scanned as inserted).  Entries that pass (0.6 % there; with several groups the common neighbours, 14 %
// on the 4M-node stream) join the warp's candidate queue and are looked up in l's table, which decides
// exactly.  R-MAT scale 20, m = c = 100: 8.83 ms per stream with a hash per entry, 5.51 ms so; the 4M-node
// stream with five groups: 157 ms with a probe per entry, 114 ms so, of which the scans alone are 18 ms.
// What bounds it: instruction issue (57 % of the slots) in the scans, the latency of the candidates'
// dependent loads where many pass.

constexpr int kIxThreads = 256;
// Blocks per SM.  Shared memory of a block (ix_words): one stream 45 KB, 48 without stored colours, 54 with the
// words of several groups, and 8 bytes per processor, of which four fit up to about 200 processors; a group's
// kernels 51 KB, 54 and 60 (also for mixed layouts), of which the last fit three times.
constexpr int kIxBlocks = 4;
constexpr uint32_t kIxWarps = kIxThreads / 32;
constexpr uint32_t kFilterLg = 13;  // words of a block's filter (32 KB); a warp's share serves warp units
constexpr uint32_t kFilterWords = 1u << kFilterLg;
constexpr uint32_t kWarpFilterLg = 10;
static_assert(kIxWarps << kWarpFilterLg <= kFilterWords, "warp filters share the block's");
static_assert(kUnitItems == 64, "two records per lane of the first warp");

// A warp's two queues, arrays of kCandQ and kMatchQ words.  Candidates: the neighbour of an entry of the
// smaller endpoint's list that passed a filter or colour test (queued as scanned, so that the probe need not
// read the list again before it can form its address: five groups, 4M nodes, 122 to 114 ms), its edge, its
// position in the list (where the stream index stands beside the list) and, for groups, the stream.  Closed wedges:
// the neighbour, the edge, the agreeing groups and the colour word (kColMulti) and, for groups, the
// stream; they are counted
// 32 at a time so that the work runs on full warps.
struct WarpQueues {
    uint32_t* base;      // candidates, then closed wedges
    uint32_t n, closed;  // how many of each are waiting (warp-uniform)
};
constexpr uint32_t kCandQ = 96, kMatchQ = 96;  // 63 + 32 candidates; 31 + 2 x 32 wedges
// Arrays of closed wedges before the streams'.
constexpr uint32_t match_arrays(int mode) { return mode == (int)kColMulti || mode == kColAny ? 4u : 2u; }
// Arrays of candidates before the streams'.
constexpr uint32_t cand_arrays(int mode) { return mode == (int)kColInEntry || mode == (int)kColWords ? 2u : 3u; }
constexpr uint32_t queue_words(int mode, bool group) {
    return (cand_arrays(mode) + (group ? 1u : 0u)) * kCandQ + (match_arrays(mode) + (group ? 1u : 0u)) * kMatchQ;
}

// Shared memory of one intersection block, in words: the filter, the records of the unit's edges and the
// warps' queues.
constexpr uint32_t ix_words(int mode, bool group) {
    return kFilterWords + 4u * kUnitItems + kIxWarps * queue_words(mode, group);
}

// The streams an intersection works on: one, passed by value to the kernel, with its block's counters
// (tally), or a group's array.
struct OneStream {
    static constexpr bool kGroup = false;
    const StreamDev& d;
    uint32_t* half;
    __device__ __forceinline__ const StreamDev& at(uint32_t) const { return d; }
};
struct ManyStreams {
    static constexpr bool kGroup = true;
    const StreamDev* __restrict__ ds;
    static constexpr uint32_t* half = nullptr;
    __device__ __forceinline__ const StreamDev& at(uint32_t sid) const { return ds[sid]; }
};

// Count `take` closed wedges from the end of the queue (n waiting).
template <bool WORK, int MODE, class S>
__device__ __forceinline__ void count_closed(const S& st, const uint32_t* mq, uint32_t n, uint32_t take, Work& wk) {
    constexpr bool GROUP = S::kGroup;
    const unsigned lane = threadIdx.x & 31u;
    if (lane < take) {
        const uint32_t i = n - take + lane, w = mq[i];
        const StreamDev& d = st.at(GROUP ? mq[match_arrays(MODE) * kMatchQ + i] : 0u);
        const uint2 sl = *reinterpret_cast<const uint2*>(d.rec + mq[kMatchQ + i]);
        uint32_t f = 0;
        if (match_arrays(MODE) == 4u && colours_of<MODE>(d) == kColMulti)
            f = count_groups(d, st.half, sl.x, sl.y, w, mq[2u * kMatchQ + i], mq[3u * kMatchQ + i]);
        else
            f = count_wedge<MODE>(d, st.half, sl.x, sl.y, w);
        if (WORK) wk.counted += f;
    }
    __syncwarp();
}

// Probe candidates 0 .. take - 1 (take <= 64) of the queue at `cq`, two per lane.  A hit whose two edges are
// older than the candidate's edge is a closed wedge.  `closed` wedges were waiting; returns how many
// are now (`all`: none, everything is counted).
template <bool WORK, int MODE, class S>
__device__ __forceinline__ uint32_t cand_probe(const S& st, const uint32_t* cq, uint32_t* mq, uint32_t take,
                                               uint32_t closed, bool all, Work& wk) {
    constexpr bool GROUP = S::kGroup;
    const unsigned lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    if (take) {
        // every stage loads for both candidates before either is used; lanes past the end repeat the last one
        uint32_t item[2], sd[2], pos[2], w[2], h[2], lgs[2], lgl[2], t[2], slot[2];
        uint2 off[2];  // blocks of the smaller and the larger endpoint
        uint4 bk[2];
        uint2 as[2], al[2];  // stream index and colour word of the smaller and the larger side's entry
        bool v[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const uint32_t k = min(32u * p + lane, take - 1u);
            v[p] = 32u * p + lane < take;
            w[p] = cq[k];
            item[p] = cq[kCandQ + k];
            pos[p] = cand_arrays(MODE) == 3u ? cq[2u * kCandQ + k] : 0u;
            sd[p] = GROUP ? cq[cand_arrays(MODE) * kCandQ + k] : 0u;
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {  // WorkItem: {s, l, off_s, off_l}, {t, lgs, cnt_s, cnt_l}
            const uint2* rec = reinterpret_cast<const uint2*>(st.at(sd[p]).rec + item[p]);
            off[p] = rec[1];
            const uint2 r = rec[2];
            t[p] = r.x;
            lgs[p] = r.y & 0xFFu;
            lgl[p] = r.y >> 8;
            if (WORK) {
                const uint32_t cls = v[p] ? (uint32_t)bin_of_cnt(rec[3].x) : 6u;
                for (uint32_t c = 0; c < 6u; ++c) {
                    const unsigned of = __ballot_sync(0xFFFFFFFFu, cls == c);
                    if (of && lane == 0) atomicAdd(&st.at(0u).ctrl->class_probes[c], (unsigned long long)__popc(of));
                }
            }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const StreamDev& d = st.at(sd[p]);
            const uint32_t col = colours_of<MODE>(d);
            as[p] = make_uint2(0u, 0u);
            bk[p] = make_uint4(kEmptyId, kEmptyId, kEmptyId, kEmptyId);
            h[p] = 0u;
            if (block_fits(d, 5, off[p].x, lgs[p]) && block_fits(d, 7, off[p].y, lgl[p]) &&
                REPT_CHECK(d.ctrl, 3, pos[p], list_slots(lgs[p]))) {
                h[p] = home_slot(w[p], lgl[p]);
                // (a plain load: this kernel may be set up while the inserts still write the pool, and a group's
                // persistent launch writes it itself, so the read-only path is not open to it)
                bk[p] = reinterpret_cast<const uint4*>(block_at(d.pool, off[p].y))[key_quad(h[p], col)];
                const uint32_t* aux_s = aux_of(block_at(d.pool, off[p].x), lgs[p], col);
                if (col == kColNone) as[p].x = aux_s[pos[p]];
                if (col == kColMulti) as[p] = reinterpret_cast<const uint2*>(aux_s)[pos[p]];
            } else {
                v[p] = false;
            }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const uint4 b = bk[p];
            slot[p] = b.x == w[p] ? h[p] : b.y == w[p] ? h[p] + 1u : b.z == w[p] ? h[p] + 2u : b.w == w[p] ? h[p] + 3u : kEmptyId;
            uint32_t ns = 4u;
            if (v[p] && slot[p] == kEmptyId && b.x != kEmptyId && b.y != kEmptyId && b.z != kEmptyId && b.w != kEmptyId) {
                const StreamDev& d = st.at(sd[p]);  // rare: the home bucket is full
                slot[p] = table_slot(block_at(d.pool, off[p].y), lgl[p], w[p], ns, colours_of<MODE>(d));
            }
            if (!v[p]) slot[p] = kEmptyId;
            if (WORK && v[p]) { ++wk.probes; wk.pslots += ns; }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const StreamDev& d = st.at(sd[p]);
            const uint32_t col = colours_of<MODE>(d);
            al[p] = make_uint2(kEmptyId, 0u);  // absent: never older
            if (slot[p] != kEmptyId) {
                const uint32_t* a = eidx_of(block_at(d.pool, off[p].y), slot[p], lgl[p], col);
                if (col == kColMulti) al[p] = *reinterpret_cast<const uint2*>(a);
                else al[p].x = *a;
            }
        }
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const StreamDev& d = st.at(sd[p]);
            const uint32_t col = colours_of<MODE>(d);
            bool has = al[p].x < t[p];
            if (interleaved(col) && has) {
                uint32_t ns;
                as[p].x = table_find(block_at(d.pool, off[p].x), lgs[p], w[p], ns, col);
            }
            has = has && as[p].x < t[p];
            if (WORK && has) ++wk.wedges;
            uint32_t groups = 0;
            if (col == kColMulti) {
                groups = agreeing_groups(d, as[p].y, al[p].y);
                has = has && groups != 0u;
            }
            const unsigned m = __ballot_sync(0xFFFFFFFFu, has);
            if (m && REPT_CHECK(st.at(0u).ctrl, 13, closed + __popc(m), (unsigned long long)kMatchQ + 1ull)) {
                if (has) {
                    const uint32_t k = closed + __popc(m & below);
                    mq[k] = w[p];
                    mq[kMatchQ + k] = item[p];
                    if (match_arrays(MODE) == 4u) {
                        mq[2u * kMatchQ + k] = groups;
                        mq[3u * kMatchQ + k] = as[p].y;
                    }
                    if (GROUP) mq[match_arrays(MODE) * kMatchQ + k] = sd[p];
                }
                closed += __popc(m);
            }
        }
        __syncwarp();
    }
#pragma unroll 1
    while (closed >= 32u || (all && closed)) {
        const uint32_t n = min(closed, 32u);
        count_closed<WORK, MODE>(st, mq, closed, n, wk);
        closed -= n;
    }
    return closed;
}

// Probe the first 64 candidates (fewer when `all`, which also counts every closed wedge) and move the
// rest to the front.
template <bool WORK, int MODE, class S>
__device__ __forceinline__ void cand_flush(const S& st, WarpQueues& q, Work& wk, bool all) {
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t take = min(q.n, 64u), rest = q.n - take;
    __syncwarp();
    q.closed = cand_probe<WORK, MODE>(st, q.base, q.base + (cand_arrays(MODE) + (S::kGroup ? 1u : 0u)) * kCandQ, take, q.closed, all, wk);
    if (lane < rest) {  // rest < 32
#pragma unroll
        for (uint32_t a = 0; a < cand_arrays(MODE) + (S::kGroup ? 1u : 0u); ++a) q.base[a * kCandQ + lane] = q.base[a * kCandQ + 64u + lane];
    }
    q.n = rest;
    __syncwarp();
}

// Filter hash of a list entry: `word` holds its id and, with kColInEntry, its colour; `cw` its colour
// word with kColWords.  Equal entries hash alike; the filter only needs that.
template <int MODE>
__device__ __forceinline__ uint32_t filter_hash(uint32_t word, uint32_t cw) {
    return (MODE == (int)kColWords || MODE == kColAny ? word + cw * 0x85EBCA6Bu : word) * 0x9E3779B1u;
}
// The product's top bits choose the word, its low bits and some from the middle the two bits.
__device__ __forceinline__ void filter_set(uint32_t* filter, uint32_t lg, uint32_t h) {
    atomicOr(filter + (h >> (32u - lg)), (1u << (h & 31u)) | (1u << ((h >> 9) & 31u)));
}
// 1 if both bits are set, else 0.
__device__ __forceinline__ uint32_t filter_test(const uint32_t* filter, uint32_t lg, uint32_t h) {
    const uint32_t v = filter[h >> (32u - lg)];
    return __funnelshift_r(v, v, h) & __funnelshift_r(v, v, h >> 9) & 1u;
}
// log2 of the filter words for n entries: one word (32 bits) per entry, at least 32 words.
__device__ __forceinline__ uint32_t filter_lg(uint32_t n, uint32_t max_lg) {
    const uint32_t lg = n <= 32u ? 5u : 32u - __clz(n - 1u);
    return lg < max_lg ? lg : max_lg;
}

// Clear the filter; lanes `rank` of `width`.
__device__ __forceinline__ void filter_clear(uint32_t* filter, uint32_t lg, uint32_t rank, uint32_t width) {
    for (uint32_t i = rank; i < (1u << lg) / 4u; i += width)
        reinterpret_cast<uint4*>(filter)[i] = make_uint4(0u, 0u, 0u, 0u);
}

// Set the n entries of the block at off_quads in the (cleared) filter; lanes `rank` of `width`.
template <int MODE>
__device__ __forceinline__ void filter_build(const StreamDev& d, uint32_t* filter, uint32_t lg, uint32_t off, uint32_t n,
                                             uint32_t rank, uint32_t width) {
    const uint32_t lgt = table_lg(n), col = colours_of<MODE>(d);
    if (!(block_fits(d, 7, off, lgt) && REPT_CHECK(d.ctrl, 6, n, list_slots(lgt) + 1u))) return;
    const uint32_t* block = block_at(d.pool, off);
    const uint4* list = reinterpret_cast<const uint4*>(list_of(block, lgt, col));
    const uint4* words = reinterpret_cast<const uint4*>(cw_of(block, lgt));
    const uint32_t last = (n - 1u) >> 2;
    for (uint32_t i = rank; i <= last; i += 2u * width) {
        uint4 q[2], cw[2];
#pragma unroll
        for (uint32_t j = 0; j < 2u; ++j) {  // past the end: the last quad again (setting bits twice is harmless)
            const uint32_t at = min(i + j * width, last);
            q[j] = list[at];
            cw[j] = make_uint4(0u, 0u, 0u, 0u);
            if (col == kColWords) cw[j] = words[at];
        }
#pragma unroll
        for (uint32_t j = 0; j < 2u; ++j) {
            const uint32_t at = 4u * min(i + j * width, last);
            filter_set(filter, lg, filter_hash<MODE>(q[j].x, cw[j].x));
            if (at + 1u < n) filter_set(filter, lg, filter_hash<MODE>(q[j].y, cw[j].y));
            if (at + 2u < n) filter_set(filter, lg, filter_hash<MODE>(q[j].z, cw[j].z));
            if (at + 3u < n) filter_set(filter, lg, filter_hash<MODE>(q[j].w, cw[j].w));
        }
    }
}

// One step's passing entries join the warp's queue: bit b of a lane's m is the entry at position
// base + 128 (b / 4) + b % 4 of edge `item`'s list of n entries (positions past its end are repeats of its
// last quad); word(b) yields its list word.  One entry a lane at a time; a full round of 64 is probed.
template <bool WORK, int MODE, class S, class Word>
__device__ __forceinline__ void queue_step(const S& st, WarpQueues& wq, uint32_t m, uint32_t base, uint32_t n,
                                           uint32_t item, uint32_t sid, Work& wk, Word&& word) {
    while (__any_sync(0xFFFFFFFFu, m != 0u)) {
        const uint32_t b = (uint32_t)__ffs((int)m) - 1u;  // (unused where m is 0)
        const uint32_t at = base + ((b >> 2) << 7) + (b & 3u);
        const bool has = m != 0u && at < n;
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, has);
        m &= m - 1u;
        if (!S::kGroup && !REPT_CHECK(st.at(0u).ctrl, 13, wq.n + __popc(mask), (unsigned long long)kCandQ + 1ull)) return;
        if (has) {
            uint32_t* to = wq.base + wq.n + __popc(mask & ((1u << (threadIdx.x & 31u)) - 1u));
            to[0] = word(b) & id_mask(st.at(sid));
            to[kCandQ] = item;
            if (cand_arrays(MODE) == 3u) to[2u * kCandQ] = at;
            if (S::kGroup) to[cand_arrays(MODE) * kCandQ] = sid;
        }
        wq.n += __popc(mask);
        if (wq.n >= 64u) cand_flush<WORK, MODE>(st, wq, wk, false);
    }
}

// The four entries of a quad against the filter: bit i is set if entry i passes.
template <int MODE>
__device__ __forceinline__ uint32_t test_quad(const uint32_t* filter, uint32_t lg, const uint4& q, const uint4& cw) {
    return filter_test(filter, lg, filter_hash<MODE>(q.x, cw.x)) | (filter_test(filter, lg, filter_hash<MODE>(q.y, cw.y)) << 1) |
           (filter_test(filter, lg, filter_hash<MODE>(q.z, cw.z)) << 2) | (filter_test(filter, lg, filter_hash<MODE>(q.w, cw.w)) << 3);
}
// Word b % 4 of a quad.
__device__ __forceinline__ uint32_t quad_word(const uint4& q, uint32_t b) {
    return b & 2u ? (b & 1u ? q.w : q.z) : (b & 1u ? q.y : q.x);
}
// Scan rows j0 .. j1 - 1 (32 quads, one per lane) of a list of n entries: four rows per step.  A lane past
// the list's end reads its last quad again.
template <bool WORK, int MODE, class S>
__device__ __forceinline__ void scan_rows(const S& st, uint32_t sid, const uint32_t* filter, uint32_t lg, uint32_t off_s,
                                          uint32_t n, uint32_t item, uint32_t j0, uint32_t j1, WarpQueues& wq, Work& wk) {
    const StreamDev& d = st.at(sid);
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t col = colours_of<MODE>(d), lgs = table_lg(n), last = (n - 1u) >> 2;
    const bool has_cw = MODE == (int)kColWords || (MODE == kColAny && col == kColWords);
    const uint32_t* block = block_at(d.pool, off_s);
    const uint4* list = reinterpret_cast<const uint4*>(list_of(block, lgs, col));
    const uint4* words = reinterpret_cast<const uint4*>(cw_of(block, lgs));
#pragma unroll 1
    for (uint32_t j = j0; j < j1; j += 4u) {
        uint4 q[4], cw[4];
#pragma unroll
        for (uint32_t h = 0; h < 4u; ++h) {
            q[h] = cw[h] = make_uint4(0u, 0u, 0u, 0u);
            if (h == 0u || j + h < j1) {  // (uniform)
                const uint32_t at = min(32u * (j + h) + lane, last);
                q[h] = list[at];
                if (has_cw) cw[h] = words[at];
            }
        }
        uint32_t m = 0;
#pragma unroll
        for (uint32_t h = 0; h < 4u; ++h)
            if (h == 0u || j + h < j1) m |= test_quad<MODE>(filter, lg, q[h], cw[h]) << (4u * h);
        queue_step<WORK, MODE>(st, wq, m, 4u * (32u * j + lane), n, item, sid, wk, [&](uint32_t b) {
            const uint32_t w0 = quad_word(q[0], b), w1 = quad_word(q[1], b), w2 = quad_word(q[2], b), w3 = quad_word(q[3], b);
            return b & 8u ? (b & 4u ? w3 : w2) : (b & 4u ? w1 : w0);
        });
    }
}
// The four entries of a quad without a filter, for an edge whose larger endpoint is l: bit i is set if entry i's
// colour may agree with the hash of {l, entry i} (colour_may_match); without one group's stored colours every
// entry passes.
template <int MODE>
__device__ __forceinline__ uint32_t hash_quad(const StreamDev& d, uint32_t l, const uint4& q, const uint4& cw) {
    const uint32_t col = colours_of<MODE>(d), mask = id_mask(d);
    if (!interleaved(col)) return 15u;
    uint32_t m = 0;
#pragma unroll
    for (uint32_t i = 0; i < 4u; ++i) {
        const uint32_t w = quad_word(q, i);
        m |= (colour_may_match(d, l, w & mask, col == kColWords ? quad_word(cw, i) : w >> kIdBits) ? 1u : 0u) << i;
    }
    return m;
}
// ... and rows j0 .. j1 - 1 scanned so, one per step.
template <bool WORK, int MODE, class S>
__device__ __forceinline__ void hash_rows(const S& st, uint32_t sid, uint32_t l, uint32_t off_s, uint32_t n, uint32_t item,
                                          uint32_t j0, uint32_t j1, WarpQueues& wq, Work& wk) {
    const StreamDev& d = st.at(sid);
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t col = colours_of<MODE>(d), lgs = table_lg(n), last = (n - 1u) >> 2;
    const bool has_cw = MODE == (int)kColWords || (MODE == kColAny && col == kColWords);
    const uint32_t* block = block_at(d.pool, off_s);
    const uint4* list = reinterpret_cast<const uint4*>(list_of(block, lgs, col));
    const uint4* words = reinterpret_cast<const uint4*>(cw_of(block, lgs));
#pragma unroll 1
    for (uint32_t j = j0; j < j1; ++j) {
        const uint32_t at = min(32u * j + lane, last);
        const uint4 q = list[at], cw = has_cw ? words[at] : make_uint4(0u, 0u, 0u, 0u);
        queue_step<WORK, MODE>(st, wq, hash_quad<MODE>(d, l, q, cw), 4u * (32u * j + lane), n, item, sid, wk,
                               [&](uint32_t b) { return quad_word(q, b); });
    }
}
// Rows of a list of n entries.
__device__ __forceinline__ uint32_t list_rows(uint32_t n) { return (n + 127u) >> 7; }

// Shorter lists, one per lane (n entries of the block at off_s, edge e; n == 0: none): their quads are laid
// end to end and dealt to the lanes, two per lane and step, so that no lane idles at a list's end.
template <bool WORK, int MODE, class S>
__device__ __forceinline__ void scan_short(const S& st, uint32_t sid, const uint32_t* filter, uint32_t lg, uint32_t off_s,
                                           uint32_t n, uint32_t e, WarpQueues& wq, Work& wk) {
    const StreamDev& d = st.at(sid);
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t col = colours_of<MODE>(d), lgs = table_lg(n);
    const bool has_cw = MODE == (int)kColWords || (MODE == kColAny && col == kColWords);
    const uint32_t list_off = off_s + (((col == kColMulti ? 3u : 2u) << lgs) >> 3);  // in 32-byte units (n > 4: a whole number)
    const uint32_t quads = (n + 3u) >> 2;
    uint32_t incl = quads;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += y;
    }
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - quads;
#pragma unroll 1
    for (uint32_t f = 0; f < total; f += 64u) {
        uint4 q[2], cw[2];
        uint32_t own[2], pos[2], m[2];
#pragma unroll
        for (uint32_t p = 0; p < 2u; ++p) {
            const uint32_t at = min(f + 32u * p + lane, total - 1u);
            uint32_t o = 0;  // the lane whose quads cover position `at`: the first with incl > at
#pragma unroll
            for (uint32_t step = 16u; step; step >>= 1)
                if (__shfl_sync(0xFFFFFFFFu, incl, o + step - 1u) <= at) o += step;
            own[p] = o;
            pos[p] = at - __shfl_sync(0xFFFFFFFFu, excl, o);
            q[p] = reinterpret_cast<const uint4*>(block_at(d.pool, __shfl_sync(0xFFFFFFFFu, list_off, o)))[pos[p]];
            cw[p] = make_uint4(0u, 0u, 0u, 0u);
            if (has_cw) {
                const uint32_t oo = __shfl_sync(0xFFFFFFFFu, off_s, o), on = __shfl_sync(0xFFFFFFFFu, n, o);
                cw[p] = reinterpret_cast<const uint4*>(cw_of(block_at(d.pool, oo), table_lg(on)))[pos[p]];
            }
        }
#pragma unroll
        for (uint32_t p = 0; p < 2u; ++p) {
            m[p] = test_quad<MODE>(filter, lg, q[p], cw[p]);
            if (f + 32u * p + lane >= total) m[p] = 0u;
        }
        if (__any_sync(0xFFFFFFFFu, (m[0] | m[1]) != 0u)) {
#pragma unroll 1
            for (uint32_t p = 0; p < 2u; ++p) {
                const uint32_t mp = p ? m[1] : m[0], o = p ? own[1] : own[0], at = 4u * (p ? pos[1] : pos[0]);
                const uint32_t on = __shfl_sync(0xFFFFFFFFu, n, o), oe = __shfl_sync(0xFFFFFFFFu, e, o);
                const uint4 qp = p ? q[1] : q[0];
                queue_step<WORK, MODE>(st, wq, mp, at, on, oe, sid, wk, [&](uint32_t b) { return quad_word(qp, b); });
            }
        }
    }
}

// A block unit as its first thread claims it: the edges order[first .. first + count) of stream sid and
// the larger endpoint l's block (n entries at off).  Before the scan: whether l's filter pays.
struct UnitClaim {
    uint32_t ok, sid, first, count, off, n, l, filter;
};
__device__ __forceinline__ UnitClaim claimed_unit(const StreamDev& d, uint32_t sid, unsigned long long at) {
    const Unit u = d.units[at];
    const WorkItem x = d.rec[d.order[u.first]];
    d.meta[x.l].w = 0u;  // the record's cursor has served
    return UnitClaim{1u, sid, u.first, min(u.count, kUnitItems), x.off_l, x.cnt_l, x.l, 1u};
}

// Work through the block units: the block builds the larger endpoint's filter while its first warp cuts
// the lists of the unit's edges into pieces of at most kPieceRows rows, which the warps then take in turn,
// so that they finish together.  `claim` (first thread only) yields the next unit, while the other warps
// scan; the first warp then adds up the unit's lists.
constexpr uint32_t kPieceRows = 8u;  // 1,024 entries
template <bool WORK, int MODE, class S, class Claim>
__device__ __forceinline__ void run_block_units(const S& st, uint32_t* filter, uint4* items, WarpQueues& wq, Work& wk,
                                                Claim&& claim) {
    __shared__ UnitClaim s_claim;
    __shared__ uint32_t s_taken;  // pieces taken
    const unsigned lane = threadIdx.x & 31u;
    auto next = [&] {
        if (threadIdx.x >= 32u) return;
        UnitClaim u{};
        if (lane == 0) u = claim();
        const uint32_t sid = __shfl_sync(0xFFFFFFFFu, u.sid, 0), first = __shfl_sync(0xFFFFFFFFu, u.first, 0),
                       count = __shfl_sync(0xFFFFFFFFu, u.count, 0);
        const StreamDev& d = st.at(sid);
        uint32_t sum = 0;  // (no line of filter_pays lies beyond 64 lists of 2^20 entries)
        for (uint32_t i = lane; i < count; i += 32u) sum += min(d.rec[d.order[first + i]].cnt_s, 1u << 20);
        sum = __reduce_add_sync(0xFFFFFFFFu, sum);
        if (lane == 0) {
            u.filter = filter_pays(colours_of<MODE>(d), u.n, sum);
            s_claim = u;
        }
        __syncwarp();
    };
    next();
    __syncthreads();
    for (;;) {
        const UnitClaim u = s_claim;
        if (!u.ok) break;
        const StreamDev& d = st.at(u.sid);
        const uint32_t lg = filter_lg(2u * u.n, kFilterLg);
        if (u.filter) filter_clear(filter, lg, threadIdx.x, blockDim.x);
        if (threadIdx.x == 0) s_taken = 0u;
        __syncthreads();
        if (threadIdx.x < 32u) {  // items[i] = {block offset, entries, edge, pieces of lists 0 .. i}
            uint32_t carry = 0;
#pragma unroll
            for (uint32_t h = 0; h < 2u; ++h) {
                const uint32_t i = 32u * h + lane;
                uint4 x = make_uint4(0u, 0u, 0u, 0u);
                if (i < u.count) {
                    const uint32_t e = d.order[u.first + i];
                    const WorkItem r = d.rec[e];
                    const uint32_t lgs = table_lg(r.cnt_s);
                    x = make_uint4(r.off_s, r.cnt_s, e, 0u);
                    if (!(block_fits(d, 5, x.x, lgs) && REPT_CHECK(d.ctrl, 6, x.y, list_slots(lgs) + 1u))) x.y = 0u;
                    if (WORK && x.y) {
                        wk.entries += x.y;
                        wk.slots += x.y;
                        atomicAdd(&d.ctrl->class_items[bin_of_cnt(x.y)], 1ull);
                    }
                }
                uint32_t incl = (list_rows(x.y) + kPieceRows - 1u) / kPieceRows;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= (uint32_t)o) incl += y;
                }
                x.w = incl + carry;
                carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
                items[i] = x;
            }
        }
        if (u.filter) filter_build<MODE>(d, filter, lg, u.off, u.n, threadIdx.x, blockDim.x);
        __syncthreads();
        next();
        const uint32_t total = items[kUnitItems - 1u].w;
        // (a loop for each kind of scan: with the choice inside one loop, R-MAT scale 20's scans took 0.8 % longer)
        auto piece = [&](auto&& scan) {
            uint32_t i = 0;
            if (lane == 0) i = atomicAdd(&s_taken, 1u);
            i = __shfl_sync(0xFFFFFFFFu, i, 0);
            if (i >= total) return false;
            // the list that piece i belongs to: as many lists end before it
            const uint32_t at = __popc(__ballot_sync(0xFFFFFFFFu, items[lane].w <= i)) +
                                __popc(__ballot_sync(0xFFFFFFFFu, items[32u + lane].w <= i));
            const uint4 x = items[at];
            const uint32_t rows = list_rows(x.y), pieces = (rows + kPieceRows - 1u) / kPieceRows;
            const uint32_t j0 = (i + pieces - x.w) * kPieceRows;
            scan(x, j0, min(j0 + kPieceRows, rows));
            return true;
        };
        if (u.filter) {
            while (piece([&](const uint4& x, uint32_t j0, uint32_t j1) {
                scan_rows<WORK, MODE>(st, u.sid, filter, lg, x.x, x.y, x.z, j0, j1, wq, wk);
            })) {}
        } else {
            while (piece([&](const uint4& x, uint32_t j0, uint32_t j1) {
                hash_rows<WORK, MODE>(st, u.sid, u.l, x.x, x.y, x.z, j0, j1, wq, wk);
            })) {}
        }
        __syncthreads();
    }
}

// Lists of at most kShortList entries are scanned end to end in warp units.
constexpr uint32_t kShortList = 128u;

// One warp unit: the warp builds l's filter in its share of the shared memory and scans the unit's lists.
template <bool WORK, int MODE, class S>
__device__ __forceinline__ void run_warp_unit(const S& st, uint32_t sid, Unit u, uint32_t* filter, WarpQueues& wq,
                                              Work& wk) {
    const StreamDev& d = st.at(sid);
    const unsigned lane = threadIdx.x & 31u;
    WorkItem x{};
    uint32_t e = 0;
    if (lane < min(u.count, kWarpUnitItems)) {
        e = d.order[u.first + lane];
        x = d.rec[e];
    }
    const uint32_t off_l = __shfl_sync(0xFFFFFFFFu, x.off_l, 0), n_l = __shfl_sync(0xFFFFFFFFu, x.cnt_l, 0);
    const uint32_t lg = filter_lg(n_l, kWarpFilterLg);
    filter_clear(filter, lg, lane, 32u);
    if (lane == 0) d.meta[x.l].w = 0u;  // the record's cursor has served
    __syncwarp();
    filter_build<MODE>(d, filter, lg, off_l, n_l, lane, 32u);
    __syncwarp();
    // lists of more than a row one by one, the others end to end
    uint32_t n = x.cnt_s;
    if (n && !(block_fits(d, 5, x.off_s, table_lg(n)) && REPT_CHECK(d.ctrl, 6, n, list_slots(table_lg(n)) + 1u))) n = 0u;
    if (WORK && n) {
        wk.entries += n;
        wk.slots += n;
        atomicAdd(&d.ctrl->class_items[bin_of_cnt(n)], 1ull);
    }
    for (unsigned lng = __ballot_sync(0xFFFFFFFFu, n > kShortList); lng; lng &= lng - 1u) {
        const int i = __ffs((int)lng) - 1;
        const uint32_t oi = __shfl_sync(0xFFFFFFFFu, x.off_s, i), ni = __shfl_sync(0xFFFFFFFFu, n, i),
                       ei = __shfl_sync(0xFFFFFFFFu, e, i);
        scan_rows<WORK, MODE>(st, sid, filter, lg, oi, ni, ei, 0u, list_rows(ni), wq, wk);
    }
    scan_short<WORK, MODE>(st, sid, filter, lg, x.off_s, n > kShortList ? 0u : n, e, wq, wk);
    __syncwarp();  // the filter is rebuilt by the next unit
}

// The small edges among edges e0 .. e1 - 1 of the batch: 32 edges at a time, their lists'
// entries laid end to end and dealt to the lanes, two per lane and round.  With one group's stored
// colours an entry passes if its colour may agree with the larger endpoint's edge (one hash); else every
// entry passes.
template <bool WORK, int MODE, class S>
__device__ __forceinline__ void run_small_chunk(const S& st, uint32_t sid, uint32_t e0, uint32_t e1, WarpQueues& wq,
                                                Work& wk) {
    const StreamDev& d = st.at(sid);
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t col = colours_of<MODE>(d), mask = id_mask(d);
#pragma unroll 1
    for (uint32_t eb = e0; eb < e1; eb += 32u) {
        const uint32_t e = eb + lane;
        uint32_t cnt = 0, off_s = 0, l = 0;
        if (e < e1 && d.mark[e] == kSmallEdge) {
            const WorkItem x = d.rec[e];
            cnt = x.cnt_s;
            off_s = x.off_s;
            l = x.l;
            if (!(block_fits(d, 5, off_s, table_lg(cnt)) && REPT_CHECK(d.ctrl, 4, cnt, kSmallBatchMax + 1u))) cnt = 0u;
            if (WORK && cnt) {
                wk.entries += cnt;
                wk.slots += cnt;
                atomicAdd(&d.ctrl->class_items[bin_of_cnt(cnt)], 1ull);
            }
        }
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= (uint32_t)o) incl += y;
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31), excl = incl - cnt;
#pragma unroll 1
        for (uint32_t f = 0; f < total; f += 64u) {
            uint32_t word[2], cw[2], own[2], ol[2], pos[2];
            bool v[2];
#pragma unroll
            for (uint32_t p = 0; p < 2u; ++p) {
                const uint32_t at = f + 32u * p + lane;
                v[p] = at < total;
                uint32_t o = 0;  // the lane whose entries cover position `at`: the first with incl > at
#pragma unroll
                for (uint32_t step = 16u; step; step >>= 1)
                    if (__shfl_sync(0xFFFFFFFFu, incl, o + step - 1u) <= at) o += step;
                own[p] = o;
                pos[p] = at - __shfl_sync(0xFFFFFFFFu, excl, o);
                const uint32_t oo = __shfl_sync(0xFFFFFFFFu, off_s, o), oc = __shfl_sync(0xFFFFFFFFu, cnt, o);
                ol[p] = __shfl_sync(0xFFFFFFFFu, l, o);
                word[p] = cw[p] = 0u;
                if (v[p]) {
                    const uint32_t lgs = table_lg(oc);
                    const uint32_t* block = block_at(d.pool, oo);
                    word[p] = list_of(block, lgs, col)[pos[p]];
                    if (col == kColWords) cw[p] = cw_of(block, lgs)[pos[p]];
                }
            }
            if (interleaved(col)) {
#pragma unroll
                for (uint32_t p = 0; p < 2u; ++p)
                    v[p] = v[p] & colour_may_match(d, ol[p], word[p] & mask, col == kColWords ? cw[p] : word[p] >> kIdBits);
            }
#pragma unroll 1
            for (uint32_t p = 0; p < 2u; ++p)
                queue_step<WORK, MODE>(st, wq, (p ? v[1] : v[0]) ? 1u : 0u, p ? pos[1] : pos[0], kEmptyId,
                                       eb + (p ? own[1] : own[0]), sid, wk,
                                       [&](uint32_t) { return p ? word[1] : word[0]; });
        }
    }
}

// UpdateTriangleCNT for every edge of the batch: block units, then warp units and small edges (odd warps
// the other way round, so that the two kinds overlap in small batches), each claimed dynamically.
// Dynamic shared memory: ix_words(MODE, false) words, then 2 c words of counters (tau^(i) of this block).
// WORK = true also tallies the table reads.
template <bool WORK, int MODE>
__device__ __forceinline__ void k_intersect_body(const StreamDev& d, const BatchDev& b) {
    extern __shared__ __align__(16) uint32_t ix_smem[];
    uint32_t* filter = ix_smem;
    uint4* items = reinterpret_cast<uint4*>(filter + kFilterWords);
    uint32_t* half = ix_smem + ix_words(MODE, false);
    for (uint32_t i = threadIdx.x; i < 2u * d.c; i += blockDim.x) half[i] = 0u;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned wid = threadIdx.x >> 5;
    WarpQueues wq{filter + kFilterWords + 4u * kUnitItems + wid * queue_words(MODE, false), 0u, 0u};
    const OneStream st{d, half};
    Work wk;
    Ctrl* ct = d.ctrl;
    __syncthreads();
    if (ct->status == 0u) {
        // WORK: warp-cycles of block units, warp units and small edges, kept under classes 5, 4 and 3
        long long c0 = WORK ? clock64() : 0;
        auto mark = [&](int cls) {
            if (WORK && lane == 0) {
                const long long c1 = clock64();
                atomicAdd(&ct->class_cycles[cls], (unsigned long long)(c1 - c0));
                c0 = c1;
            }
        };
        int kind = kBinBig;
        run_block_units<WORK, MODE>(st, filter, items, wq, wk, [&]() -> UnitClaim {
            for (; kind >= kBinBlock; --kind) {
                if (ct->bin_count[kind] == 0ull) continue;
                const unsigned long long i = atomicAdd(&ct->bin_next[kind], 1ull);
                if (i < ct->bin_count[kind]) return claimed_unit(d, 0u, kind == kBinBig ? i : d.unit_cap + i);
            }
            return UnitClaim{};
        });
        mark(5);
#pragma unroll 1
        for (uint32_t part = 0; part < 2u; ++part) {
            const int bin = (part ^ wid) & 1u ? kBinSmall : kBinWarp;
            const unsigned long long count = ct->bin_count[bin];
            for (;;) {
                unsigned long long i = 0;
                if (lane == 0) i = atomicAdd(&ct->bin_next[bin], 1ull);
                i = __shfl_sync(0xFFFFFFFFu, i, 0);
                if (i >= count) break;
                if (bin == kBinWarp)
                    run_warp_unit<WORK, MODE>(st, 0u, d.units[d.unit_cap - 1ull - i], filter + (wid << kWarpFilterLg), wq, wk);
                else
                    run_small_chunk<WORK, MODE>(st, 0u, (uint32_t)i * b.chunk, (uint32_t)min((i + 1ull) * b.chunk, b.n), wq, wk);
            }
            mark(bin == kBinWarp ? 4 : 3);
        }
        cand_flush<WORK, MODE>(st, wq, wk, true);
    }
    if (WORK) {
        for (int o = 16; o > 0; o >>= 1) {
            wk.entries += __shfl_down_sync(0xFFFFFFFFu, wk.entries, o);
            wk.slots += __shfl_down_sync(0xFFFFFFFFu, wk.slots, o);
            wk.probes += __shfl_down_sync(0xFFFFFFFFu, wk.probes, o);
            wk.pslots += __shfl_down_sync(0xFFFFFFFFu, wk.pslots, o);
            wk.wedges += __shfl_down_sync(0xFFFFFFFFu, wk.wedges, o);
            wk.counted += __shfl_down_sync(0xFFFFFFFFu, wk.counted, o);
        }
        if (lane == 0) {
            atomicAdd(&d.ctrl->small_entries, wk.entries);
            atomicAdd(&d.ctrl->small_slots, wk.slots);
            atomicAdd(&d.ctrl->probes, wk.probes);
            atomicAdd(&d.ctrl->probe_slots, wk.pslots);
            atomicAdd(&d.ctrl->wedges, wk.wedges);
            atomicAdd(&d.ctrl->counted, wk.counted);
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < d.c; i += blockDim.x) {
        const unsigned long long n = ((unsigned long long)half[2u * i + 1u] << 32) | half[2u * i];
        if (n) atomicAdd(&d.proc[i], n);
    }
}

// ---------------------------------------------------------------------------------------------
// Intersection for a group of streams with one grid: every block and warp may work on any stream.  The
// streams' lists of each kind of work are concatenated (k_group_prefix writes, per kind, the prefix of
// the streams' counts); claims come from one cursor per kind, and each finds its stream from the prefix.
// Candidates and closed wedges carry their stream and tau^(i) goes straight to global memory.

// Per kind c: pref[c * (k + 1) + i] = sum of the counts of streams < i; cursors reset.  One
// block of any multiple of 32 threads up to 1024.
__device__ __forceinline__ void group_prefix_body(const StreamDev* __restrict__ ds, uint32_t k,
                                                  unsigned long long* pref, unsigned long long* cursor) {
    __shared__ unsigned long long warp_sum[32];
    __shared__ unsigned long long carry;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, wid = tid >> 5, warps = blockDim.x >> 5;
    for (int c = 0; c < kBins; ++c) {
        if (tid == 0) carry = 0ull;
        __syncthreads();
        for (uint32_t base = 0; base < k; base += blockDim.x) {
            const uint32_t i = base + tid;
            const unsigned long long v = i < k && ds[i].ctrl->status == 0u ? ds[i].ctrl->bin_count[c] : 0ull;
            unsigned long long incl = v;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= (uint32_t)o) incl += y;
            }
            if (lane == 31) warp_sum[wid] = incl;
            __syncthreads();
            if (wid == 0) {
                const unsigned long long w = lane < warps ? warp_sum[lane] : 0ull;
                unsigned long long wi = w;
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
                    if (lane >= (uint32_t)o) wi += y;
                }
                warp_sum[lane] = wi - w;
            }
            __syncthreads();
            const unsigned long long excl = carry + warp_sum[wid] + incl - v;
            if (i < k) pref[c * (k + 1) + i] = excl;
            __syncthreads();
            if (tid == blockDim.x - 1) carry = excl + v;
            __syncthreads();
        }
        if (tid == 0) {
            pref[c * (k + 1) + k] = carry;
            cursor[c] = 0ull;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(1024) k_group_prefix(const StreamDev* __restrict__ ds, uint32_t k,
                                                       unsigned long long* __restrict__ pref,
                                                       unsigned long long* __restrict__ cursor) {
    group_prefix_body(ds, k, pref, cursor);
}

// Stream of item `i`: the last stream whose prefix is <= i.
__device__ __forceinline__ uint32_t group_stream_search(const unsigned long long* pc, uint32_t k,
                                                        unsigned long long i) {
    uint32_t lo = 0, hi = k - 1;  // pc[0] = 0 <= i
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (pc[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// MODE: the colour storage of every stream, or kColAny.
template <int MODE>
__device__ __forceinline__ void intersect_group_body(const StreamDev* __restrict__ ds, const BatchDev* __restrict__ bs,
                                                     uint32_t k, const unsigned long long* pref,
                                                     unsigned long long* cursor, uint32_t* smem) {
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
    uint32_t* filter = smem;
    uint4* items = reinterpret_cast<uint4*>(filter + kFilterWords);
    WarpQueues wq{filter + kFilterWords + 4u * kUnitItems + wid * queue_words(MODE, true), 0u, 0u};
    const ManyStreams st{ds};
    Work wk;
    int kind = kBinBig;
    run_block_units<false, MODE>(st, filter, items, wq, wk, [&]() -> UnitClaim {
        for (; kind >= kBinBlock; --kind) {
            const unsigned long long* pc = pref + kind * (k + 1);
            if (pc[k] == 0ull) continue;
            const unsigned long long i = atomicAdd(&cursor[kind], 1ull);
            if (i < pc[k]) {
                const uint32_t sid = group_stream_search(pc, k, i);
                return claimed_unit(ds[sid], sid, i - pc[sid] + (kind == kBinBig ? 0ull : ds[sid].unit_cap));
            }
        }
        return UnitClaim{};
    });
#pragma unroll 1
    for (uint32_t part = 0; part < 2u; ++part) {
        const int bin = (part ^ wid) & 1u ? kBinSmall : kBinWarp;
        const unsigned long long* pc = pref + bin * (k + 1);
        for (;;) {
            unsigned long long i = 0;
            if (lane == 0) i = atomicAdd(&cursor[bin], 1ull);
            i = __shfl_sync(0xFFFFFFFFu, i, 0);
            if (i >= pc[k]) break;
            const uint32_t sid = group_stream_search(pc, k, i);
            i -= pc[sid];
            if (bin == kBinWarp)
                run_warp_unit<false, MODE>(st, sid, ds[sid].units[ds[sid].unit_cap - 1ull - i],
                                              filter + (wid << kWarpFilterLg), wq, wk);
            else
                run_small_chunk<false, MODE>(st, sid, (uint32_t)i * bs[sid].chunk,
                                                (uint32_t)min((i + 1ull) * bs[sid].chunk, bs[sid].n), wq, wk);
        }
    }
    cand_flush<false, MODE>(st, wq, wk, true);
}

// Dynamic shared memory: ix_words(MODE, true) words.
template <int MODE>
__global__ void __launch_bounds__(kIxThreads, kIxBlocks) k_intersect_group(const StreamDev* __restrict__ ds,
                                                                           const BatchDev* __restrict__ bs, uint32_t k,
                                                                           const unsigned long long* __restrict__ pref,
                                                                           unsigned long long* __restrict__ cursor) {
    extern __shared__ __align__(16) uint32_t ix_smem[];
    intersect_group_body<MODE>(ds, bs, k, pref, cursor, ix_smem);
}

// Algorithm 2's triangle-pair counters, folded in after the intersection.  Edge e of group k was a
// wedge edge of kcnt closed wedges this batch, all for the processor i = k*m + h_k(e).  In stream
// order they saw the counter values B, B+1, ..., B+kcnt-1 (B its value before the batch), so their
// contribution to eta^(i) and to eta_x, eta_y of e's endpoints is kcnt*B + kcnt*(kcnt-1)/2, whatever
// their order; then the counter advances by kcnt.  (The counter of a newly stored edge starts at 0.)
__global__ void k_pairs(StreamDev d) {
    if (d.ctrl->status) return;
    const unsigned long long n = d.ctrl->n_pairs;
    for (unsigned long long q = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; q < n;
         q += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t idx = d.pair_list[q];
        const uint32_t t = idx / d.groups, k = idx % d.groups;
        const unsigned long long kc = d.pair_evt[idx], base = d.pair_tau[idx];
        const unsigned long long add = kc * base + kc * (kc - 1) / 2;
        const uint2 e = d.edge_ends[t];
        const uint32_t i = k * d.m + colour_of(e.x, e.y, group_seed(d.seed, k), d.fm);
        atomicAdd(&d.eta_proc[i], add);
        atomicAdd(&d.eta_local[e.x], add);
        atomicAdd(&d.eta_local[e.y], add);
        d.pair_tau[idx] = (uint32_t)(base + kc);
        d.pair_evt[idx] = 0u;
    }
}

// Algorithm 2's estimates (c > m, c mod m != 0): the two group estimates combined with the plug-in
// inverse-variance weights; with both weights zero the full groups' estimate.  Same expression order
// as the scalar formulas of Section III-B.2.
__device__ __forceinline__ double combine_estimates(double t1, double t2, double eta_hat, double md, double c1,
                                                    double c2) {
    const double w1 = t1 * (md - 1.0) / c1;
    const double w2 = (t1 * (md * md - c2) + 2.0 * eta_hat * (md - c2)) / c2;
    return (w1 + w2 > 0.0) ? (w2 * t1 + w1 * t2) / (w1 + w2) : t1;
}

// tau_hat into *global (the first warp of the first block) and, with `out`, the local estimates.
__global__ void k_estimates_partial(const unsigned long long* __restrict__ proc, const unsigned long long* __restrict__ eta,
                                    const unsigned long long* __restrict__ l1, const unsigned long long* __restrict__ l2,
                                    const unsigned long long* __restrict__ el, uint32_t n, uint32_t m, uint32_t c,
                                    double* __restrict__ global, double* __restrict__ out) {
    const uint32_t c1 = c / m, c2 = c % m;
    const double md = (double)m;
    if (blockIdx.x == 0 && threadIdx.x < 32u) {
        unsigned long long s1 = 0, s2 = 0, se = 0;
        for (uint32_t i = threadIdx.x; i < c; i += 32u) {
            if (i < c1 * m) s1 += proc[i]; else s2 += proc[i];
            se += eta[i];
        }
        for (int o = 16; o > 0; o >>= 1) {
            s1 += __shfl_down_sync(0xFFFFFFFFu, s1, o);
            s2 += __shfl_down_sync(0xFFFFFFFFu, s2, o);
            se += __shfl_down_sync(0xFFFFFFFFu, se, o);
        }
        if (threadIdx.x == 0) {
            const double t1 = (double)s1 * (md / (double)c1), t2 = (double)s2 * (md * md / (double)c2);
            const double eta_hat = (double)se * (md * md * md / (double)c);
            *global = combine_estimates(t1, t2, eta_hat, md, (double)c1, (double)c2);
        }
    }
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; out && v < n; v += gridDim.x * blockDim.x) {
        const double a1 = (double)l1[v] * (md / (double)c1), a2 = (double)l2[v] * (md * md / (double)c2);
        const double eh = (double)el[v] * (md * md * md / (double)c);
        out[v] = combine_estimates(a1, a2, eh, md, (double)c1, (double)c2);
    }
}

// sum_i tau_v^(i) over all processors when the local counts are split in two.
__global__ void k_add_local(const unsigned long long* __restrict__ a, const unsigned long long* __restrict__ b,
                            uint32_t n, unsigned long long* __restrict__ out) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) out[v] = a[v] + b[v];
}

// Kernel entry points.  Each batch kernel exists twice: for one stream (state and batch passed by
// value) and for many streams at once (`_multi`: blockIdx.y selects the stream, whose state and batch
// descriptors are read from device arrays; blockIdx.x / gridDim.x then range over that stream's blocks).
__device__ __forceinline__ Grid launch_grid() { return Grid{blockIdx.x, gridDim.x}; }

__global__ void k_classify(StreamDev d, BatchDev b) {
    follow_previous();
    k_classify_body(d, b, launch_grid());
}

__global__ void k_classify_multi(const StreamDev* __restrict__ ds, const BatchDev* __restrict__ bs) {
    __shared__ StreamDev sd;
    __shared__ BatchDev sb;
    if (threadIdx.x == 0) {
        sd = ds[blockIdx.y];
        sb = bs[blockIdx.y];
    }
    __syncthreads();
    k_classify_body(sd, sb, launch_grid());
}

__global__ void k_plan(StreamDev d) {
    follow_previous();
    k_plan_body(d, launch_grid());
}

__global__ void k_plan_multi(const StreamDev* __restrict__ ds, const BatchDev* __restrict__ bs) {
    (void)bs;
    __shared__ StreamDev sd;
    if (threadIdx.x == 0) sd = ds[blockIdx.y];
    __syncthreads();
    k_plan_body(sd, launch_grid());
}

__global__ void __launch_bounds__(256) k_commit(StreamDev d) {
    follow_previous();
    __shared__ __align__(16) uint32_t smem[kCommitSmemWords];
    k_commit_body(d, launch_grid(), smem);
}

__global__ void __launch_bounds__(256) k_commit_multi(const StreamDev* __restrict__ ds, const BatchDev* __restrict__ bs) {
    (void)bs;
    __shared__ __align__(16) uint32_t smem[kCommitSmemWords];
    __shared__ StreamDev sd;
    if (threadIdx.x == 0) sd = ds[blockIdx.y];
    __syncthreads();
    k_commit_body(sd, launch_grid(), smem);
}

__global__ void __launch_bounds__(256) k_rehash_big(StreamDev d) {
    follow_previous();
    __shared__ __align__(16) uint32_t smem[kMoveSmemWords];
    k_rehash_big_body(d, launch_grid(), smem);
}

__global__ void __launch_bounds__(256) k_rehash_big_multi(const StreamDev* __restrict__ ds,
                                                            const BatchDev* __restrict__ bs) {
    (void)bs;
    __shared__ StreamDev sd;
    __shared__ __align__(16) uint32_t smem[kMoveSmemWords];
    if (threadIdx.x == 0) sd = ds[blockIdx.y];
    __syncthreads();
    k_rehash_big_body(sd, launch_grid(), smem);
}

// Two blocks of 1024 threads per SM (32 registers a thread), so that the whole grid is resident.  Dynamic
// shared memory: kHugeSmemWords words.
__global__ void __launch_bounds__(1024, 2) k_rehash_huge(StreamDev d) {
    follow_previous();
    extern __shared__ __align__(16) uint32_t hsmem[];
    k_rehash_huge_body(d, launch_grid(), hsmem);
}

__global__ void __launch_bounds__(1024, 2) k_rehash_huge_multi(const StreamDev* __restrict__ ds,
                                                              const BatchDev* __restrict__ bs) {
    (void)bs;
    extern __shared__ __align__(16) uint32_t hsmem[];
    __shared__ StreamDev sd;
    if (threadIdx.x == 0) sd = ds[blockIdx.y];
    __syncthreads();
    k_rehash_huge_body(sd, launch_grid(), hsmem);
}

// 5 blocks of 256 threads per SM (48 registers).
__global__ void __launch_bounds__(256, 5) k_insert(StreamDev d, BatchDev b) {
    follow_previous();
    k_insert_body(d, b, launch_grid());
}

__global__ void k_insert_multi(const StreamDev* __restrict__ ds, const BatchDev* __restrict__ bs) {
    __shared__ StreamDev sd;
    __shared__ BatchDev sb;
    if (threadIdx.x == 0) {
        sd = ds[blockIdx.y];
        sb = bs[blockIdx.y];
    }
    __syncthreads();
    k_insert_body(sd, sb, launch_grid());
}

__global__ void __launch_bounds__(256) k_units(StreamDev d, BatchDev b) {
    follow_previous();
    k_units_body(d, b, launch_grid());
}

__global__ void __launch_bounds__(256) k_units_multi(const StreamDev* __restrict__ ds, const BatchDev* __restrict__ bs) {
    __shared__ StreamDev sd;
    __shared__ BatchDev sb;
    if (threadIdx.x == 0) {
        sd = ds[blockIdx.y];
        sb = bs[blockIdx.y];
    }
    __syncthreads();
    k_units_body(sd, sb, launch_grid());
}

__global__ void __launch_bounds__(256) k_order(StreamDev d, BatchDev b) {
    follow_previous();
    k_order_body(d, b, launch_grid());
}

__global__ void __launch_bounds__(256) k_order_multi(const StreamDev* __restrict__ ds, const BatchDev* __restrict__ bs) {
    __shared__ StreamDev sd;
    __shared__ BatchDev sb;
    if (threadIdx.x == 0) {
        sd = ds[blockIdx.y];
        sb = bs[blockIdx.y];
    }
    __syncthreads();
    k_order_body(sd, sb, launch_grid());
}

// Every step of a small batch before its intersection in one launch: a single cluster of thread blocks runs
// them in turn, with the cluster's hardware barrier between them (its release and acquire order global
// memory as well), so that a batch of a few thousand edges pays for two launches instead of nine.
// Dynamic shared memory: kStateSmemWords words.
constexpr uint32_t kStateBlocks = 8, kStateThreads = 1024;
constexpr uint32_t kStateSmemWords = 2u * (kStateThreads / 32u) * kMoveSlots;
static_assert(kStateSmemWords >= kHugeSmemWords && kStateSmemWords >= kCommitSmemWords * (kStateThreads / 256u),
              "the steps share the memory");

// (not the .aligned forms: the steps end in code that the lanes of a warp leave at different times, and those
// forms are undefined for a warp that has not met again)
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __cluster_dims__(kStateBlocks, 1, 1) __launch_bounds__(kStateThreads, 1) k_state(StreamDev d, BatchDev b) {
    follow_previous();
    extern __shared__ __align__(16) uint32_t hsmem[];
    const Grid g = launch_grid();
    k_classify_body(d, b, g);
    cluster_barrier();
    k_plan_body(d, g);
    cluster_barrier();
    k_commit_body(d, g, hsmem);
    cluster_barrier();
    k_rehash_big_body(d, g, hsmem);
    // the tables that k_rehash_huge builds in place are emptied by every block and filled by any; without such a
    // table (the same answer in every block: the count rests between the commit and the insert) the blocks need
    // not meet, which a batch of 4,096 edges would pay with 3.7 us of 70
    if (n_giants(d)) cluster_barrier();
    else __syncthreads();
    k_rehash_huge_body(d, g, hsmem);
    cluster_barrier();
    k_insert_body(d, b, g);
    cluster_barrier();
    k_units_body(d, b, g);
    cluster_barrier();
    k_order_body(d, b, g);
}

// ---------------------------------------------------------------------------------------------
// One persistent launch for a whole group round: every step of the batch path (classify, plan,
// commit, both block moves, insert, sort, the group's intersection) for every stream, separated by
// grid-wide barriers.  The grid is co-resident (a cooperative launch); each step runs over virtual
// blocks (stream, block of that stream) exactly as the launch per step would, so the counts are the
// same.  Every barrier wait is bounded in time: when it runs out, the block records kStTimeout in
// every stream's status (REPT_E_TIMEOUT at the next synchronising call) and returns, and the other
// blocks, seeing timed_out, stop waiting and return too.  No block ever waits without a limit.

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// All blocks of the grid meet; false if the wait gave up (after wait_ns nanoseconds) or another
// block's did.
__device__ __forceinline__ bool grid_barrier(GroupSync* gs, unsigned long long wait_ns) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned int* vgen = &gs->gen;
        volatile unsigned int* vto = &gs->timed_out;
        int ok = 1;
        const unsigned int g = *vgen;  // cannot advance before this block arrives
        __threadfence();               // this block's writes of the step before the barrier
        const unsigned int target = gridDim.x + gs->extra;
        if (atomicAdd(&gs->count, 1u) == target - 1u) {
            atomicExch(&gs->count, 0u);
            __threadfence();
            atomicAdd(&gs->gen, 1u);
        } else {
            const unsigned long long t0 = global_ns();
            while (*vgen == g) {
                if (*vto || global_ns() - t0 > wait_ns) {
                    atomicExch(&gs->timed_out, 1u);
                    ok = 0;
                    break;
                }
                __nanosleep(100);
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Virtual blocks per stream of each step (the multi-launch shape's grid x dimensions).
struct PersistShape {
    uint32_t x_edge, x_big, x_huge;
};

// Dynamic shared memory of the persistent kernel: the larger of the block moves' and the group
// intersection's needs.
static_assert(ix_words(kColAny, true) >= kHugeSmemWords, "the block moves fit");
constexpr uint32_t kPersistSmemWords = kMoveSmemWords > ix_words(kColAny, true) ? kMoveSmemWords : ix_words(kColAny, true);

__global__ void __launch_bounds__(256, 3) k_group_persistent(const StreamDev* __restrict__ ds,
                                                           const BatchDev* __restrict__ bs, uint32_t k,
                                                           PersistShape sh, unsigned long long* pref,
                                                           unsigned long long* cursor, GroupSync* gs,
                                                           unsigned long long wait_ns) {
    extern __shared__ __align__(16) uint32_t psmem[];
    __shared__ StreamDev sd;
    __shared__ BatchDev sb;
    __shared__ uint32_t s_cur;
    if (threadIdx.x == 0) s_cur = 0xFFFFFFFFu;
    __syncthreads();
    // run `body` for every virtual block (stream, block x of X) this block is dealt
    auto step = [&](uint32_t X, auto&& body) {
        const unsigned long long total = (unsigned long long)k * X;
        for (unsigned long long vb = blockIdx.x; vb < total; vb += gridDim.x) {
            const uint32_t sid = (uint32_t)(vb / X);
            if (sid != s_cur) {  // uniform over the block
                __syncthreads();
                if (threadIdx.x == 0) {
                    sd = ds[sid];
                    sb = bs[sid];
                    s_cur = sid;
                }
                __syncthreads();
            }
            body(Grid{(uint32_t)(vb % X), X});
        }
    };
    bool ok = true;
    step(sh.x_edge, [&](Grid g) { k_classify_body(sd, sb, g); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) step(sh.x_edge, [&](Grid g) { k_plan_body(sd, g); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) step(sh.x_edge, [&](Grid g) { k_commit_body(sd, g, psmem); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) step(sh.x_big, [&](Grid g) { k_rehash_big_body(sd, g, psmem); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) step(sh.x_huge, [&](Grid g) { k_rehash_huge_body(sd, g, psmem); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) step(sh.x_edge, [&](Grid g) { k_insert_body(sd, sb, g); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) step(sh.x_edge, [&](Grid g) { k_units_body(sd, sb, g); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) step(sh.x_edge, [&](Grid g) { k_order_body(sd, sb, g); });
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok && blockIdx.x == 0) group_prefix_body(ds, k, pref, cursor);
    ok = ok && grid_barrier(gs, wait_ns);
    if (ok) {
        intersect_group_body<kColAny>(ds, bs, k, pref, cursor, psmem);
        return;
    }
    // a wait ran out: the round is not applied for any stream (every step checks the status first)
    if (threadIdx.x == 0)
        for (uint32_t i = blockIdx.x; i < k; i += gridDim.x) atomicOr(&ds[i].ctrl->status, kStTimeout);
}

// Streams whose entries carry their colour (one hash group, m <= 256).
template <bool WORK>
__global__ void __launch_bounds__(kIxThreads, kIxBlocks) k_intersect(StreamDev d, BatchDev b) {
    follow_previous();
    k_intersect_body<WORK, (int)kColInEntry>(d, b);
}

// Streams whose entries have colour words (one hash group whose colour does not fit the entry: m > 256
// or more than 2^24 nodes).
template <bool WORK>
__global__ void __launch_bounds__(kIxThreads, kIxBlocks) k_intersect_words(StreamDev d, BatchDev b) {
    follow_previous();
    k_intersect_body<WORK, (int)kColWords>(d, b);
}

// Streams of several hash groups, with a colour word beside every stream index.
template <bool WORK>
__global__ void __launch_bounds__(kIxThreads, kIxBlocks) k_intersect_multi(StreamDev d, BatchDev b) {
    follow_previous();
    k_intersect_body<WORK, (int)kColMulti>(d, b);
}

// Streams without stored colours (too many hash groups for a word, or too little memory for one).
template <bool WORK>
__global__ void __launch_bounds__(kIxThreads, kIxBlocks) k_intersect_probe(StreamDev d, BatchDev b) {
    follow_previous();
    k_intersect_body<WORK, (int)kColNone>(d, b);
}

// A handle's change of layout, between a batch's k_plan and its k_commit or between batches: the batch's
// requests again, the quads that all blocks take, then every block into the new pool.
__global__ void k_plan_again(StreamDev d) { k_plan_body<true>(d, launch_grid()); }

__global__ void __launch_bounds__(256) k_layout_quads(StreamDev d) {
    unsigned long long sum = 0;
    for (unsigned long long x = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; x < d.n_nodes;
         x += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t cnt = d.meta[x].y;
        if (cnt) sum += block_quads(table_lg(cnt), d.colours);
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, o);
    if ((threadIdx.x & 31u) == 0 && sum) atomicAdd(&d.ctrl->layout_quads, sum);
}

// From kColMulti to kColNone or back, a block of the grid per node: both keep split tables whose keys stand
// alike, so that everything is copied in place order (colour words are formed anew).  pool_top starts at 0
// and hands out the new places.
__global__ void __launch_bounds__(256) k_relayout(StreamDev d, const uint2* __restrict__ old, unsigned long long old_quads,
                                                  uint32_t from_colours) {
    __shared__ unsigned long long s_off;
    const uint32_t col = d.colours;
    for (unsigned long long x = blockIdx.x; x < d.n_nodes; x += gridDim.x) {
        const uint4 m = d.meta[x];
        const uint32_t cnt = m.y, lg = table_lg(cnt), quads = block_quads(lg, col);
        if (cnt == 0u) continue;
        if (threadIdx.x == 0) s_off = atomicAdd(&d.ctrl->pool_top, (unsigned long long)quads);
        __syncthreads();
        const unsigned long long off = s_off;
        // (the pool has room for k_layout_quads' sum, and blocks lie in the old one: checked all the same)
        if (off + quads <= d.pool_quads && (unsigned long long)m.x + block_quads(lg, from_colours) <= old_quads) {
            const uint32_t* from = block_at(old, m.x);
            uint32_t* to = block_at(d.pool, off);
            for (uint32_t h = threadIdx.x; h < 1u << lg; h += blockDim.x) {
                const uint32_t id = from[h];
                bool kept;
                to[h] = id;
                if (id != kEmptyId)
                    table_store(to, lg, h, *eidx_of(from, h, lg, from_colours),
                                col == kColMulti ? colour_word(d, (uint32_t)x, id, kept) : 0u, col);
            }
            const uint32_t *ids = list_of(from, lg, from_colours), *aux = aux_of(from, lg, from_colours);
            for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x) {
                const uint32_t id = ids[j], t = aux[from_colours == kColMulti ? 2ull * j : j];
                bool kept;
                list_of(to, lg, col)[j] = id;
                if (col == kColMulti)
                    reinterpret_cast<uint2*>(aux_of(to, lg, col))[j] = make_uint2(t, colour_word(d, (uint32_t)x, id, kept));
                else
                    aux_of(to, lg, col)[j] = t;
            }
        } else if (threadIdx.x == 0) {
            atomicOr(&d.ctrl->status, kStInternal);
        }
        __syncthreads();  // every thread has read the record
        if (threadIdx.x == 0) d.meta[x].x = (uint32_t)off;
    }
}

// Turn the blocks of a version 3 snapshot, whose lists are {entry word, stream index} pairs, into lists of
// entry words in place, a block of the grid per node: a list takes the same room in both, and its pairs
// fill the table before the words close up.
__global__ void __launch_bounds__(256) k_unpair(StreamDev d) {
    __shared__ int s_bad;
    const uint32_t col = d.colours, mask = id_mask(d);
    for (unsigned long long x = blockIdx.x; x < d.n_nodes; x += gridDim.x) {
        const uint4 m = d.meta[x];
        const uint32_t cnt = m.y, lg = table_lg(cnt);
        if (cnt == 0u) continue;
        const bool fits = (unsigned long long)m.x + block_quads(lg, col) <= d.pool_quads;
        if (threadIdx.x == 0) s_bad = !fits;
        if (fits) {
            uint32_t* block = block_at(d.pool, m.x);
            uint32_t* list = list_of(block, lg, col);
            init_table_keys(block, lg, col, threadIdx.x, blockDim.x);
            __syncthreads();
            for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x)
                if (!table_insert(block, lg, list[2ull * j] & mask, list[2ull * j + 1u], 0u, col)) s_bad = 1;
            __syncthreads();
            for (uint32_t j0 = 0; j0 < cnt; j0 += blockDim.x) {  // every word moves towards the front
                const uint32_t j = j0 + threadIdx.x;
                const uint32_t word = j < cnt ? list[2ull * j] : 0u;
                __syncthreads();
                if (j < cnt) list[j] = word;
                __syncthreads();
            }
            if (col == kColNone) {
                uint32_t ns;
                for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x)
                    aux_of(block, lg, col)[j] = table_find(block, lg, list[j], ns, col);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0 && s_bad) atomicOr(&d.ctrl->status, kStInternal);
        __syncthreads();
    }
}

// tau_hat = f * sum_{i < c_used} tau^(i) into *global (first block) and tau_hat_v = f * sum_i tau_v^(i) into
// out, f formed in double on the host; either output may be NULL.
__global__ void k_estimates(const unsigned long long* __restrict__ proc, uint32_t c_used,
                            const unsigned long long* __restrict__ local, uint32_t n, double f,
                            double* __restrict__ global, double* __restrict__ out) {
    if (blockIdx.x == 0 && global) {
        __shared__ unsigned long long part[32];
        unsigned long long s = 0;
        for (uint32_t i = threadIdx.x; i < c_used; i += blockDim.x) s += proc[i];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
        if ((threadIdx.x & 31u) == 0) part[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x < 32) {
            s = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0ull;
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, o);
            if (threadIdx.x == 0) *global = (double)s * f;
        }
    }
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; out && v < n; v += gridDim.x * blockDim.x)
        out[v] = (double)local[v] * f;
}

}  // namespace
}  // namespace rept
