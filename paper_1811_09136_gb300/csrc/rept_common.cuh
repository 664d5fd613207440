// Device-side data layout and helpers of the REPT streaming counter.
//
// HBM layout of one stream (one rept_state):
//   meta[n_nodes]   uint4 {off, cnt, 0, grp}: node x's block starts at slot
//                   4*off of the pool and holds cnt entries; its size is a
//                   function of cnt alone (table_lg below), so a node's block
//                   is re-allocated exactly when cnt crosses a power-of-two
//                   boundary.  grp counts the batch's grouped edges whose
//                   larger endpoint is x (zero between batches).
//   cnt_add[n_nodes]  the current batch's new entries of x, as k_classify
//                   counts them; k_plan takes each touched node's count and
//                   clears it, so it is zero between batches.
//   pool[]          32-byte quads: per node, an open-addressing (linear probing,
//                   4-key buckets) table of 2^lg neighbour ids and their stream
//                   indices (for single-group streams with stored colours
//                   each 32-byte bucket holds its 4 ids and then their 4
//                   indices, so that an insert or a probe hit touches one
//                   sector; the others keep all ids
//                   first and the indices after them, ids packed densely), then
//                   the neighbour ids as a packed list, 4 bytes each, which is
//                   all that the intersection's scans read (block_quads).
//                   An entry (w, t) of x is the stored edge {x, w} that
//                   arrived at stream index t.  Empty keys are all-ones.  The
//                   tables of all processors share one union adjacency: an
//                   edge is stored once if any processor keeps it, and which
//                   processors keep it is recomputed from the hash or read from
//                   a stored colour word when needed
//                   (Section III-A: processor i keeps colour i).
//   local[n_nodes]  uint64 sum over processors of tau_v^(i)
//   proc[c]         uint64 tau^(i)
// Per-batch scratch: touched[] (nodes with new entries), grow_rel[] (their new
// table's offset relative to this batch's allocation), the work records, and
// the control block.
#pragma once

#include <algorithm>
#include <cstdint>
#include <cstdio>

#include "rept.h"

namespace rept {

constexpr uint32_t kEmptyId = 0xFFFFFFFFu;
constexpr uint64_t kGoldenGamma = 0x9E3779B97F4A7C15ull;  // SplitMix64 increment
constexpr uint32_t kIdBits = 24;                             // node-id bits of a list entry with a colour
constexpr uint32_t kIdMask = (1u << kIdBits) - 1u;
constexpr uint32_t kNoGrow = 0xFFFFFFFFu;
constexpr uint32_t kMaxProcessors = 4096;  // per-block tau^(i) histogram lives in shared memory
// Work kinds of the intersection.  An edge whose smaller endpoint holds at most tile_max entries is
// small: warps take them straight from the batch, a chunk of edges at a time.  The others are grouped
// by their larger endpoint l into units of edges of one l; a unit is worked on by a warp when l holds at
// most kWarpUnitNodes entries, else by a thread block (those of the largest l's, above kBigUnitNodes
// entries, first).  kWarpUnitNodes at 512: 1 to 4 % slower on 36 workloads; at 2,048: R-MAT scale 20 2 % faster in
// batches of 2^17, 1 % slower at 2^20.  kBigUnitNodes at 2,048 or 16,384: no difference beyond 1 %.
constexpr int kBins = 4;
constexpr int kBinSmall = 0, kBinWarp = 1, kBinBlock = 2, kBinBig = 3;
constexpr int kClasses = 6;  // work-counter classes (bin_of_cnt)
constexpr unsigned long long kSmallBatch = 1ull << 15;  // smaller batches: make_batch
constexpr uint32_t kSmallBatchMax = 64u;
constexpr uint32_t kWarpUnitItems = 32u;  // edges per warp unit: at most one per lane
constexpr uint32_t kWarpUnitEntries = 8192u;
constexpr uint32_t kUnitItems = 64u;      // ... and at most of a block unit
constexpr uint32_t kWarpUnitNodes = 1024u;
constexpr uint32_t kBigUnitNodes = 4096u;
// Marks (StreamDev::mark): node ids are below kSmallEdge (n_nodes < 2^32 - 1)
constexpr uint32_t kNoWork = 0xFFFFFFFFu, kSmallEdge = 0xFFFFFFFEu;

// status bits (sticky)
constexpr unsigned kStRange = 1u, kStCapacity = 2u, kStInternal = 4u, kStTimeout = 8u, kStDuplicate = 16u;
constexpr unsigned kStBounds = 32u;  // REPT_DEBUG_BOUNDS builds: an index check failed

// The REPT_E_* code (rept.h) that a sticky status word reports, most specific condition first.  A
// failed index check of the REPT_DEBUG_BOUNDS build is an internal error.
inline int status_to_code(unsigned st) {
    if (st & kStRange) return REPT_E_RANGE;
    if (st & kStCapacity) return REPT_E_CAPACITY;
    if (st & kStTimeout) return REPT_E_TIMEOUT;
    if (st & kStInternal) return REPT_E_INTERNAL;
    if (st & kStDuplicate) return REPT_E_DUPLICATE;
    if (st & kStBounds) return REPT_E_INTERNAL;
    return REPT_OK;
}

// REPT_DEBUG_BOUNDS builds: print the first failed index check ({site, index, bound, failures}, the
// `dbg` words of the control block) to stderr.
inline void report_failed_check(const unsigned long long* dbg) {
    if (dbg[3])
        std::fprintf(stderr, "rept: index check at site %llu failed: index %llu, bound %llu (%llu failures)\n",
                     dbg[0], dbg[1], dbg[2], dbg[3]);
}

// x mod m for 64-bit x and 32-bit m >= 2 without a division: Lemire, Kaser, Kurz, "Faster Remainder
// by Direct Computation" (2019).  With the 128-bit magic M = floor((2^128 - 1) / m) + 1, the low 128
// bits of M * x, multiplied by m, hold x mod m in their top 64 bits; 128 >= 64 + log2(m) bits of magic
// make this exact for every 64-bit x.
struct FastMod {
    uint64_t mh, ml;  // M = mh * 2^64 + ml
    uint64_t qinv;    // m = q * 2^k with q odd: q^-1 mod 2^64
    uint64_t lim;     // floor((2^64 - 1) / m)
    uint32_t m;
    uint32_t k;
};

__host__ __device__ __forceinline__ uint64_t mulhi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

inline FastMod make_fastmod(uint32_t m) {
    FastMod f{0, 0, 0, 0, m, 0};
    if (m >= 2) {
        // divisibility test constants: the odd part's inverse by Newton's iteration (q*q = 1 mod 8
        // gives 3 correct bits; each step doubles them), and the largest quotient
        uint32_t k = 0;
        while (((m >> k) & 1u) == 0u) ++k;
        const uint64_t q = m >> k;
        uint64_t inv = q;
        for (int it = 0; it < 6; ++it) inv *= 2u - q * inv;
        f.qinv = inv;
        f.k = k;
        f.lim = ~0ull / m;
        // floor((2^128 - 1) / m) + 1, by long division of the all-ones 128-bit value
        const uint64_t ones = ~0ull;
        const uint64_t qh = ones / m, rh = ones % m;
        const unsigned __int128 low = ((unsigned __int128)rh << 64) | ones;
        const uint64_t ql = (uint64_t)(low / m);
        f.ml = ql + 1;
        f.mh = qh + (f.ml == 0 ? 1 : 0);
    }
    return f;
}

__host__ __device__ __forceinline__ uint32_t fast_mod(uint64_t x, const FastMod& f) {
    if (f.m < 2) return 0u;
    const uint64_t ll = f.ml * x;                        // low 128 bits of M * x: (lh, ll)
    const uint64_t lh = mulhi64(f.ml, x) + f.mh * x;
    const uint64_t a = lh * (uint64_t)f.m;               // (lh, ll) * m >> 128
    const uint64_t b = mulhi64(ll, (uint64_t)f.m);
    return (uint32_t)(mulhi64(lh, (uint64_t)f.m) + ((a + b) < a ? 1u : 0u));
}

// x mod m == j for j < m, without forming the remainder: x >= j and n = x - j divisible by m.  With
// m = q * 2^k (q odd), n is a multiple of m exactly when (n * q^-1 mod 2^64) rotated right by k is at
// most floor((2^64 - 1) / m) (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994, Section 9): one 64-bit multiply instead of a remainder.
// mod_equals_in_range assumes m >= 2 and j < m; mod_equals takes any m and j.
__host__ __device__ __forceinline__ bool mod_equals_in_range(uint64_t x, uint32_t j, const FastMod& f) {
    if (x < j) return false;
    const uint64_t y = (x - j) * f.qinv;
#ifdef __CUDA_ARCH__
    // rotate right by k < 32 (m < 2^32): each half is a funnel shift of the two halves
    const uint32_t lo = (uint32_t)y, hi = (uint32_t)(y >> 32);
    const uint64_t r = ((uint64_t)__funnelshift_r(hi, lo, f.k) << 32) | __funnelshift_r(lo, hi, f.k);
#else
    const uint64_t r = (y >> f.k) | (y << ((64u - f.k) & 63u));
#endif
    return r <= f.lim;
}

// The same test without a branch: every lane forms the product, so lanes of a warp never part ways
// over it (x - j wraps when x < j, and the first factor then makes the result false).
__host__ __device__ __forceinline__ bool mod_equals_nobranch(uint64_t x, uint32_t j, const FastMod& f) {
    const uint64_t y = (x - j) * f.qinv;
#ifdef __CUDA_ARCH__
    const uint32_t lo = (uint32_t)y, hi = (uint32_t)(y >> 32);
    const uint64_t r = ((uint64_t)__funnelshift_r(hi, lo, f.k) << 32) | __funnelshift_r(lo, hi, f.k);
#else
    const uint64_t r = (y >> f.k) | (y << ((64u - f.k) & 63u));
#endif
    return (x >= j) & (r <= f.lim);
}

__host__ __device__ __forceinline__ bool mod_equals(uint64_t x, uint32_t j, const FastMod& f) {
    if (f.m < 2) return j == 0u;
    if (j >= f.m) return false;
    return mod_equals_in_range(x, j, f);
}

struct Ctrl {
    unsigned long long n_touched;   // nodes in touched[] this batch
    unsigned long long need_quads;  // table space requested by this batch, in 4-slot units
    unsigned long long pool_top;    // 4-slot units handed out so far
    unsigned long long self_loops;
    unsigned long long stored;      // stored (kept) edges
    unsigned int status;
    unsigned int n_giant;  // nodes whose table k_rehash_huge moves in pieces, many blocks each
    // work counters of k_intersect<true> (see rept_stats)
    unsigned long long small_entries, small_slots, probes, probe_slots, wedges, counted;
    unsigned long long class_items[kClasses], class_probes[kClasses], class_cycles[kClasses];
    // per-batch work lists of the intersection
    unsigned long long n_groups;           // larger endpoints of grouped edges (glist)
    unsigned long long n_items;            // grouped edges with a place in order[]
    unsigned long long bin_count[kBins];   // small chunks and units of each kind
    unsigned long long bin_next[kBins];    // claimed so far
    unsigned long long n_pairs;  // entries of pair_list this batch
    unsigned long long n_big;   // nodes whose table k_rehash_big moves, a warp each
    unsigned long long n_huge;  // nodes whose table k_rehash_huge moves, a block each
    unsigned long long huge_next;
    unsigned long long layout_quads;  // quads of all blocks in the layout that k_layout_quads was asked for
    unsigned long long dbg[4];  // REPT_DEBUG_BOUNDS builds: first failed check {site, index, bound}, count
};

// What the intersection needs about one arriving edge t = (s, l), s the endpoint with the smaller
// table: both tables' offsets (in 4-slot units) and sizes, written by k_insert once the batch's tables
// are final.  Record e belongs to the batch's edge e.
struct __align__(16) WorkItem {
    uint32_t s, l, off_s, off_l;
    uint32_t t;      // stream index of the edge
    uint32_t lgs;    // log2 table sizes: smaller | larger << 8
    uint32_t cnt_s;  // entries of the smaller endpoint
    uint32_t cnt_l;  // entries of the larger endpoint
};

// Edges order[first .. first + count) of one larger endpoint.
struct __align__(8) Unit {
    uint32_t first, count;
};

// Scratch bytes per batch edge of the work lists beside the records: two unit lists, order, mark,
// glist.
constexpr unsigned long long kListBytes = 3ull * sizeof(uint32_t) + 2ull * sizeof(Unit);

// Everything a kernel needs to know about one stream's state.
struct StreamDev {
    uint32_t m, c, groups, n_nodes;
    uint64_t seed;
    FastMod fm;         // x mod m
    uint4* meta;  // per node {block offset in 4-slot units, entries, 0, grouped edges of this batch with this
                  // larger endpoint, then their cursor into order[]}; the last is zero between batches
    uint32_t* cnt_add;  // [n_nodes] new entries per node as k_classify counts them (a compact array, so
                        // that its atomics stay in L2); k_plan takes each touched node's count and clears
                        // it, so it is zero between batches
    uint2* pool;
    unsigned long long pool_quads;
    // How list entries carry their edge's colours (the intersection tests colours before it probes):
    // kColNone: not at all; kColInEntry: every list entry w of node x carries h_0(x, w) in its top 8
    // bits (w itself in the low kIdBits), for one hash group, 2 <= m <= 256 and n_nodes <= 2^kIdBits;
    // kColWords: a parallel array of 32-bit words beside the list holds h_0(x, w), for one hash group
    // otherwise; kColMulti: several hash groups, a 32-bit word beside every stream index in tables and
    // lists holds h_k(x, w) of every group k in bits [k * cbits, (k + 1) * cbits) or, when a group
    // keeps colour 0 only (parallel MASCOT), one bit per group that is set if it keeps the edge
    uint32_t colours;
    uint32_t cbits;  // kColWords, kColMulti: bits per group colour
    uint32_t cmask;  // (1 << cbits) - 1
    uint32_t ctop;   // kColMulti: the top bit of every group's colour (groups of this state only)
    unsigned long long* local;
    unsigned long long* proc;
    uint32_t* touched;
    uint32_t* grow_rel;
    struct WorkItem* rec;   // [max_batch] work record of each edge that can close wedges
    uint32_t* mark;         // [max_batch] per edge: its larger endpoint (grouped), kSmallEdge or kNoWork
    uint32_t* order;        // [max_batch] grouped edges, those of one larger endpoint side by side
    uint32_t* glist;        // [max_batch] larger endpoints with grouped edges
    struct Unit* units;     // [2 * max_batch] first half: the largest l's block units from the front and
                            // warp units from the back; second half: the other block units
    unsigned long long unit_cap;  // max_batch
    uint32_t* big;      // [big_cap] touched-list indices of nodes with a large table to move: the
                        // k_rehash_big list from the front, the k_rehash_huge list from the back
    unsigned long long big_cap;
    Ctrl* ctrl;
    // c > m with c mod m != 0 (Algorithm 2): the partial group's local counts and the triangle-pair
    // counters; all NULL otherwise
    uint32_t c1;                    // full groups: processors i < c1 * m feed `local`, the rest `local2`
    uint32_t keep;                  // colours each hash group keeps: m (REPT), 1 (parallel MASCOT)
    uint32_t pstride;               // processors per hash group: m (REPT), 1 (parallel MASCOT)
    // colour sharding: this state keeps processors [pbeg, pbeg + pcount) only (all c by default),
    // which belong to hash groups [kbeg, kend)
    uint32_t pbeg, pcount, kbeg, kend;
    unsigned long long* local2;     // [n_nodes] sum of tau_v^(i) over the partial group
    unsigned long long* eta_proc;   // [c] eta^(i)
    unsigned long long* eta_local;  // [n_nodes] sum over processors of eta_v^(i)
    uint2* edge_ends;               // [pair_cap] endpoints of the stored edge with stream index t
    uint32_t* pair_tau;             // [pair_cap * groups] tau_(e)^(i) of edge e in group k (Algorithm 2)
    uint32_t* pair_evt;             // [pair_cap * groups] this batch's closed wedges through (e, k)
    uint32_t* pair_list;            // [pair_cap * groups] the (e, k) with events this batch: e * groups + k
    unsigned long long pair_cap;    // stream indices covered by the pair arrays
    unsigned long long* local_proc; // [c * n_nodes] tau_v^(i), processor-major (REPT_FLAG_LOCAL_PER_PROCESSOR)
};

// The work lists of n edges, one after the other from d.units on (kListBytes * n bytes).
inline void set_list_pointers(StreamDev& d, unsigned long long n) {
    d.unit_cap = n;
    d.order = reinterpret_cast<uint32_t*>(d.units + 2 * n);
    d.mark = d.order + n;
    d.glist = d.mark + n;
}

// The block a batch kernel's body runs as: its index among the nbx blocks that share one stream's
// work (blockIdx.x and gridDim.x for a launch per stream, or a virtual block of the persistent group
// kernel, which runs every step of the batch path for every stream of a group).
struct Grid {
    uint32_t bx, nbx;
};

// Grid-wide barrier state of the persistent group kernel (one per group, in device memory).  The
// host clears count and timed_out before each launch and sets extra: the arrivals a barrier waits for
// beyond the grid's blocks (0; a test sets 1 so that the wait can only run out).
struct GroupSync {
    unsigned int count;      // blocks arrived at the current barrier
    unsigned int gen;        // barriers completed (advanced by the last block to arrive)
    unsigned int timed_out;  // some block's wait gave up
    unsigned int extra;
};

// One batch of edges appended to a stream.
struct BatchDev {
    const uint32_t* src;
    const uint32_t* dst;
    unsigned long long n;
    unsigned long long t0;  // stream index of src[0], dst[0]
    uint32_t small_max;     // edges whose smaller endpoint has more entries are grouped
    uint32_t chunk;         // edges of a small chunk
    uint32_t unit_edges;    // edges of a block unit
};

// A batch of a stream.  Grouping pays through the lists that share a filter; in a small batch few do, so lists
// of up to kSmallBatchMax entries stay ungrouped there (`tile_max`: the handle's bound in other batches), and
// the edges are dealt out in smaller chunks.  Bound 256 and so: R-MAT of 2M edges in batches of 2^13, 2^14 and 2^15
// edges 23.3, 12.4, 8.2 ms and 22.1, 10.9, 6.5, five groups there 31.6, 18.6, 12.9 and 28.1, 14.6, 9.3; bound 32 the
// same, but 1 % slower in batches of 4,096.  The line at 2^14 or 2^16 for 2^15, chunks of half the edges: within 3 %;
// the other batches' chunk of 64 edges 1.2 to 2.5 times slower in batches of 4,096.  Block units hold fewer
// edges in smaller batches, so that there are units for every SM; the batches of a group's round (`round` edges
// together) fill the GPU together and so share their filters among more (48 streams, 65,536 edges each a round:
// 48.3 ms with units by the stream's own batch, 46.7 ms so).
inline BatchDev make_batch(const uint32_t* src, const uint32_t* dst, unsigned long long n, unsigned long long t0,
                           uint32_t tile_max, unsigned long long round) {
    const bool few = n < kSmallBatch;
    return BatchDev{src, dst, n, t0, few ? kSmallBatchMax : tile_max, few ? std::max((uint32_t)(n >> 10), 4u) : 64u,
                    (uint32_t)std::min(std::max(round >> 14, 16ull), (unsigned long long)kUnitItems)};
}

// Index checks of the REPT_DEBUG_BOUNDS build (a stand-in for a memory checker): a failed check
// records {site, index, bound} once, counts, raises kStBounds, and the caller skips the access.
// Release builds compile them away.
#ifdef REPT_DEBUG_BOUNDS
__device__ __forceinline__ bool dbg_ok(Ctrl* c, unsigned site, unsigned long long idx, unsigned long long bound) {
    if (idx < bound) return true;
    if (atomicAdd(&c->dbg[3], 1ull) == 0ull) {
        c->dbg[0] = site;
        c->dbg[1] = idx;
        c->dbg[2] = bound;
    }
    atomicOr(&c->status, kStBounds);
    return false;
}
#define REPT_CHECK(c, site, idx, bound) dbg_ok((c), (site), (idx), (bound))
#else
#define REPT_CHECK(c, site, idx, bound) true
#endif

// One output step of SplitMix64 from state x (Steele, Lea, Flood 2014).
__host__ __device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    uint64_t z = x + kGoldenGamma;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// h_k({a, b}) given the group seed s_k.
__device__ __forceinline__ uint32_t colour_of(uint32_t a, uint32_t b, uint64_t s_k, const FastMod& fm) {
    uint64_t lo = a < b ? a : b, hi = a < b ? b : a;
    return fast_mod(splitmix64(((lo << 32) | hi) ^ s_k), fm);
}

__device__ __forceinline__ uint64_t group_seed(uint64_t seed, uint32_t k) { return seed + (uint64_t)k * kGoldenGamma; }

// Do the wedge edges {s, w} and {l, w} have the same colour in the group of seed s_k?  Their hash
// values are congruent modulo m exactly when m divides their (exact, non-negative) difference, which
// the divisibility test decides without a remainder; only then is the colour j itself formed.
__device__ __forceinline__ bool same_colour(uint32_t s, uint32_t l, uint32_t w, uint64_t s_k, const FastMod& fm,
                                            uint32_t& j) {
    const uint64_t ks = ((uint64_t)(s < w ? s : w) << 32) | (s < w ? w : s);
    const uint64_t kl = ((uint64_t)(l < w ? l : w) << 32) | (l < w ? w : l);
    const uint64_t zs = splitmix64(ks ^ s_k), zl = splitmix64(kl ^ s_k);
    if (!mod_equals_nobranch(zs >= zl ? zs - zl : zl - zs, 0u, fm)) return false;
    j = fast_mod(zs, fm);
    return true;
}

// Is edge {u, v} kept by some processor (k*m + h_k(u,v) < c for some group k)?
// The processor that keeps colour j of hash group k, if any: REPT's processor i = k*m + j (i < c);
// parallel MASCOT's sampler i = k keeps colour 0 only (an independent p = 1/m sample per group).
// Only the processors of this state's shard count (pbeg + pcount <= c, so i < c as well).
__device__ __forceinline__ bool processor_of(const StreamDev& d, uint32_t k, uint32_t j, uint32_t& i) {
    i = k * d.pstride + j;
    return j < d.keep && i - d.pbeg < d.pcount;
}

__device__ __forceinline__ bool kept_by_any(const StreamDev& d, uint32_t u, uint32_t v) {
    for (uint32_t k = d.kbeg; k < d.kend; ++k) {
        uint32_t i, j = colour_of(u, v, group_seed(d.seed, k), d.fm);
        if (processor_of(d, k, j, i)) return true;
    }
    return false;
}

constexpr uint32_t kColNone = 0u, kColInEntry = 1u, kColWords = 2u, kColMulti = 3u;

// The mask that takes a node id out of the first word of a list entry.
__host__ __device__ __forceinline__ uint32_t id_mask(const StreamDev& d) {
    return d.colours == kColInEntry ? kIdMask : ~0u;
}
// Single-group streams with colours keep interleaved tables (key_word).
__host__ __device__ __forceinline__ bool interleaved(uint32_t colours) {
    return colours == kColInEntry || colours == kColWords;
}

// With one hash group, a wedge (s, w), (l, w) can count only if h_0(s, w) = h_0(l, w) = js for a kept
// colour js.  js is stored with s's list entry; this asks the same of the hash of {l, w} alone, as a
// superset test: it never rejects an entry whose wedge can count, and may pass a few whose wedge cannot;
// count_wedge decides every queued wedge exactly.  z mod m = js implies that m divides z - js, i.e. that
// r = rotr((z - js) q^-1, k) <= floor((2^64 - 1) / m); only the high words are compared (a pass rate of
// about 1/m + 2^-32).  Every entry of a list carries a kept colour (its edge is stored because this
// state's processor of that colour keeps it), and z < js, which the exact test excludes, has
// probability below 2^-56.
__device__ __forceinline__ bool colour_may_match(const StreamDev& d, uint32_t l, uint32_t w, uint32_t js) {
    const uint64_t lo = l < w ? l : w, hi = l < w ? w : l;
    const uint64_t z = splitmix64(((lo << 32) | hi) ^ d.seed);
    const uint64_t y = (z - js) * d.fm.qinv;
    const uint32_t r_hi = __funnelshift_r((uint32_t)(y >> 32), (uint32_t)y, d.fm.k);
    return r_hi <= (uint32_t)(d.fm.lim >> 32);
}

// The colour word of edge {u, v} (kColWords, kColMulti) and, in `kept`, whether some processor keeps it.
__device__ __forceinline__ uint32_t colour_word(const StreamDev& d, uint32_t u, uint32_t v, bool& kept) {
    uint32_t cw = 0;
    bool any = false;
    uint64_t sk = group_seed(d.seed, d.kbeg);
    for (uint32_t k = d.kbeg; k < d.kend; ++k, sk += kGoldenGamma) {
        uint32_t i;
        const uint32_t j = colour_of(u, v, sk, d.fm);
        const bool keeps = processor_of(d, k, j, i);
        cw |= (d.keep == 1u ? (keeps ? 1u : 0u) : j) << (k * d.cbits);
        any |= keeps;
    }
    kept = any;
    return cw;
}

// log2 of the table capacity for cnt entries: capacity = max(4, nextpow2(2*cnt)); 0 when empty.
__host__ __device__ __forceinline__ uint32_t table_lg(uint32_t cnt) {
    if (cnt == 0) return 0;
    uint32_t x = 2u * cnt - 1u;  // ceil(log2(2*cnt)) = bit length of (2*cnt - 1)
#ifdef __CUDA_ARCH__
    uint32_t lg = 32u - __clz(x);
#else
    uint32_t lg = 32u - (uint32_t)__builtin_clz(x);
#endif
    return lg < 2u ? 2u : lg;
}

// A node's block in the pool, 32-byte aligned, in 32-bit words: its hash table of 2^lg slots
// (2 words a slot, 3 with kColMulti; key_word, eidx_of), then its list: list_slots(lg) entry words
// (id and, with kColInEntry, colour) in insertion order, followed by their stream indices (kColNone) or
// {stream index, colour word} pairs (kColMulti); single-group streams leave that part unused (a
// candidate's age is looked up in the table) and, with kColWords, keep the colour words after it.
__host__ __device__ __forceinline__ uint32_t list_slots(uint32_t lg) { return lg >= 3u ? (1u << (lg - 1u)) : 4u; }
__host__ __device__ __forceinline__ uint32_t word_slots(uint32_t lg) { return lg >= 4u ? (1u << (lg - 2u)) : 4u; }
__host__ __device__ __forceinline__ uint32_t block_quads(uint32_t lg, uint32_t colours) {
    const uint32_t slots = (1u << lg) + list_slots(lg);
    if (colours == kColMulti) return (uint32_t)((3ull * slots + 7ull) >> 3);
    return (slots + (colours == kColWords ? word_slots(lg) : 0u)) >> 2;
}

// Offsets of blocks are 32-bit quads.
constexpr unsigned long long kMaxQuads = 0xFFFFFFFFull;

// Pool quads that guarantee no batch can run out: a node's block holds at most 2 quads per entry (3 with
// colour words: at one entry, less beyond), and its successive blocks form a doubling series bounded by
// twice the last one, so at most 4 (6) quads per stored entry, i.e. 8 (12) per stream edge.
inline unsigned long long quads_bound(unsigned long long edges, uint32_t colours) {
    return (colours == kColWords || colours == kColMulti ? 12ull : 8ull) * edges + 64ull;
}

// How a configuration stores its colours (StreamDev::colours) where the pool has room, and the bits of a
// colour word that each hash group takes.  kColMulti is the one layout that a handle may do without.
inline uint32_t widest_colours(uint32_t m, uint32_t c, uint32_t n_nodes, bool mascot, uint32_t& bits) {
    const uint64_t groups = mascot ? c : ((uint64_t)c + m - 1u) / m;
    bits = 0;
    while (bits < 32u && (1ull << bits) < m) ++bits;
    if (groups == 1u && m >= 2u) {
        if (m <= 256u && n_nodes <= (1u << kIdBits)) return kColInEntry;
        if (!mascot) return kColWords;
    }
    if (mascot || m == 1u) bits = 1u;  // a bit per group that keeps the edge
    return groups * bits <= 32u ? kColMulti : kColNone;
}

// May a pool of `quads` quads hold the colour words of several groups, when its handle can have `memory` bytes
// and blocks can start at `most` quads at most?  The words make the pool half as large again, and a stream
// that outgrows it with them is taken over into a pool without them, which for twice the entries is 4/3 as
// large: both have to fit side by side.
inline bool words_fit(unsigned long long quads, unsigned long long memory, unsigned long long most) {
    return quads <= most && quads <= memory / 32ull && 7ull * 32ull * quads / 3ull <= memory;
}

// Where the list of a block with a table of 2^lg slots starts, the stream indices or pairs beside it (kColNone,
// kColMulti), and its colour words (kColWords).  A block of 2^30 slots (a node of more than 2^28 entries)
// is longer than 2^32 words, so the offsets are 64 bits wide.  (32-bit offsets, which wrap there: intersection of
// partial groups, 2M edges, 1.23 ms and 1.25 ms so, R-MAT scale 20 5.48 and 5.48; counted in 16-byte
// units in 32 bits 1.26 and 5.51.)
template <class Word>
__host__ __device__ __forceinline__ Word* list_of(Word* block, uint32_t lg, uint32_t colours) {
    return block + ((colours == kColMulti ? 3ull : 2ull) << lg);
}
template <class Word>
__host__ __device__ __forceinline__ Word* aux_of(Word* block, uint32_t lg, uint32_t colours) {
    return list_of(block, lg, colours) + list_slots(lg);
}
template <class Word>
__host__ __device__ __forceinline__ Word* cw_of(Word* block, uint32_t lg) {
    return block + 2ull * ((1u << lg) + list_slots(lg));
}

// Work-counter class of an edge whose smaller endpoint holds cnt entries (rept_stats.class_*).
__host__ __device__ __forceinline__ int bin_of_cnt(uint32_t cnt) {
    return cnt <= 4u ? 0 : cnt <= 8u ? 1 : cnt <= 16u ? 2 : cnt <= 32u ? 3 : cnt <= 256u ? 4 : 5;
}

// Does a filter of the larger endpoint's list of n entries pay for a block unit's lists of `scanned` entries
// together?  Building costs each of the n entries about as much as a test, and past one entry per bit or so the
// filter lets most entries through.  Without it an entry costs a hash (one group's stored colours) or is looked
// up at once (else), so that the line lies elsewhere.  Passes of a Chung-Lu graph with hubs of a million (40M
// edges, m = c = 100; filter always, so): batches of 2^14 edges 798 and 312 ms, 2^16 283 and 116, 2^20 66 and 32;
// five groups there, 2^18 165 and 160.  R-MAT scale 20: 10.86 and 10.92.  Half and twice the numbers: within
// 2 %, but 65,536 for 24,576 347 ms at 2^14.  (In warp units too, the first three took 3 % less and the groups'
// kernels spilled for it: 48 streams 47.3 and 48.6 ms.)
__host__ __device__ __forceinline__ bool filter_pays(uint32_t colours, uint32_t n, unsigned long long scanned) {
    return interleaved(colours) ? n <= 24576u && n <= 4ull * scanned : n <= 262144u && n <= 16ull * scanned;
}

// Home slot of neighbour w in a table of 2^lg slots: the first slot of a 4-slot (32-byte) bucket
// chosen by Fibonacci hashing.  Probing is linear from there, so a lookup reads whole sectors.
__device__ __forceinline__ uint32_t home_slot(uint32_t w, uint32_t lg) {
    return ((w * 0x9E3779B1u) >> (32u - lg)) & ~3u;
}

// The word offset, from the start of a table of 2^lg slots, of slot h's neighbour id, and the place of its
// stream index.  Interleaved tables: bucket h / 4 occupies words 8 (h / 4) .. 8 (h / 4) + 7, ids first.
// Others: ids in words 0 .. 2^lg - 1, then the stream indices (with kColMulti, each followed by its
// colour word).  key_quad: the 16-byte quad that holds the four ids of the bucket that starts at slot h
// (h a multiple of 4).
__host__ __device__ __forceinline__ uint32_t key_word(uint32_t h, uint32_t colours) {
    return interleaved(colours) ? (((h >> 2) << 3) | (h & 3u)) : h;
}
template <class Word>
__host__ __device__ __forceinline__ Word* eidx_of(Word* table, uint32_t h, uint32_t lg, uint32_t colours) {
    if (interleaved(colours)) return table + (key_word(h, colours) + 4u);
    return colours == kColMulti ? table + (1u << lg) + 2ull * h : table + ((1u << lg) + h);
}
__host__ __device__ __forceinline__ uint32_t key_quad(uint32_t h, uint32_t colours) {
    return interleaved(colours) ? h >> 1 : h >> 2;
}

// Warp-aggregated atomicAdd: every active lane of the full warp calls it with its own
// increment; returns the lane's exclusive offset from a single atomic per warp.
__device__ __forceinline__ unsigned long long warp_reserve(unsigned long long* ctr, unsigned long long inc) {
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long incl = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned long long y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (unsigned)o) incl += y;
    }
    unsigned long long total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    unsigned long long base = 0;
    if (lane == 31 && total) base = atomicAdd(ctr, total);
    base = __shfl_sync(0xFFFFFFFFu, base, 31);
    return base + incl - inc;
}

// The same for lanes that each take one place or none.
__device__ __forceinline__ unsigned long long warp_reserve_one(unsigned long long* ctr, bool take) {
    const unsigned lane = threadIdx.x & 31u, mask = __ballot_sync(0xFFFFFFFFu, take);
    unsigned long long base = 0;
    if (lane == 0 && mask) base = atomicAdd(ctr, (unsigned long long)__popc(mask));
    return __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(mask & ((1u << lane) - 1u));
}

// The same for a thread block (at most 32 warps; every thread calls it): one atomic per block.  The
// atomics of a grid on one counter follow each other about 1.3 ns apart, so a warp's each for 2^20
// edges takes 40 us.  `part`: shared memory of the caller, two of them used in turn need no barrier
// between calls.  Sum: wide enough for the sum of a block's requests.
template <class Sum>
struct BlockReserve {
    Sum warp[32];
    unsigned long long base;
};
template <class Sum>
__device__ __forceinline__ unsigned long long block_reserve(BlockReserve<Sum>& part, unsigned long long* ctr, uint32_t inc) {
    const unsigned lane = threadIdx.x & 31u, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
    Sum incl = inc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Sum y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (unsigned)o) incl += y;
    }
    if (lane == 31) part.warp[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const Sum w = lane < warps ? part.warp[lane] : 0u;
        Sum wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const Sum y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
            if (lane >= (unsigned)o) wi += y;
        }
        part.warp[lane] = wi - w;
        if (lane == 31) part.base = wi ? atomicAdd(ctr, (unsigned long long)wi) : 0ull;
    }
    __syncthreads();
    return part.base + part.warp[wid] + incl - inc;
}

}  // namespace rept
