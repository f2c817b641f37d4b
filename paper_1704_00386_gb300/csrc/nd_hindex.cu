// The iterated h-index update (Def. 4) as GPU passes: SND (Alg. 2) and AND
// with or without notification (Alg. 3, Section 4.3).
//
// One pass = one launch of a persistent grid.  R-cliques are grouped into
// four degree buckets (by default d_s in [1,8], [9,64], [65,2048], >2048)
// and evaluated by a group of 4 or 8 lanes, a warp, or a whole CTA.  The CTA
// rows are taken one per block from a per-pass counter; the rest are warp
// tasks, taken in chunks of consecutive tasks per warp from a second
// counter.  A group of 4 or 8:
//   1. streams the r-clique's incidence row (coalesced, q ids per s-clique),
//      gathers the q tau values of each s-clique and keeps
//      rho = min(...) in registers (Def. 4, step 1);
//   2. counts rho >= tau(R).  If at least tau(R) of them are, H = tau(R):
//      the preserve-tau early exit of Section 4.4, valid because the update
//      never raises tau (Thm. 1);
//   3. otherwise H lies in [count, tau(R)) and is found by binary search on
//      h over the register-resident rho values, testing
//      #{rho >= h} >= h (Def. 3).  No histogram, no sort.
// A warp or a CTA (longer rows) streams its row instead (warp_hindex): it
// counts rho >= tau(R) and stops at tau(R) of them; a row that fails, or is
// expected to, goes through a shared-memory histogram of rho over the values
// that can be H, whose suffix sums give H.
// (The routines that search a row are in nd_search.cuh.)
// What bounds a pass: the L1 wavefronts of the gathers, and in the early
// passes the instructions of the search.  R-MAT scale-20 k-truss (1.17G
// incidences), SND to convergence in 57 passes: 109.0 ms, against 184.3 ms
// with 64-bit row offsets, a runtime division per binned value, whole rows
// read in every pass and 16-bit values cached in shared memory between a
// count and its search; AND 48.0 against 72.9 ms, AND-nn 64.4 against 105.8.
// The paper's linear-time hashmap h-index (Section 4.4) is replaced by this
// tau-bounded count; both compute Def. 3 exactly.
//
// SND reads tau_p and writes tau (ping-pong buffers, no copy).  AND reads and
// writes one tau array in place; tau only decreases, so a stale read is a
// larger value and at worst delays a decrease by a pass.  With notification, an
// r-clique is evaluated only if its bit is set in the current frontier; when
// its tau drops to h it sets the next-frontier bit of every neighbour R' with
// h <= tau(R') (Alg. 3, the orange lines).  It does not re-activate itself.
//
// (2,3) uses the adjacency layout: incidence entries are the CSR slots of
// the other two edges, the gathers read a 16-bit copy of tau indexed by CSR
// slot, and the frontier has one bit per slot.  (3,4) does the same with the
// slots of the edges' triangle lists, three per triangle.  k_pass_otf is the same update
// with no stored incidence: it finds each edge's triangles again by
// intersecting adjacency lists on every pass.
#include "nd_internal.cuh"
#include "nd_search.cuh"

namespace {

#ifndef ND_WARP_CHUNK
#define ND_WARP_CHUNK 16  // consecutive warp tasks per counter grab
#endif
constexpr int kWarpChunk = ND_WARP_CHUNK;  // at most: warp_chunk
#ifndef ND_NOTIFY_UNROLL
#define ND_NOTIFY_UNROLL 4  // notification entries in flight per lane ((2,3))
#endif
constexpr int kNotifyUnroll = ND_NOTIFY_UNROLL;
#ifndef ND_FRONT_L1
#define ND_FRONT_L1 1  // 0: read the next frontier's words from L2 only
#endif

// a word of the next frontier, which this pass only sets bits in: read
// through L1, where a stale clear bit only costs a redundant, idempotent
// atomic (a set bit is never stale).  Measured against L2-only reads: the
// k-core AND of R-MAT scale 24 took 73.8 against 89.9 ms, where the frontier
// words of the hub vertices are read again and again; the truss and (3,4)
// AND did not change.
__device__ __forceinline__ uint32_t ld_front(const uint32_t* p) {
#if ND_FRONT_L1
    return __ldca(p);
#else
    return __ldcg(p);
#endif
}
// histogram words per warp: 512 bins in the passes where most rows search, 256
// in the late ones.  Every KB of them is taken from L1 and its gathers.
// Measured (R-MAT scale-20 k-truss / scale-24 k-core / Chung-Lu 100K (3,4)):
// the first 16 SND passes 43.2 / 24.0 / 18.6 ms with 256 words, 44.0 / 25.7 /
// 20.3 with 512; passes 17-32 28.3 / 20.7 / 17.8 ms with 128 words, 29.0 /
// 20.5 / 17.5 with 256.
constexpr int kHistWords = 256;
constexpr int kLateHistWords = 128;
static_assert(kHistWords % 128 == 0 && kLateHistWords % 128 == 0, "cleared and selected in blocks of 128 words");

// The kinds of incidence rows a pass kernel is built for: Q = 1, 2, 3 for
// (1,2), (2,3) and (3,4) in the layouts above; kIds for a (3,4) handle whose
// entries are triangle ids.
constexpr int kIds = 4;
// ids per entry; (3,4) rows hold them as three runs of d words, so that a warp
// loads 32 entries with three coalesced loads
template <int Q>
constexpr int kWords = Q == kIds ? 3 : Q;
// are the ids slots?
template <int Q>
constexpr bool kSlots = Q == 2 || Q == 3;

// Work of one pass: rows longer than the CTA threshold are taken one per
// block from a per-pass counter; all other rows form warp tasks that warps
// take in chunks from a second counter.

struct SweepParams {
    const uint32_t* __restrict__ inc;
    const int32_t* tin;   // SND: tau of the previous pass; AND: same array as tout
    int32_t* tout;
    // gathers: a copy of tau in 16 bits saturated at 65535, exact for every
    // row with tau(R) <= 65535 (the row only looks at min(rho, tau(R))); a
    // row above that (a CTA row) gathers tin.  Indexed by slot for (2,3) and
    // (3,4), where an updated r-clique writes all of its slots (epos, tpos), and
    // by vertex for (1,2); kIds gathers tin.
    const uint16_t* gin;
    uint16_t* gout;
    const uint2* __restrict__ epos;     // (2,3): the two slots of an edge
    const uint32_t* __restrict__ tpos;  // (3,4): the three slots of a triangle
    const uint32_t* __restrict__ eid;   // slot -> r-clique
    // (2,3) without a stored incidence: the graph and the edge endpoints
    const int64_t* __restrict__ rp;
    const int32_t* __restrict__ col;
    const int32_t* __restrict__ eu;
    const int32_t* __restrict__ ev;
    const int32_t* __restrict__ hub_of;  // hub index of a vertex, -1 for the others; null: no hub tables
    const uint2* __restrict__ hub_bits;  // per hub hub_words x (neighbour bits of 32 ids, neighbours below them)
    int64_t hub_words;
    const int32_t* __restrict__ by_degree;  // with hub tables: the adjacency lists by degree class, and
    const uint32_t* __restrict__ slot_of;   // the CSR slot of every entry
    bool bounded;                           // tau <= d_s throughout: a run from d_s
    const nd_item* __restrict__ items;
    int64_t lo[ND_NB], hi[ND_NB];  // bucket ranges in items
    int chunk;                     // warp tasks per counter grab (warp_chunk)
    bool direct;                   // AND: rows are expected to fail the count (see warp_hindex)
    const uint32_t* cur;  // AND + notification: frontier read in this pass
    uint32_t* next;       // and the frontier written for the next pass
    uint32_t* spare;      // INLINE: the one of the pass after that, to be cleared
    int64_t spare_words;
    // relabelled (1,2) runs from d_s: the largest degree, so the largest tau, of
    // the ids from 2^o on; rows are ordered by floor(log2 id).  Null: no bound
    const int32_t* __restrict__ oct_max;
    const uint32_t* members;  // PartialAnd: only members are notified (null = everyone)
    // batches, SND and AND-nn: graph of every r-clique, the graphs that changed
    // in the previous pass (gact_in) and those changing in this one (gact_out);
    // null for a single graph
    const uint32_t* __restrict__ gid;
    const uint8_t* gact_in;
    uint8_t* gact_out;
    // AND with notification and batches: the active work items, and where each
    // bucket's begin there (their numbers are in ctr)
    const uint32_t* __restrict__ list;
    int64_t list_lo[ND_NB];
    unsigned long long* ctr;         // this pass's counters (ND_CTR_*)
    const unsigned long long* prev;  // previous pass (null on the first)
};

// tau loads.  SND reads last pass's array through the read-only path.  AND
// reads the array it is updating with plain (L1-cacheable) loads: a value
// seen early or from another SM's stale line is never smaller than the true
// one, because tau only decreases, so it can only delay a decrease to a later
// pass (the writer notifies) or over-notify; every pass is a new launch, which
// starts from fresh caches.
template <bool RO>
__device__ __forceinline__ int32_t ld_tau(const int32_t* p) {
    if (RO) return __ldg(p);
    return *p;
}

template <bool RO>
__device__ __forceinline__ int32_t ld_tau(const uint16_t* p) {
    if (RO) return (int32_t)__ldg(p);
    return (int32_t)*p;
}

// rho(S,R) for the s-clique at incidence j: min of the other r-cliques' tau
// (for (2,3) the entries index the CSR-position copy of tau).
// SND reads each row once per pass, so its ids are loaded evict-first and do
// not push the gathered tau values out of L2.  AND re-reads the row of a
// changed r-clique to notify its neighbours, so its ids are cached normally.
template <bool RO>
__device__ __forceinline__ uint32_t ld_id(const uint32_t* p) {
    return RO ? __ldcs(p) : __ldg(p);
}

// rho of entry j of a row, as a functor for the h-index routines below: the
// row's base address once, 32-bit offsets from it (the passes are bound by
// instructions as much as by the gathers; 64-bit offsets per entry cost both
// registers and issue slots)
template <int Q, bool RO, typename T>
struct Rho {
    static constexpr bool kCarry = RO && Q != 2;  // see warp_hindex
    const uint32_t* __restrict__ row;
    int d;  // (3,4): the length of the row's runs
    const T* tau;
    __device__ __forceinline__ int32_t operator()(int j) const {
        if constexpr (Q == 1) {
            return ld_tau<RO>(tau + ld_id<RO>(row + j));
        } else if constexpr (Q == 2) {
            const uint2* p = reinterpret_cast<const uint2*>(row) + j;
            const uint2 id = RO ? __ldcs(p) : __ldg(p);
            return min(ld_tau<RO>(tau + id.x), ld_tau<RO>(tau + id.y));
        } else {
            const uint32_t* p = row + j;
            const uint32_t a = ld_id<RO>(p), b = ld_id<RO>(p + d), c = ld_id<RO>(p + 2 * (int64_t)d);
            return min(min(ld_tau<RO>(tau + a), ld_tau<RO>(tau + b)), ld_tau<RO>(tau + c));
        }
    }
};

// rows of slots with tau(R) > 65535 (so d_s > 65535, CTA rows): exact values,
// slot -> r-clique -> tau
template <int Q, bool RO>
struct RhoExact {
    static constexpr bool kCarry = RO && Q != 2;
    const uint32_t* __restrict__ row;
    int d;
    const uint32_t* __restrict__ eid;
    const int32_t* tau;
    __device__ __forceinline__ int32_t operator()(int j) const {
        if constexpr (Q == 2) {
            const uint2 id = __ldg(reinterpret_cast<const uint2*>(row) + j);
            return min(ld_tau<RO>(tau + __ldg(eid + id.x)), ld_tau<RO>(tau + __ldg(eid + id.y)));
        } else {
            const uint32_t* p = row + j;
            return min(min(ld_tau<RO>(tau + __ldg(eid + __ldg(p))), ld_tau<RO>(tau + __ldg(eid + __ldg(p + d)))),
                       ld_tau<RO>(tau + __ldg(eid + __ldg(p + 2 * (int64_t)d))));
        }
    }
};

constexpr int32_t kTau16Max = 65535;

// the row of a work item
template <int Q>
__device__ __forceinline__ const uint32_t* row_of(const SweepParams& P, int64_t jb) {
    return P.inc + kWords<Q> * jb;
}

// the gather of a row whose tau is at most 65535: the 16-bit copy, or the
// int32 values where entries are r-clique ids in no order (kIds)
template <int Q, bool RO>
__device__ __forceinline__ auto make_rho(const SweepParams& P, int64_t jb, uint32_t d) {
    if constexpr (Q == kIds) return Rho<3, RO, int32_t>{row_of<Q>(P, jb), (int)d, P.tin};
    else return Rho<Q, RO, uint16_t>{row_of<Q>(P, jb), (int)d, P.gin};
}

// the new tau of R, also written to all of its slots.
// SND writes the buffer of two passes ago: where that holds h already (old),
// all its copies do, and nothing is written.
template <int Q>
__device__ __forceinline__ void store_tau(const SweepParams& P, uint32_t R, int32_t h, int32_t old) {
    if (h == old) return;
    P.tout[R] = h;
    const uint16_t v = (uint16_t)min(h, kTau16Max);
    if (Q == 2) {
        const uint2 ep = __ldg(P.epos + R);
        P.gout[ep.x] = v;
        P.gout[ep.y] = v;
    } else if (Q == 3) {
#pragma unroll
        for (int k = 0; k < 3; ++k) P.gout[__ldg(P.tpos + 3 * (int64_t)R + k)] = v;
    } else if (Q == 1) {
        P.gout[R] = v;
    }
}

// notify the r-clique at slot pos, whose tau read from the 16-bit copy is tv,
// if h <= tau (the exact int32 value when h > 65535).
// The caller has just seen its frontier bit clear, with a relaxed L2 read:
// a bit set meanwhile only costs a redundant atomic, and a set bit is never
// cleared within a pass.
__device__ __forceinline__ void notify_clear(const SweepParams& P, uint32_t pos, int32_t h, int32_t tv) {
    if (h > kTau16Max) tv = ld_tau<false>(P.tin + __ldg(P.eid + pos));
    if (h > tv) return;
    if (P.members) {  // PartialAnd: members only
        const uint32_t Rp = __ldg(P.eid + pos);
        if (!((__ldg(P.members + (Rp >> 5)) >> (Rp & 31)) & 1u)) return;
    }
    atomicOr(P.next + (pos >> 5), 1u << (pos & 31));
}

// the same, testing the bit first and reading tau only if it is clear
__device__ __forceinline__ void notify_pos(const SweepParams& P, uint32_t pos, int32_t h) {
    if ((ld_front(P.next + (pos >> 5)) >> (pos & 31)) & 1u) return;
    notify_clear(P, pos, h, ld_tau<false>(P.gin + pos));
}

__device__ __forceinline__ unsigned front_bit(const uint32_t* f, uint32_t i) {
    return (__ldg(f + (i >> 5)) >> (i & 31)) & 1u;
}

// is R in the current frontier?  With slots: any bit of its slots
template <int Q>
__device__ __forceinline__ bool in_frontier(const SweepParams& P, uint32_t R) {
    if constexpr (Q == 2) {
        const uint2 ep = __ldg(P.epos + R);
        return front_bit(P.cur, ep.x) | front_bit(P.cur, ep.y);
    } else if constexpr (Q == 3) {
        const uint32_t* p = P.tpos + 3 * (int64_t)R;
        const uint32_t a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
        return front_bit(P.cur, a) | front_bit(P.cur, b) | front_bit(P.cur, c);
    } else {
        return front_bit(P.cur, R);
    }
}

// the ids of entry j of a row of d entries
template <int Q>
__device__ __forceinline__ void entry_ids(const uint32_t* __restrict__ row, int d, int j,
                                          uint32_t (&id)[kWords<Q>]) {
    if constexpr (Q == 2) {
        const uint2 x = __ldg(reinterpret_cast<const uint2*>(row) + j);
        id[0] = x.x;
        id[1] = x.y;
    } else {
#pragma unroll
        for (int k = 0; k < kWords<Q>; ++k) id[k] = __ldg(row + j + (int64_t)k * d);
    }
}

// one neighbour whose next-frontier bit was clear: set it if h <= tau
template <int Q>
__device__ __forceinline__ void notify_one(const SweepParams& P, uint32_t id, int32_t h) {
    if constexpr (kSlots<Q>) {
        notify_clear(P, id, h, ld_tau<false>(P.gin + id));
    } else {
        const uint32_t bit = 1u << (id & 31);
        if (P.members && !(__ldg(P.members + (id >> 5)) & bit)) return;  // PartialAnd
        if (h <= ld_tau<false>(P.tin + id)) atomicOr(P.next + (id >> 5), bit);
    }
}

// U entries of one lane (ok: those that exist): which of their neighbours'
// next-frontier bits are clear, then those neighbours.  A neighbour whose bit
// is already set needs nothing, so the words (2 MB for 16M r-cliques,
// cache-resident) are read before any tau, all of them before any is tested,
// and one branch skips an entry block whose bits are all set, which most are.
// (Warp-wide merging of bits that share a word was measured slower: the match
// runs for every neighbour, while most neighbours need no write.)
template <int Q, int U>
__device__ __forceinline__ void notify_block(const SweepParams& P, const uint32_t (&id)[U][kWords<Q>],
                                             const bool (&ok)[U], int32_t h) {
    constexpr int W = kWords<Q>;
    uint32_t wd[U][W];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < W; ++k) wd[u][k] = ok[u] ? ld_front(P.next + (id[u][k] >> 5)) : 0xffffffffu;
    unsigned clear = 0;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < W; ++k) clear |= ((~wd[u][k] >> (id[u][k] & 31)) & 1u) << (u * W + k);
    if (!clear) return;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int k = 0; k < W; ++k)
            if ((clear >> (u * W + k)) & 1u) notify_one<Q>(P, id[u][k], h);
}

// notify every neighbour whose tau could still depend on R (Alg. 3, orange
// lines): set its next-frontier bit if h <= tau(R').  With slots there is one
// bit per slot, so the test reads the 16-bit copy and the bit sits next to it
// (no r-clique id on this path).
template <int Q>
__device__ __forceinline__ void notify_row(const SweepParams& P, const uint32_t* __restrict__ row, int d, int32_t h,
                                           int first, int step) {
    constexpr int W = kWords<Q>;
    constexpr int U = W == 3 ? 2 : kNotifyUnroll;
    // a relabelled (1,2) row: from this id on every tau is below h
    const uint32_t limit = Q == 1 && P.oct_max ? id_limit(P.oct_max, h) : 0xffffffffu;
    for (unsigned j0 = 0; j0 < (unsigned)d; j0 += U * step) {  // past d it may leave 31 bits
        uint32_t id[U][W];
        bool ok[U];
        if ((unsigned)d - j0 >= (unsigned)(U * step)) {  // a whole block: no test per entry
#pragma unroll
            for (int u = 0; u < U; ++u) {
                entry_ids<Q>(row, d, (int)(j0 + u * step + first), id[u]);
                ok[u] = true;
            }
        } else {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const unsigned j = j0 + u * step + first;
                ok[u] = j < (unsigned)d;
                if (ok[u]) {
                    entry_ids<Q>(row, d, (int)j, id[u]);
                } else {
#pragma unroll
                    for (int k = 0; k < W; ++k) id[u][k] = 0u;
                }
            }
        }
        if (Q == 1) {
            if (id[0][0] >= limit) break;  // so are this lane's later entries
#pragma unroll
            for (int u = 0; u < U; ++u) ok[u] = ok[u] && id[u][0] < limit;
        }
        notify_block<Q, U>(P, id, ok, h);
    }
}

// notification for one entry j of a row whose tau dropped to h (the merged
// walk of group rows below gives each lane entries of different rows)
template <int Q>
__device__ __forceinline__ void notify_entry(const SweepParams& P, int64_t jb, int d, int j, int32_t h) {
    uint32_t id[1][kWords<Q>];
    const bool ok[1] = {true};
    entry_ids<Q>(row_of<Q>(P, jb), d, j, id[0]);
    notify_block<Q, 1>(P, id, ok, h);
}

// batches: R changed, so its graph is still changing
template <bool GB>
__device__ __forceinline__ void graph_changed(const SweepParams& P, uint32_t R) {
    if constexpr (GB) P.gact_out[__ldg(P.gid + R)] = 1;
}

__device__ __forceinline__ nd_item load_item(const nd_item* __restrict__ items, int64_t i) {
    longlong2 v = __ldg(reinterpret_cast<const longlong2*>(items) + i);
    nd_item it;
    it.jb = v.x;
    it.R = (uint32_t)(unsigned long long)v.y;
    it.d = (uint32_t)((unsigned long long)v.y >> 32);
    return it;
}

// counters of one thread over a pass.  FULL (no-storage passes): evaluated
// rows and their incidences too; k_active_list counts them for the passes that
// take its list, and the others evaluate every row, so the host knows both.
template <bool FULL>
struct Tally {
    unsigned changed = 0, evals = 0;
    unsigned long long incs = 0;
    __device__ __forceinline__ void row(uint32_t d, bool ch) {
        if (FULL) {
            evals++;
            incs += d;
        }
        changed += ch;
    }
};

// tau(R) (t0), its value clipped at d_s for the search (t: a no-op for every
// valid tau, which is <= d_s; changes are detected against the stored value),
// and what the output buffer holds (old; for AND the same array)
template <bool AND>
__device__ __forceinline__ void load_tau(const SweepParams& P, const nd_item& it, int32_t& t0, int32_t& t,
                                         int32_t& old) {
    t0 = ld_tau<!AND>(P.tin + it.R);
    old = AND ? t0 : P.tout[it.R];
    t = min(t0, (int32_t)min(it.d, (uint32_t)INT32_MAX));
}

// work item i of a pass, or of its list
template <bool LISTED>
__device__ __forceinline__ nd_item pass_item(const SweepParams& P, int64_t i) {
    return load_item(P.items, LISTED ? (int64_t)__ldg(P.list + i) : i);
}

// one r-clique per group of G lanes of the calling warp (run: the group has
// one).  NOTIFY: the entries of all rows that changed are then walked by the
// 32 lanes together, instead of each row by its own G lanes while the other
// groups wait.
template <int Q, int G, int C, bool AND, bool NOTIFY, bool GB, bool INLINE>
__device__ __forceinline__ void run_groups(const SweepParams& P, const nd_item& it, bool run, Tally<INLINE>& n) {
    if (INLINE) run = run && in_frontier<Q>(P, it.R);
    constexpr int NG = 32 / G;
    const int lane = threadIdx.x & 31;
    int32_t t0, t, old;
    load_tau<AND>(P, it, t0, t, old);
    const int d = run ? (int)it.d : 0;
    if (!run) t = 0;
    const int dmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)d);
    const int32_t h = group_hindex<G, C>(make_rho<Q, !AND>(P, it.jb, it.d), d, dmax, t);
    if (run && (lane & (G - 1)) == 0) {
        n.row(it.d, h != t0);
        if (h != t0) graph_changed<GB>(P, it.R);
        store_tau<Q>(P, it.R, h, old);
    }
    if constexpr (NOTIFY) {
        // entry e of the changed rows' concatenation belongs to the last row q
        // that begins at or before e (the beginnings are kept in registers)
        const int dn = h != t0 ? d : 0;
        int begin[NG], tot = 0;
#pragma unroll
        for (int q = 0; q < NG; ++q) {
            begin[q] = tot;
            tot += __shfl_sync(0xffffffffu, dn, q * G);
        }
        for (int e0 = 0; e0 < tot; e0 += 32) {
            const int e = e0 + lane;
            int q = 0, b = 0;
#pragma unroll
            for (int r = 1; r < NG; ++r)
                if (e >= begin[r] && begin[r] < tot) {  // an empty row's beginning is the next one's
                    q = r;
                    b = begin[r];
                }
            const int64_t jr = __shfl_sync(0xffffffffu, it.jb, q * G);
            const int32_t hh = __shfl_sync(0xffffffffu, h, q * G);
            const int dr = __shfl_sync(0xffffffffu, dn, q * G);
            if (e < tot) notify_entry<Q>(P, jr, dr, e - b, hh);
        }
    }
}

// one r-clique per warp (rows of the warp bucket), streamed
template <int Q, bool AND, bool NOTIFY, bool GB, int HW, bool INLINE>
__device__ __forceinline__ void run_warp_row(const SweepParams& P, const nd_item& it, unsigned* bins,
                                             Tally<INLINE>& n) {
    const uint32_t R = it.R;
    if (INLINE && !in_frontier<Q>(P, R)) return;
    int32_t t0, t, old;
    load_tau<AND>(P, it, t0, t, old);
    const bool direct = P.direct || (!AND && old != t0);
    int32_t h;
    if (Q == 1 && P.oct_max)
        h = warp_hindex<true, HW>(make_rho<Q, !AND>(P, it.jb, it.d),
                                  IdBound{P.inc + it.jb, P.oct_max, direct ? 0u : id_limit(P.oct_max, t)}, (int)it.d, t,
                                  direct, bins);
    else
        h = warp_hindex<true, HW>(make_rho<Q, !AND>(P, it.jb, it.d), NoBound{}, (int)it.d, t, direct, bins);
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        n.row(it.d, h != t0);
        if (h != t0) graph_changed<GB>(P, R);
        store_tau<Q>(P, R, h, old);
    }
    if (AND && NOTIFY && h != t0) notify_row<Q>(P, row_of<Q>(P, it.jb), (int)it.d, h, lane, 32);
    __syncwarp();  // the bins are free again
}

// one r-clique per CTA (rows past the warp threshold)
template <int Q, bool AND, bool NOTIFY, bool GB, int WORDS, bool INLINE>
__device__ __forceinline__ void run_cta(const SweepParams& P, int64_t i, unsigned* bins, int* bounds,
                                        Tally<INLINE>& n) {
    const nd_item it = pass_item<(NOTIFY && !INLINE) || GB>(P, i);
    const uint32_t R = it.R;
    if (INLINE && !in_frontier<Q>(P, R)) return;  // the same R for the whole block
    int32_t t0, t, old;
    load_tau<AND>(P, it, t0, t, old);
    __syncthreads();  // AND: every thread has read tau(R) before it is written
    const int d = (int)it.d;
    const bool direct = P.direct || (!AND && old != t0);
    int32_t h;
    if (kSlots<Q> && t > kTau16Max) {  // only then can a saturated value matter
        h = cta_hindex<WORDS>(RhoExact<Q, !AND>{row_of<Q>(P, it.jb), d, P.eid, P.tin}, NoBound{}, d, t, direct, bins,
                              bounds);
    } else if (Q == 1 && t > kTau16Max) {
        h = cta_hindex<WORDS>(Rho<1, !AND, int32_t>{row_of<Q>(P, it.jb), d, P.tin}, NoBound{}, d, t, direct, bins,
                              bounds);
    } else if (Q == 1 && P.oct_max) {
        const IdBound bound{P.inc + it.jb, P.oct_max, id_limit(P.oct_max, t)};
        h = cta_hindex<WORDS>(make_rho<Q, !AND>(P, it.jb, it.d), bound, d, t, direct, bins, bounds);
    } else {
        h = cta_hindex<WORDS>(make_rho<Q, !AND>(P, it.jb, it.d), NoBound{}, d, t, direct, bins, bounds);
    }
    if (threadIdx.x == 0) {
        n.row(it.d, h != t0);
        if (h != t0) graph_changed<GB>(P, R);
        store_tau<Q>(P, R, h, old);
    }
    if (AND && NOTIFY && h != t0) notify_row<Q>(P, row_of<Q>(P, it.jb), d, h, threadIdx.x, kThreads);
    __syncthreads();
}

// Before each pass of AND with notification: the work items whose r-clique is
// in the frontier (of a batch's SND and AND-nn passes: whose graph changed in
// the pass before), compacted bucket by bucket, in order inside a tile; the pass
// then takes dense tasks from the list, and splits few rows over all warps.
// (With the frontier tested by each warp for its own chunk of work items, a
// chunk of long rows that happened to be active together kept one warp busy:
// 0.2 ms for a pass of 9,000 of 3.8M edges.)  It also clears the next frontier
// and counts the pass's evaluations.  Streams 16 B per work item and its slots;
// one atomic per tile.
constexpr int kListTile = 2048;

struct ListParams {
    const uint2* __restrict__ epos;
    const uint32_t* __restrict__ tpos;
    const uint32_t* __restrict__ gid;  // batches: the graph of every r-clique, and the graphs still changing
    const uint8_t* gact_in;
    const nd_item* __restrict__ items;
    const uint32_t* cur;
    uint32_t* next;
    int64_t words;               // of the next frontier to clear
    int64_t lo[ND_NB + 1];       // bucket ranges in items
    int64_t tile_lo[ND_NB + 1];  // tiles of kListTile items, none across buckets
    int64_t first, last;         // the tiles of this list
    uint32_t* list;
    unsigned long long* ctr;
    const unsigned long long* prev;
};

constexpr int kByGraph = 0;  // k_active_list: by graph instead of by frontier bit (Q)
template <int Q>
__global__ void __launch_bounds__(kThreads) k_active_list(ListParams L) {
    if (L.prev != nullptr && *(volatile const unsigned long long*)L.prev == 0ull) return;  // converged
    constexpr int K = kListTile / kThreads;
    __shared__ unsigned wsum[kThreads / 32];
    __shared__ unsigned long long s_base, s_in[kThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < L.words; i += (int64_t)gridDim.x * kThreads)
        L.next[i] = 0u;
    unsigned long long evals = 0, incs = 0;
    for (int64_t t = L.first + blockIdx.x; t < L.last; t += gridDim.x) {
        int b = 0;
        while (t >= L.tile_lo[b + 1]) ++b;
        const int64_t i0 = L.lo[b] + (t - L.tile_lo[b]) * kListTile + (int64_t)w * (kListTile / (kThreads / 32)) + lane;
        uint32_t R[K], d[K];
        bool act[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int64_t i = i0 + 32 * k;
            const uint2 x = i < L.lo[b + 1] ? __ldg(reinterpret_cast<const uint2*>(L.items + i) + 1) : make_uint2(0u, 0u);
            R[k] = x.x;
            d[k] = x.y;  // 0: past the bucket
        }
        if constexpr (Q == kByGraph) {
            uint32_t g[K];
#pragma unroll
            for (int k = 0; k < K; ++k) g[k] = __ldg(L.gid + R[k]);
#pragma unroll
            for (int k = 0; k < K; ++k) act[k] = d[k] && L.gact_in[g[k]];
        } else if constexpr (Q == 2) {
            uint2 ep[K];
#pragma unroll
            for (int k = 0; k < K; ++k) ep[k] = __ldg(L.epos + R[k]);
#pragma unroll
            for (int k = 0; k < K; ++k) act[k] = d[k] && (front_bit(L.cur, ep[k].x) | front_bit(L.cur, ep[k].y));
        } else if constexpr (Q == 3) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const uint32_t* p = L.tpos + 3 * (int64_t)R[k];
                const uint32_t a0 = __ldg(p), a1 = __ldg(p + 1), a2 = __ldg(p + 2);
                act[k] = d[k] && (front_bit(L.cur, a0) | front_bit(L.cur, a1) | front_bit(L.cur, a2));
            }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) act[k] = d[k] && front_bit(L.cur, R[k]);
        }
        unsigned c = 0;
        uint32_t at[K];
        unsigned long long in = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const unsigned m = __ballot_sync(0xffffffffu, act[k]);
            at[k] = c + __popc(m & ((1u << lane) - 1u));
            c += __popc(m);
            if (act[k]) in += d[k];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) in += __shfl_xor_sync(0xffffffffu, in, o);
        if (lane == 0) { wsum[w] = c; s_in[w] = in; }
        __syncthreads();
        unsigned before = 0, total = 0;
#pragma unroll
        for (int v = 0; v < kThreads / 32; ++v) {
            if (v < w) before += wsum[v];
            total += wsum[v];
        }
        if (threadIdx.x == 0) {
            s_base = total ? atomicAdd(L.ctr + ND_CTR_LIST + b, (unsigned long long)total) : 0ull;
            evals += total;
            for (int v = 0; v < kThreads / 32; ++v) incs += s_in[v];
        }
        __syncthreads();
        // the bucket's part of the list begins at its first tile here
        uint32_t* const out = L.list + (max(L.tile_lo[b], L.first) - L.first) * kListTile + s_base + before;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (act[k]) out[at[k]] = (uint32_t)(i0 + 32 * k);
        __syncthreads();
    }
    if (threadIdx.x == 0 && evals) {
        atomicAdd(L.ctr + ND_CTR_EVALS, evals);
        atomicAdd(L.ctr + ND_CTR_INCS, incs);
    }
}

// the block's counters, added to the pass's
template <bool FULL>
__device__ __forceinline__ void flush_tally(const SweepParams& P, const Tally<FULL>& n) {
    __shared__ unsigned s_ch[kThreads / 32], s_ev[kThreads / 32];
    __shared__ unsigned long long s_in[kThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned ch = __reduce_add_sync(0xffffffffu, n.changed);
    unsigned ev = 0;
    unsigned long long in = 0;
    if (FULL) {
        ev = __reduce_add_sync(0xffffffffu, n.evals);
        in = n.incs;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) in += __shfl_xor_sync(0xffffffffu, in, o);
    }
    if (lane == 0) { s_ch[wid] = ch; s_ev[wid] = ev; s_in[wid] = in; }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long a = 0, e = 0, c = 0;
        for (int w = 0; w < kThreads / 32; ++w) { a += s_ch[w]; e += s_ev[w]; c += s_in[w]; }
        if (a) atomicAdd(P.ctr + ND_CTR_CHANGED, a);
        if (e) atomicAdd(P.ctr + ND_CTR_EVALS, e);
        if (c) atomicAdd(P.ctr + ND_CTR_INCS, c);
    }
}

// warp tasks per counter grab: kWarpChunk where there are many, fewer where
// that would leave the resident warps with less than kChunksPerWarp grabs
// each.  A graph of 2,000 vertices has 250 tasks: in chunks of 16 they kept 16
// warps busy, one after the other (26 us per pass).  R-MAT of 100,003 vertices:
// the first 16 SND passes 3.2 ms with 8 grabs, 3.9 with 4, 3.2 with 16 (whose
// late passes are 12% slower).
constexpr int kChunksPerWarp = 8;
__host__ __device__ __forceinline__ int warp_chunk(int64_t tasks, int grid) {
    const int64_t c = tasks / ((int64_t)(grid > 0 ? grid : 1) * (kThreads / 32) * kChunksPerWarp);
    return (int)(c < 1 ? 1 : (c > kWarpChunk ? kWarpChunk : c));
}

// AND ends its passes on the longest warp rows: the last kTailTasks tasks of
// every resident warp come in chunks of kTailChunk, so that no warp is left
// with a chunk of them.  AND without notification, the first eight passes, in
// whole chunks / with the tail: 2.76 / 2.13 ms for R-MAT of 100,003 vertices,
// 27.4 / 25.8 ms for scale 20 (k-truss).
constexpr int kTailTasks = 8, kTailChunk = 2;

// lanes of a group, and entries per lane of its longest row
template <int G, int C>
struct GroupOf {
    static constexpr int lanes = G, entries = C;
};

constexpr int kPassBlocks = 6;  // resident blocks per SM the register budget of every pass kernel targets

// GB: a batch handle's SND / AND-nn pass, which leaves out the rows of graphs
// that have converged, and marks those that change
// LATE: the passes after the first of a run, where few rows search: a
// quarter of the histogram, and the shared memory it frees serves as L1 for
// the gathers
// INLINE: AND with notification on a handle of at most kInlineItems work items
// takes no list: a launch costs more than the rows' own frontier tests.  The
// pass clears the frontier of the pass after next, of four (a clear by memset
// or with the list costs a launch of its own).  A 2,000-vertex k-core: 16
// passes in 0.13 instead of 0.23 ms.
template <int Q, bool AND, bool NOTIFY, bool GB, bool LATE, bool INLINE = false>
__global__ void __launch_bounds__(kThreads, kPassBlocks) k_pass(SweepParams P) {
    if (P.prev != nullptr && *(volatile const unsigned long long*)P.prev == 0ull) return;  // converged
    constexpr bool LISTED = (NOTIFY && !INLINE) || GB;
    constexpr int HW = LATE ? kLateHistWords : kHistWords;
    constexpr int kWords = (kThreads / 32) * HW;  // a CTA row uses every warp's histogram
    __shared__ __align__(16) unsigned hist[kThreads / 32][HW];
    __shared__ int bounds[kThreads / 32];
    __shared__ unsigned long long s_chunk;
    unsigned* const bins = hist[threadIdx.x >> 5];
    Tally<INLINE> n;
    if (INLINE)
        for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < P.spare_words; i += (int64_t)gridDim.x * kThreads)
            P.spare[i] = 0u;
    // the rows of each bucket: [lo, lo + rows) of the work items, or of the list
    auto lo = [&](int b) { return LISTED ? P.list_lo[b] : P.lo[b]; };
    auto rows = [&](int b) { return LISTED ? (int64_t)__ldcg(P.ctr + ND_CTR_LIST + b) : P.hi[b] - P.lo[b]; };
    // phase 1: rows longer than the CTA threshold, one per block at a time,
    // taken from a per-pass counter (longest rows first)
    const int64_t n3 = rows(3);
    auto cta_phase = [&]() {
        if (n3 <= 0) return;
        for (;;) {
            if (threadIdx.x == 0) s_chunk = atomicAdd(P.ctr + ND_CTR_CTA, 1ull);
            __syncthreads();
            const int64_t c = (int64_t)s_chunk;
            __syncthreads();
            if (c >= n3) break;
            run_cta<Q, AND, NOTIFY, GB, kWords, INLINE>(P, lo(3) + c, &hist[0][0], bounds, n);
        }
    };
    // AND updates in place, so a row evaluated later in a pass already sees
    // what earlier rows lowered: AND takes the shortest rows first and the
    // CTA rows last (the first eight passes with notification on the R-MAT
    // scale-20 k-truss: 33.2 against 34.4 ms longest first).  SND, whose pass
    // reads only the previous pass, takes the longest rows first, for balance,
    // and so does (1,2), whose longest rows are hub vertices of up to hundreds
    // of thousands of entries (R-MAT scale-24 k-core: 15.1 against 15.6 ms).
    constexpr bool kShortFirst = AND && Q != 1;
    constexpr bool kCtaFirst = !kShortFirst;
    if (kCtaFirst) cta_phase();
    // phase 2: warp tasks (one warp row, four 8-lane rows or eight 4-lane
    // rows), longest first (SND) or shortest first (AND).  Each warp takes
    // chunks of consecutive tasks from a per-pass counter (one atomic per
    // chunk, no barrier): consecutive r-cliques share a vertex and gather from
    // the same part of tau.
    const int64_t n2 = rows(2), n1 = rows(1), n0 = rows(0);
    const int64_t t1 = (n1 + 3) / 4, t0 = (n0 + 7) / 8;
    const int64_t tasks = n2 + t1 + t0;
    const int lane32 = threadIdx.x & 31;
    const int chunk = LISTED ? warp_chunk(tasks, gridDim.x) : P.chunk;
    // the last tasks in small chunks
    const int64_t tail = kShortFirst ? min(tasks, (int64_t)gridDim.x * (kThreads / 32) * kTailTasks) : 0;
    const int tc = min(kTailChunk, chunk);
    const int64_t big = (tasks - tail + chunk - 1) / chunk;
    const int64_t nchunks = big + (tail + tc - 1) / tc;
    for (;;) {
        unsigned long long c = 0;
        if (lane32 == 0) c = atomicAdd(P.ctr + ND_CTR_CHUNK, 1ull);
        c = __shfl_sync(0xffffffffu, c, 0);
        if ((int64_t)c >= nchunks) break;
        // [t, te) in the order of the pass
        int64_t t = (int64_t)c < big ? (int64_t)c * chunk : tasks - tail + ((int64_t)c - big) * tc;
        int64_t te = (int64_t)c < big ? min(t + (int64_t)chunk, tasks - tail) : min(t + (int64_t)tc, tasks);
        if (kShortFirst) {
            const int64_t x = tasks - te;
            te = tasks - t;
            t = x;
        }
        const int64_t e2 = min(te, n2);
        if (t < e2) {
            // warp rows: the next row's work item is loaded before this one runs
            nd_item it = pass_item<LISTED>(P, lo(2) + t);
            while (t < e2) {
                nd_item nx;
                if (t + 1 < e2) nx = pass_item<LISTED>(P, lo(2) + t + 1);
                run_warp_row<Q, AND, NOTIFY, GB, HW, INLINE>(P, it, bins, n);
                it = nx;
                ++t;
            }
        }
        // group rows, the same: the next task's items are loaded before this
        // one runs (the first group's item stands in where a group has none).
        // SND 2 to 4% faster; with notification, whose registers are short, 2
        // to 5% slower, so not there.
        auto group_tasks = [&](int64_t from, int64_t to, int64_t begin, int64_t count, auto group) {
            constexpr int G = decltype(group)::lanes, NG = 32 / G;
            if (from >= to) return;
            auto item = [&](int64_t task) {
                const int64_t i = NG * task + lane32 / G;
                return pass_item<LISTED>(P, begin + (i < count ? i : NG * task));
            };
            nd_item it = item(from);
            for (int64_t k = from; k < to; ++k) {
                nd_item nx;
                if (!NOTIFY && k + 1 < to) nx = item(k + 1);
                run_groups<Q, G, decltype(group)::entries, AND, NOTIFY, GB, INLINE>(P, it, NG * k + lane32 / G < count, n);
                if (NOTIFY && k + 1 < to) nx = item(k + 1);
                it = nx;
            }
        };
        group_tasks(max(t, n2) - n2, min(te, n2 + t1) - n2, lo(1), n1, GroupOf<8, 8>{});
        group_tasks(max(t, n2 + t1) - n2 - t1, te - n2 - t1, lo(0), n0, GroupOf<4, 2>{});
    }
    if (!kCtaFirst) cta_phase();
    flush_tally(P, n);
}

// tau_0 = d_s in a; b (SND's other buffer): -1, which no pass has stored, for
// every row that a pass evaluates, so that the first pass writes them all and
// takes them for rows that have just changed (see warp_hindex)
__global__ void k_init_tau(int64_t N, const int64_t* __restrict__ inc_ptr, int32_t* __restrict__ a,
                           int32_t* __restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        int32_t d = (int32_t)(inc_ptr[i + 1] - inc_ptr[i]);
        a[i] = d;
        if (b) b[i] = d ? -1 : 0;
    }
}

// tau -> its CSR-position copies: both entries of every edge
__global__ void k_tau_to_adj(int64_t N, const uint2* __restrict__ epos, const int32_t* __restrict__ tau,
                             uint16_t* __restrict__ a, uint16_t* __restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint2 ep = epos[i];
        const uint16_t v = (uint16_t)min(max(tau[i], 0), kTau16Max);
        a[ep.x] = v;
        a[ep.y] = v;
        if (b) {
            b[ep.x] = v;
            b[ep.y] = v;
        }
    }
}

// the same for the three list slots of every triangle
__global__ void k_tau_to_lists(int64_t N, const uint32_t* __restrict__ tpos, const int32_t* __restrict__ tau,
                               uint16_t* __restrict__ a, uint16_t* __restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 3 * N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = tpos[i];
        const uint16_t v = (uint16_t)min(max(tau[i / 3], 0), kTau16Max);
        a[p] = v;
        if (b) b[p] = v;
    }
}

// tau -> its 16-bit gather copies indexed by r-clique id ((1,2))
__global__ void k_tau_to_16(int64_t N, const int32_t* __restrict__ tau, uint16_t* __restrict__ a,
                            uint16_t* __restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const uint16_t v = (uint16_t)min(max(tau[i], 0), kTau16Max);
        a[i] = v;
        if (b) b[i] = v;
    }
}

// PartialAnd with the (2,3) layout: both CSR positions of every member
__global__ void k_member_pos(int64_t N, const uint32_t* __restrict__ members, const uint2* __restrict__ epos,
                             uint32_t* __restrict__ f) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!((members[i >> 5] >> (i & 31)) & 1u)) continue;
        const uint2 ep = epos[i];
        atomicOr(f + (ep.x >> 5), 1u << (ep.x & 31));
        atomicOr(f + (ep.y >> 5), 1u << (ep.y & 31));
    }
}

// and with the (3,4) layout: the three list slots of every member
__global__ void k_member_lists(int64_t N, const uint32_t* __restrict__ members, const uint32_t* __restrict__ tpos,
                               uint32_t* __restrict__ f) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (!((members[i >> 5] >> (i & 31)) & 1u)) continue;
        for (int k = 0; k < 3; ++k) {
            const uint32_t p = tpos[3 * i + k];
            atomicOr(f + (p >> 5), 1u << (p & 31));
        }
    }
}

__global__ void k_fill_front(int64_t N, uint32_t* __restrict__ f) {
    const int64_t words = (N + 31) / 32;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < words;
         w += (int64_t)gridDim.x * blockDim.x) {
        int64_t rem = N - w * 32;
        f[w] = rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u);
    }
}

__global__ void k_member_mask(const uint32_t* __restrict__ ids, int64_t count, int64_t N,
                              uint32_t* __restrict__ mask, int* __restrict__ err, const int32_t* __restrict__ to_new) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t R = ids[i];
        if ((int64_t)R >= N) { atomicOr(err, 1); continue; }
        if (to_new) R = (uint32_t)to_new[R];  // relabelled (1,2) handle
        atomicOr(mask + (R >> 5), 1u << (R & 31));
    }
}

__global__ void k_count_equal(const int32_t* __restrict__ a, const int32_t* __restrict__ b, int64_t n,
                              unsigned long long* __restrict__ out) {
    unsigned long long c = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        c += (a[i] == b[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

__global__ void k_add_const(const int32_t* __restrict__ in, int64_t n, int32_t c, int32_t* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        out[i] = in[i] + c;
}

// ---- (2,3) without a stored incidence ----------------------------------------
// The paper's own mode (its s-cliques are not stored but found again on every
// pass, Section 4.1 "Time complexity" and Section 5): for row R = edge (x,y)
// the triangles are the w in both N(x) and N(y).  Its entries are indexed by
// the slots of the shorter list N(s): entry j is w = N(s)[j], present if w is
// in the longer list N(l) (binary search).  A present entry has
// rho = min(tau at P(s,w), tau at P(l,w)), two slots of the CSR-position copy
// (the same slots the stored layout lists); a missing one returns -1, which
// no h-index step counts (every bound is >= 0).  One warp per row, longest
// rows first, in chunks from a counter.
//
// Finding the w: 32 entries of the shorter list at a time, in order.
//  - Where the longer list is a hub's, its table (k_hub_tables) holds one bit
//    per vertex and a count per 32 of them: one 8-byte load tells whether w is
//    a neighbour and at which entry.  No order is needed for that, so the
//    shorter list is walked by degree class, high first: the w of high degree
//    close most triangles and hold the largest tau, and past a class no tau
//    exceeds its degrees (DegreeBound).
//  - Otherwise blocks of the longer list pass through shared memory, or, where
//    it is much longer, every lane searches it (nd_list_cursor).
// A search of the whole list per entry (the only way before) takes some 250 L1
// wavefronts per 32 entries of a list of 4,000, because its lanes part after
// the first steps.  The blocks alone were little faster: about 150 instructions
// per 32 entries; a table takes 25.  SND of an R-MAT k-truss of 50,021 vertices
// (33.4M incidences, 101 passes): 109 ms with searches, 95 with blocks, 45 with
// tables, 34 with the lists by degree class (late passes 0.31 ms; 0.43 in CSR
// order).
template <bool RO, bool EXACT>
struct OtfRow {
    static constexpr bool kCarry = false;
    const int32_t* __restrict__ scol;   // N(s), sn entries: in CSR order from slot sb, or
    const uint32_t* __restrict__ slot;  // with a table, by degree class, and their slots
    int64_t sb, lb;  // first slots of N(s) and of the longer list N(l)
    int sn;
    const uint2* __restrict__ table;  // of the longer list's vertex, or null
    const uint16_t* tau16;
    const uint32_t* __restrict__ eid;
    const int32_t* tau32;
    mutable nd_list_cursor longer;

    // the entry of w in the longer list, -1 if it is none
    static __device__ __forceinline__ int at_table(uint2 x, int32_t w) {
        const unsigned below = (1u << (w & 31)) - 1u;
        return (x.x >> (w & 31)) & 1u ? (int)(x.y + __popc(x.x & below)) : -1;
    }

    // f(k) for the entries [i, end) of N(s), 32 at a time: entry i + lane is in
    // N(l) at k, or k = -1.  Sweeps start at 0 and go on where they stopped.
    template <typename G>
    __device__ __forceinline__ void match(int i, int end, G&& f) const {
        const int lane = threadIdx.x & 31;
        if (table) {
            for (; end - i >= 64; i += 64) {  // two blocks in flight
                int32_t w[2];
                uint2 x[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) w[u] = __ldg(scol + i + 32 * u + lane);
#pragma unroll
                for (int u = 0; u < 2; ++u) x[u] = __ldg(table + (w[u] >> 5));
#pragma unroll
                for (int u = 0; u < 2; ++u) f(i + 32 * u + lane, at_table(x[u], w[u]));
            }
            for (; i < end; i += 32) {
                const int j = i + lane;
                int k = -1;
                if (j < end) {
                    const int32_t w = __ldg(scol + j);
                    k = at_table(__ldg(table + (w >> 5)), w);
                }
                f(j, k);
            }
            return;
        }
        if (i == 0) longer.restart(sn);
        for (; i < end; i += 32) {
            const int j = i + lane;
            const int32_t w = j < end ? __ldg(scol + j) : 0;
            f(j, longer.find(w, j < end, __reduce_max_sync(0xffffffffu, w)));
        }
    }
    __device__ __forceinline__ int32_t rho(int j, int k) const {
        if (k < 0) return -1;
        const int64_t ps = slot ? (int64_t)__ldg(slot + j) : sb + j, pl = lb + k;
        if (EXACT) return min(ld_tau<RO>(tau32 + __ldg(eid + ps)), ld_tau<RO>(tau32 + __ldg(eid + pl)));
        return min(ld_tau<RO>(tau16 + ps), ld_tau<RO>(tau16 + pl));
    }
};

// a list by degree class: past an entry of degree d, no edge to a later entry
// has a tau above the largest degree of d's class, less one
struct DegreeBound {
    const int32_t* __restrict__ scol;  // null: the list is in another order
    const int64_t* __restrict__ rp;
    int32_t t;
    __device__ __forceinline__ bool past(int j) const {
        if (!scol) return false;
        const int32_t w = __ldg(scol + j - 1);
        const unsigned d = (unsigned)(__ldg(rp + w + 1) - __ldg(rp + w));
        return (0xffffffffu >> __clz(d)) - 1 < (unsigned)t;
    }
};

template <int STEP, bool RO, bool EXACT, typename G>
__device__ __forceinline__ void stream_row(const OtfRow<RO, EXACT>& row, int i, int end, G&& f) {
    row.match(i, end, [&](int j, int k) { f(j, row.rho(j, k)); });
}

// rows per counter grab.  What a row needs before its first list entry is a
// chain of five loads (work item, endpoints, list bounds, hub number); the
// lanes of a warp walk the chains of a whole grab at once.
// Rows of the warp bucket come four at a time and CTA rows alone: in grabs of
// eight, a few warps held the longest rows and a first pass took 1.26 instead
// of 0.66 ms.
constexpr int kOtfChunk = 8, kOtfChunk2 = 4;

template <bool AND, bool NOTIFY>
__global__ void __launch_bounds__(kThreads, kPassBlocks) k_pass_otf(SweepParams P) {
    if (P.prev != nullptr && *(volatile const unsigned long long*)P.prev == 0ull) return;  // converged
    __shared__ __align__(16) unsigned hist[kThreads / 32][kHistWords];
    __shared__ int32_t blocks[kThreads / 32][nd_list_cursor::kBlock];
    Tally<true> n;
    const int lane = threadIdx.x & 31;
    unsigned* const bins = hist[threadIdx.x >> 5];
    int32_t* const buf = blocks[threadIdx.x >> 5];
    const int64_t first = P.lo[0], rows = P.hi[ND_NB - 1] - P.lo[0];
    const int64_t n3 = P.hi[3] - P.lo[3], n2 = P.hi[2] - P.lo[2], g2 = (n2 + kOtfChunk2 - 1) / kOtfChunk2;
    for (;;) {
        unsigned long long c = 0;
        if (lane == 0) c = atomicAdd(P.ctr + ND_CTR_CHUNK, 1ull);
        c = __shfl_sync(0xffffffffu, c, 0);
        // the grab's rows [r0, r0 + take): one at a time of the CTA bucket,
        // kOtfChunk2 of the warp bucket, then kOtfChunk
        int64_t g = (int64_t)c, r0 = 0;
        int take = 1;
        if (g < n3) {
            r0 = g;
        } else if ((g -= n3) < g2) {
            r0 = n3 + g * kOtfChunk2;
            take = (int)min((int64_t)kOtfChunk2, n3 + n2 - r0);
        } else {
            r0 = n3 + n2 + (g - g2) * kOtfChunk;
            if (r0 >= rows) break;
            take = (int)min((int64_t)kOtfChunk, rows - r0);
        }
        // lane l: row r0 + l of the pass, longest rows first
        bool run = lane < take;
        uint32_t R = 0, d = 0, my_sb = 0, my_lb = 0;  // CSR slots fit 32 bits for (2,3)
        int32_t my_t0 = 0, my_old = 0;
        int my_sn = 0, my_ln = 0, my_hub = -1;
        if (run) {
            const nd_item it = load_item(P.items, first + rows - 1 - r0 - lane);
            R = it.R;
            d = it.d;
            if (AND && NOTIFY) run = in_frontier<2>(P, R);
        }
        if (run) {
            my_t0 = ld_tau<!AND>(P.tin + R);
            my_old = AND ? my_t0 : P.tout[R];
            const int32_t x = __ldg(P.eu + R), y = __ldg(P.ev + R);
            const int64_t xb = __ldg(P.rp + x), xe = __ldg(P.rp + x + 1);
            const int64_t yb = __ldg(P.rp + y), ye = __ldg(P.rp + y + 1);
            const bool xs = (xe - xb) <= (ye - yb);
            my_sb = (uint32_t)(xs ? xb : yb);
            my_lb = (uint32_t)(xs ? yb : xb);
            my_sn = (int)(xs ? xe - xb : ye - yb);
            my_ln = (int)(xs ? ye - yb : xe - xb);
            if (P.hub_of) my_hub = __ldg(P.hub_of + (xs ? y : x));
        }
        for (unsigned todo = __ballot_sync(0xffffffffu, run); todo; todo &= todo - 1) {
            const int l = __ffs(todo) - 1;
            const int64_t sb = __shfl_sync(0xffffffffu, my_sb, l), lb = __shfl_sync(0xffffffffu, my_lb, l);
            const int sn = __shfl_sync(0xffffffffu, my_sn, l), ln = __shfl_sync(0xffffffffu, my_ln, l);
            const int hub = __shfl_sync(0xffffffffu, my_hub, l);
            const int32_t t0 = __shfl_sync(0xffffffffu, my_t0, l), old = __shfl_sync(0xffffffffu, my_old, l);
            const int32_t t = min(t0, (int32_t)__shfl_sync(0xffffffffu, d, l));
            const bool direct = P.direct || (!AND && old != t0);
            const uint2* const table = hub >= 0 ? P.hub_bits + hub * P.hub_words : nullptr;
            const int32_t* const scol = (table && P.by_degree ? P.by_degree : P.col) + sb;
            const uint32_t* const slot = table && P.by_degree ? P.slot_of + sb : nullptr;
            const nd_list_cursor longer{P.col + lb, ln, buf, false, 0, 0};
            const OtfRow<!AND, false> row{scol, slot, sb, lb, sn, table, P.gin, P.eid, P.tin, longer};
            int32_t h;
            if (t > kTau16Max) {
                const OtfRow<!AND, true> exact{scol, slot, sb, lb, sn, table, P.gin, P.eid, P.tin, longer};
                h = warp_hindex<false, kHistWords>(exact, NoBound{}, sn, t, direct, bins);
            } else {
                h = warp_hindex<false, kHistWords>(row, DegreeBound{slot && P.bounded ? scol : nullptr, P.rp, t}, sn, t,
                                                   direct, bins);
            }
            if (lane == l) {
                n.row(d, h != t0);
                store_tau<2>(P, R, h, old);
            }
            if (AND && NOTIFY && h != t0) {
                // notify the other two edges of every triangle, found again
                const DegreeBound bound{slot && P.bounded ? scol : nullptr, P.rp, h};
                for (int i = 0; i < sn;) {
                    const int end = min(sn, i + 256);
                    row.match(i, end, [&](int j, int k) {
                        if (k < 0) return;
                        notify_pos(P, slot ? __ldg(slot + j) : (uint32_t)(sb + j), h);
                        notify_pos(P, (uint32_t)(lb + k), h);
                    });
                    i = end;
                    if (bound.past(i)) break;  // no later edge has a tau of h or more
                }
            }
            __syncwarp();  // the bins and the block of the list are free again
        }
    }
    flush_tally(P, n);
}

// vertices by floor(log2 degree)
__global__ void k_degree_classes(int64_t n, const int64_t* __restrict__ rp, unsigned long long* __restrict__ cnt) {
    __shared__ unsigned c[32];
    if (threadIdx.x < 32) c[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t d = rp[v + 1] - rp[v];
        if (d > 0) atomicAdd(&c[31 - __clz((unsigned)min(d, (int64_t)INT32_MAX))], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32 && c[threadIdx.x]) atomicAdd(cnt + threadIdx.x, (unsigned long long)c[threadIdx.x]);
}

// hub numbers of the vertices of at least min_degree neighbours
__global__ void k_number_hubs(int64_t n, const int64_t* __restrict__ rp, int64_t min_degree,
                              int32_t* __restrict__ hub_of, int32_t* __restrict__ hubs, int* __restrict__ count) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        int h = -1;
        if (rp[v + 1] - rp[v] >= min_degree) {
            h = atomicAdd(count, 1);
            hubs[h] = (int32_t)v;
        }
        hub_of[v] = h;
    }
}

// the table of every hub, one block each: word w covers the vertices
// [32 w, 32 w + 32), x = which of them are neighbours, y = neighbours below.
// The list is sorted, so a word's entries are one run: its thread searches the
// run's first entry, whose index is y, and walks the run.
__global__ void __launch_bounds__(kThreads) k_hub_tables(const int32_t* __restrict__ hubs,
                                                         const int64_t* __restrict__ rp,
                                                         const int32_t* __restrict__ col, int64_t words,
                                                         uint2* __restrict__ tables) {
    const int32_t v = hubs[blockIdx.x];
    const int64_t b = rp[v];
    const int d = (int)(rp[v + 1] - b);
    uint2* const t = tables + (int64_t)blockIdx.x * words;
    for (int64_t w = threadIdx.x; w < words; w += kThreads) {
        const int64_t lo = 32 * w;  // below n, so a vertex id
        int j = nd_lower_bound_n(col + b, d, (int32_t)lo);
        const unsigned below = (unsigned)j;
        unsigned bits = 0;
        for (; j < d; ++j) {
            const int64_t x = (int64_t)__ldg(col + b + j) - lo;
            if (x >= 32) break;
            bits |= 1u << x;
        }
        t[w] = make_uint2(bits, below);
    }
}

typedef void (*pass_fn)(SweepParams);

// the pass kernel of a run; late: for the passes from kLateFrom on
constexpr int kLateFrom = ND_BATCH;
template <int Q>
pass_fn pick_q(int mode, bool batch, bool late, bool in_line) {
    if (in_line) return k_pass<Q, true, true, false, false, true>;
    if (mode == ND_AND) return late ? k_pass<Q, true, true, false, true> : k_pass<Q, true, true, false, false>;
    if (mode == ND_SND) {
        if (batch) return late ? k_pass<Q, false, false, true, true> : k_pass<Q, false, false, true, false>;
        return late ? k_pass<Q, false, false, false, true> : k_pass<Q, false, false, false, false>;
    }
    if (batch) return late ? k_pass<Q, true, false, true, true> : k_pass<Q, true, false, true, false>;
    return late ? k_pass<Q, true, false, false, true> : k_pass<Q, true, false, false, false>;
}
pass_fn pick(const nd_incidence* h, int mode, bool late, bool in_line) {
    // mode: ND_SND, ND_AND (notify), ND_AND_NN
    if (h->otf) return mode == ND_SND ? k_pass_otf<false, false> : (mode == ND_AND ? k_pass_otf<true, true> : k_pass_otf<true, false>);
    const bool batch = h->gid && mode != ND_AND;  // converged graphs are skipped
    if (h->q == 1) return pick_q<1>(mode, batch, late, in_line);
    if (h->q == 2) return pick_q<2>(mode, batch, late, in_line);
    return h->t_pos ? pick_q<3>(mode, batch, late, in_line) : pick_q<kIds>(mode, batch, late, in_line);
}

// bucket ranges of a pass
void plan_buckets(const nd_incidence* h, SweepParams& P) {
    for (int b = 0; b < ND_NB; ++b) {
        P.lo[b] = h->bucket_lo[b];
        P.hi[b] = h->bucket_lo[b + 1];
    }
}

// work units of a pass: CTA rows + warp tasks (see k_pass); the grid never
// exceeds what the work needs
int64_t pass_units(const nd_incidence* h, const SweepParams& P) {
    if (h->otf) return P.hi[ND_NB - 1] - P.lo[0];  // one warp per row
    return (P.hi[3] - P.lo[3]) + (P.hi[2] - P.lo[2]) + (P.hi[1] - P.lo[1] + 3) / 4 + (P.hi[0] - P.lo[0] + 7) / 8;
}

// persistent grid: as many blocks as fit on the GPU at once (never more than
// the work needs)
int pass_grid(const nd_incidence* h, const void* fn, int64_t units) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, 0) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    int64_t g = (int64_t)per_sm * (h->sm_count > 0 ? h->sm_count : 152);
    const int64_t need = (units + kThreads / 32 - 1) / (kThreads / 32);
    if (g > need) g = need;
    return (int)(g < 1 ? 1 : g);
}

nd_status ensure_state(nd_incidence* h, bool and_mode, cudaStream_t st) {
    const int64_t N = h->num_r > 0 ? h->num_r : 1;
    if (!h->tau[0]) ND_TRY(nd_alloc((void**)&h->tau[0], sizeof(int32_t) * N, st, h));
    if (!and_mode && !h->tau[1]) ND_TRY(nd_alloc((void**)&h->tau[1], sizeof(int32_t) * N, st, h));
    const int64_t slots = nd_slots(h);
    if (h->q != 3 || slots > 0) {
        // 16-bit gather copies: one per slot, or per vertex for (1,2)
        const int64_t E = slots > 0 ? slots : N;
        if (!h->tg[0]) ND_TRY(nd_alloc((void**)&h->tg[0], sizeof(uint16_t) * E, st, h));
        if (!and_mode && !h->tg[1]) ND_TRY(nd_alloc((void**)&h->tg[1], sizeof(uint16_t) * E, st, h));
    }
    // one frontier bit per slot (notification sets the bit of the slot it has
    // just read), or per r-clique
    const int64_t words = ((slots > 0 ? slots : N) + 31) / 32;
    if (and_mode && !h->front[0]) {
        ND_TRY(nd_alloc((void**)&h->front[0], sizeof(uint32_t) * words, st, h));
        ND_TRY(nd_alloc((void**)&h->front[1], sizeof(uint32_t) * words, st, h));
    }
    if (!h->counters) ND_TRY(nd_alloc((void**)&h->counters, sizeof(unsigned long long) * ND_SLOT * ND_RING, st, h));
    return ND_OK;
}


// The list of a pass (k_active_list).  A handle keeps
// room for all of its work items; where it may not (the memory limit), a run
// takes a sixteenth of that as scratch and makes each pass in parts.
struct ListPlan {
    int64_t tile_lo[ND_NB + 1] = {0, 0, 0, 0, 0};
    int64_t tiles = 0, room = 0;  // all tiles; those a list holds
    uint32_t* list = nullptr;
    int64_t words = 0;  // of the next frontier
};

nd_status plan_list(nd_incidence* h, int64_t words, nd_tmp<uint32_t>& scratch, ListPlan* L, cudaStream_t st) {
    for (int b = 0; b < ND_NB; ++b)
        L->tile_lo[b + 1] = L->tile_lo[b] + (h->bucket_lo[b + 1] - h->bucket_lo[b] + kListTile - 1) / kListTile;
    L->tiles = L->tile_lo[ND_NB];
    L->words = words;
    if (L->tiles == 0) return ND_OK;
    if (h->list && h->list_tiles < L->tiles) nd_release_spare(h, st);  // other buckets than before
    if (!h->list && nd_alloc_spare((void**)&h->list, sizeof(uint32_t) * kListTile * L->tiles, st, h) == ND_OK)
        h->list_tiles = L->tiles;
    L->list = h->list;
    L->room = L->tiles;
    if (!h->list) {
        // parts of a sixteenth, or of what the device still has room for
        nd_status e;
        for (L->room = (L->tiles + 15) / 16; (e = scratch.alloc(L->room * kListTile)) != ND_OK && L->room > 1;)
            L->room = (L->room + 3) / 4;
        ND_TRY(e);
        nd_set_error("");
        L->list = scratch;
    }
    return ND_OK;
}

typedef void (*list_fn)(ListParams);
list_fn pick_list(const nd_incidence* h, bool by_graph) {
    if (by_graph) return k_active_list<kByGraph>;
    return h->q == 2 ? k_active_list<2> : (h->t_pos ? k_active_list<3> : k_active_list<1>);
}

// the parameters of the list of the tiles [first, last) for the pass P, whose
// list ranges it sets; returns the blocks to launch
int list_params(const nd_incidence* h, const ListPlan& L, int64_t first, int64_t last, SweepParams& P, ListParams* out) {
    out->epos = P.epos;
    out->tpos = P.tpos;
    out->gid = P.gid;
    out->gact_in = P.gact_in;
    out->items = P.items;
    out->cur = P.cur;
    out->next = P.next;
    out->words = first == 0 && !P.gid ? L.words : 0;
    for (int b = 0; b <= ND_NB; ++b) {
        out->lo[b] = h->bucket_lo[b];
        out->tile_lo[b] = L.tile_lo[b];
    }
    out->first = first;
    out->last = last;
    out->list = L.list;
    out->ctr = P.ctr;
    out->prev = P.prev;
    P.list = L.list;
    for (int b = 0; b < ND_NB; ++b) {
        const int64_t lo = L.tile_lo[b] > first ? L.tile_lo[b] : first;
        P.list_lo[b] = (lo - first) * kListTile;  // unused where the bucket has no tile here
    }
    const int cap = (h->sm_count > 0 ? h->sm_count : 152) * 8;
    const int for_words = nd_blocks_for(out->words, kThreads * 16, cap);
    const int for_tiles = (int)(last - first < cap ? last - first : cap);
    return for_tiles > for_words ? for_tiles : for_words;
}

// the smallest shared-memory carve-out (percent of the SM's maximum) that
// holds the resident blocks of a pass kernel (all are built for kPassBlocks)
nd_status request_carveout(const void* fn) {
    cudaFuncAttributes fa;
    int dev = 0, max_sm = 0;
    ND_CUDA(cudaFuncGetAttributes(&fa, fn));
    ND_CUDA(cudaGetDevice(&dev));
    ND_CUDA(cudaDeviceGetAttribute(&max_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
    if (max_sm <= 0) return ND_OK;
    const int64_t need = kPassBlocks * ((int64_t)fa.sharedSizeBytes + 1024);
    int pct = (int)((100 * need + max_sm - 1) / max_sm);  // rounded up to a supported carve-out
    if (pct > 100) pct = 100;
    ND_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, pct));
    return ND_OK;
}

// AND passes whose rows go straight to the histogram.  AND over a run with 0 /
// 2 / 4 / 6 / 8 of them: 55.7 / 53.9 / 52.6 / 53.0 / 53.9 ms on the R-MAT
// scale-20 k-truss, 71.9 / 68.0 / 66.1 / 62.9 / 62.7 on the scale-24 k-core
constexpr int kAndDirect = 6;

// AND with notification without a list (INLINE): small handles, with room for
// two more frontiers
constexpr int64_t kInlineItems = 1 << 15, kInlineBits = 1 << 22;
bool take_inline(nd_incidence* h, int64_t words, cudaStream_t st) {
    if (h->bucket_lo[ND_NB] > kInlineItems || 32 * words > kInlineBits) return false;
    for (int b = 2; b < 4; ++b) {
        if (h->front[b]) continue;
        if (nd_alloc_spare((void**)&h->front[b], sizeof(uint32_t) * words, st, h) != ND_OK) return false;
        nd_drop_graphs(h);  // those of AND take a list
    }
    return true;
}

// parameters of one pass: its counter slot, the slot of the pass before it
// (-1: none), its index in the run (by whose parity SND reads tau[parity]
// and writes the other buffer; AND reads the frontier front[parity])
// and whether an AND pass takes its rows for changing ones (its first passes)
SweepParams pass_params(const nd_incidence* h, int mode, const SweepParams& P0, int slot, int prev_slot,
                        int index, bool direct) {
    const int parity = index & 1;
    SweepParams P = P0;
    P.direct = direct;
    P.ctr = h->counters + ND_SLOT * slot;
    P.prev = prev_slot < 0 ? nullptr : h->counters + ND_SLOT * prev_slot;
    if (P.gid) {
        P.gact_in = h->gact[parity];
        P.gact_out = h->gact[parity ^ 1];
    }
    if (mode != ND_SND) {
        P.tin = h->tau[0];
        P.tout = h->tau[0];
        P.gin = h->tg[0];
        P.gout = h->tg[0];
        P.cur = h->front[P0.spare_words > 0 ? index & 3 : parity];
        P.next = h->front[P0.spare_words > 0 ? (index + 1) & 3 : parity ^ 1];
        P.spare = h->front[(index + 2) & 3];
    } else {
        P.tin = h->tau[parity];
        P.tout = h->tau[parity ^ 1];
        P.gin = h->tg[parity];
        P.gout = h->tg[parity ^ 1];
        P.cur = nullptr;
        P.next = nullptr;
    }
    return P;
}

// A full batch of passes as one CUDA graph: clear the batch's counters, then
// for each pass (AND: clear the next frontier) the pass kernel, then copy
// the counters to the pinned host mirror.  Built explicitly (not by stream
// capture) so that it also serves the legacy default stream.  On any
// failure the handle falls back to ordinary launches for this kind.
void make_batch_graph(nd_incidence* h, int mode, int kind, const SweepParams& P0, int grid0, pass_fn fn0,
                      int grid1, pass_fn fn1, const ListPlan& L) {
    const int base = (kind == 2) ? ND_BATCH : 0;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ex = nullptr;
    bool ok = cudaGraphCreate(&g, 0) == cudaSuccess;
    cudaGraphNode_t last = nullptr;
    if (ok) {
        cudaMemsetParams ms = {};
        ms.dst = h->counters + ND_SLOT * base;
        ms.value = 0;
        ms.elementSize = 4;
        ms.width = (size_t)ND_SLOT * ND_BATCH * 2;
        ms.height = 1;
        ok = cudaGraphAddMemsetNode(&last, g, nullptr, 0, &ms) == cudaSuccess;
    }
    for (int k = 0; ok && k < ND_BATCH; ++k) {
        // a batch starts at an even pass; its first pass reads the last slot
        // of the other half (the caller puts the previous pass's counters there)
        const int prev_slot = k > 0 ? base + k - 1 : (kind == 0 ? -1 : (base ^ ND_BATCH) + ND_BATCH - 1);
        SweepParams P = pass_params(h, mode, P0, base + k, prev_slot, k, mode != ND_SND && kind == 0 && k < kAndDirect);
        if (ok && P.gid) {  // batches: the graphs changing in this pass, from none
            cudaMemsetParams ms = {};
            ms.dst = P.gact_out;
            ms.value = 0;
            ms.elementSize = 1;
            ms.width = (size_t)h->ngraphs;
            ms.height = 1;
            cudaGraphNode_t n = nullptr;
            ok = cudaGraphAddMemsetNode(&n, g, &last, 1, &ms) == cudaSuccess;
            last = n;
        }
        if (ok && ((mode == ND_AND && !P.spare_words) || P.gid)) {
            ListParams lp;
            const int blocks = list_params(h, L, 0, L.tiles, P, &lp);
            cudaKernelNodeParams kp = {};
            void* args[] = {&lp};
            kp.func = (void*)pick_list(h, P.gid != nullptr);
            kp.gridDim = dim3(blocks);
            kp.blockDim = dim3(kThreads);
            kp.kernelParams = args;
            cudaGraphNode_t n = nullptr;
            ok = cudaGraphAddKernelNode(&n, g, &last, 1, &kp) == cudaSuccess;
            last = n;
        }
        if (!ok) break;
        cudaKernelNodeParams kp = {};
        void* args[] = {&P};
        const bool late = (kind == 0 ? k : ND_BATCH + k) >= kLateFrom;
        kp.func = (void*)(late ? fn1 : fn0);
        kp.gridDim = dim3(late ? grid1 : grid0);
        kp.blockDim = dim3(kThreads);
        kp.sharedMemBytes = 0;
        kp.kernelParams = args;
        cudaGraphNode_t n = nullptr;
        ok = cudaGraphAddKernelNode(&n, g, &last, 1, &kp) == cudaSuccess;
        last = n;
    }
    if (ok) {
        cudaGraphNode_t n = nullptr;
        ok = cudaGraphAddMemcpyNode1D(&n, g, &last, 1, h->h_counters + ND_SLOT * base, h->counters + ND_SLOT * base,
                                      sizeof(unsigned long long) * ND_SLOT * ND_BATCH,
                                      cudaMemcpyDeviceToHost) == cudaSuccess;
    }
    if (ok) ok = cudaGraphInstantiate(&ex, g, 0) == cudaSuccess;
    if (g) cudaGraphDestroy(g);
    if (!ok) {
        cudaGetLastError();  // clear, and use ordinary launches instead
        h->pass_graph_failed[mode][kind] = true;
        return;
    }
    h->pass_graph[mode][kind] = ex;
}

}  // namespace

nd_status nd_init_tau(nd_incidence* h, int32_t* tau, cudaStream_t st) {
    if (h->num_r == 0) return ND_OK;
    int blocks = nd_blocks_for(h->num_r, kThreads, h->sm_count * 8);
    nd_prof_scope ps("init_tau", st);
    k_init_tau<<<blocks, kThreads, 0, st>>>(h->num_r, h->inc_ptr, tau, nullptr);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

nd_status nd_member_mask(const uint32_t* ids, int64_t count, int64_t N, uint32_t* mask, int* err, cudaStream_t st,
                         const int32_t* to_new) {
    if (count == 0) return ND_OK;
    nd_prof_scope ps("member_mask", st);
    k_member_mask<<<nd_blocks_for(count, kThreads, 152 * 8), kThreads, 0, st>>>(ids, count, N, mask, err, to_new);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

nd_status nd_count_equal_dev(const int32_t* a, const int32_t* b, int64_t n, unsigned long long* out_dev,
                             cudaStream_t st) {
    ND_CUDA(cudaMemsetAsync(out_dev, 0, sizeof(unsigned long long), st));
    if (n == 0) return ND_OK;
    nd_prof_scope ps("count_equal", st);
    k_count_equal<<<nd_blocks_for(n, kThreads, 152 * 8), kThreads, 0, st>>>(a, b, n, out_dev);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

nd_status nd_classic_truss(const int32_t* in, int64_t n, int32_t* out, cudaStream_t st) {
    if (n == 0) return ND_OK;
    int blocks = nd_blocks_for(n, kThreads, 152 * 8);
    nd_prof_scope ps("classic_truss", st);
    k_add_const<<<blocks, kThreads, 0, st>>>(in, n, 2, out);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

namespace {

// The hub tables of a handle without a stored incidence.  The largest degree
// class whose tables, with those of the classes above, fit kHubBytes (an L2's
// worth: past that the probes would go to DRAM) bounds the hubs.  They are
// spare memory of the handle: a program that calls it again finds them built,
// and where the device or the handle's limit has no room a run does without.
// Building them takes 0.14 to 0.35 ms (426,000 to 7.6M entries), which the first
// pass of a run over triangle-rich rows wins back (SND of one pass over an
// R-MAT of 426,000 entries: 0.40 ms with them built, 0.83 with searches).  Not
// worth it, and so not built: small graphs; rows of few triangles (uniform
// random, 1.3M entries with 131,000 incidences: the whole SND 0.54 against 0.47
// ms); PartialAnd of few members (ten of a Chung-Lu k-truss of 60,000 vertices:
// 0.49 against 0.41 ms).
constexpr int64_t kHubBytes = int64_t(128) << 20;
constexpr int64_t kHubMinEntries = 1 << 18;  // below, the tables cost more than the passes
constexpr int kHubMinClass = 5;              // lists of 32 entries are searched as fast
constexpr int64_t kHubMemberShare = 8;       // PartialAnd: members at least one row in so many

bool hub_tables_pay(const nd_incidence* h, const nd_run_opts* opts) {
    if (h->num_hubs == 0 || h->nnz < kHubMinEntries || h->num_inc < h->nnz) return false;
    return !opts || !opts->members || opts->num_members >= h->bucket_lo[ND_NB] / kHubMemberShare;
}

nd_status make_hub_tables(nd_incidence* h, cudaStream_t st) {
    const int64_t words = (h->n + 31) / 32;
    const int blocks = nd_blocks_for(h->n, kThreads, h->sm_count * 8);
    nd_prof_scope ps("hub_tables", st, 3);
    if (h->num_hubs < 0) {
        nd_tmp<unsigned long long> cnt(st);
        ND_TRY(cnt.alloc(32));
        ND_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * 32, st));
        k_degree_classes<<<blocks, kThreads, 0, st>>>(h->n, h->rp, cnt);
        ND_CUDA(cudaGetLastError());
        ND_CUDA(cudaMemcpyAsync(h->h_read, cnt, sizeof(unsigned long long) * 32, cudaMemcpyDeviceToHost, st));
        ND_TRY(nd_wait(st));
        int64_t hubs = 0;
        int k = 32;
        while (k > kHubMinClass && (hubs + h->h_read[k - 1]) * words * (int64_t)sizeof(uint2) <= kHubBytes)
            hubs += h->h_read[--k];
        h->num_hubs = hubs;
        h->hub_degree = k < 31 ? 1 << k : INT32_MAX;
    }
    const int64_t hubs = h->num_hubs;
    if (hubs == 0) return ND_OK;
    nd_tmp<int32_t> list(st);
    nd_tmp<int> count(st);
    nd_status rc = nd_alloc_spare((void**)&h->hub_of, sizeof(int32_t) * h->n, st, h);
    if (rc == ND_OK) rc = nd_alloc_spare((void**)&h->by_degree, sizeof(int32_t) * h->nnz, st, h);
    if (rc == ND_OK) rc = nd_alloc_spare((void**)&h->slot_of, sizeof(uint32_t) * h->nnz, st, h);
    if (rc == ND_OK) rc = nd_alloc_spare((void**)&h->hub_bits, sizeof(uint2) * hubs * words, st, h);
    if (rc == ND_OK) rc = list.alloc(hubs);
    if (rc == ND_OK) rc = count.alloc(1);
    if (rc == ND_OK) rc = nd_rows_by_degree(h, h->by_degree, h->slot_of, st);
    if (rc != ND_OK) return rc;
    ND_CUDA(cudaMemsetAsync(count, 0, sizeof(int), st));
    k_number_hubs<<<blocks, kThreads, 0, st>>>(h->n, h->rp, h->hub_degree, h->hub_of, list, count);
    ND_CUDA(cudaGetLastError());
    k_hub_tables<<<(unsigned)hubs, kThreads, 0, st>>>(list, h->rp, h->col, words, h->hub_bits);
    ND_CUDA(cudaGetLastError());
    return ND_OK;
}

}  // namespace

// Runs passes of `mode` until a pass changes nothing or max_passes passes ran.
// Passes are enqueued in batches; each pass reads the previous pass's counter
// on the device and returns at once if it was zero, so the host only reads
// the counters back once per batch.
nd_status nd_run(nd_incidence* h, int mode, int32_t max_passes, const int32_t* tau_in_dev,
                 int32_t** tau_result, int32_t* updating, int64_t* evals, bool* converged,
                 cudaStream_t st, nd_run_opts* opts) {
    const uint32_t* members = (opts && mode != ND_SND) ? opts->members : nullptr;
    const double stop_active = (opts && mode != ND_SND) ? opts->stop_active : 0.0;
    if (opts) opts->stopped = false;
    const bool and_mode = (mode != ND_SND);
    const int64_t N = h->num_r;
    ND_TRY(ensure_state(h, and_mode, st));
    h->last_changed.clear();
    h->last_evals.clear();
    h->last_incs.clear();
    *updating = 0;
    *evals = 0;
    *converged = false;
    int blocks = nd_blocks_for(N, kThreads, h->sm_count * 8);
    if (N > 0) {
        if (tau_in_dev) {
            ND_CUDA(cudaMemcpyAsync(h->tau[0], tau_in_dev, sizeof(int32_t) * N, cudaMemcpyDeviceToDevice, st));
            if (!and_mode)
                ND_CUDA(cudaMemcpyAsync(h->tau[1], tau_in_dev, sizeof(int32_t) * N, cudaMemcpyDeviceToDevice, st));
        } else {
            nd_prof_scope ps("init_tau", st);
            k_init_tau<<<blocks, kThreads, 0, st>>>(N, h->inc_ptr, h->tau[0], and_mode ? nullptr : h->tau[1]);
            ND_CUDA(cudaGetLastError());
        }
        if (h->q != 3 || h->t_pos) {
            nd_prof_scope ps("init_tau", st);
            if (h->t_pos)
                k_tau_to_lists<<<nd_blocks_for(3 * N, kThreads, h->sm_count * 8), kThreads, 0, st>>>(
                    N, h->t_pos, h->tau[0], h->tg[0], and_mode ? nullptr : h->tg[1]);
            else if (h->adj)
                k_tau_to_adj<<<blocks, kThreads, 0, st>>>(N, h->e_pos, h->tau[0], h->tg[0],
                                                          and_mode ? nullptr : h->tg[1]);
            else
                k_tau_to_16<<<blocks, kThreads, 0, st>>>(N, h->tau[0], h->tg[0], and_mode ? nullptr : h->tg[1]);
            ND_CUDA(cudaGetLastError());
        }
    }
    *tau_result = h->tau[0];
    if (N == 0 || max_passes <= 0) {
        *converged = (N == 0);
        return ND_OK;
    }
    const int64_t fbits = nd_slots(h) > 0 ? nd_slots(h) : N;  // frontier bits (see ensure_state)
    const int64_t words = (fbits + 31) / 32;
    if (mode == ND_AND && members) {
        // PartialAnd: the members start active (end of Section 4.3)
        if (h->t_pos) {
            ND_CUDA(cudaMemsetAsync(h->front[0], 0, sizeof(uint32_t) * words, st));
            nd_prof_scope ps("fill_front", st);
            k_member_lists<<<blocks, kThreads, 0, st>>>(N, members, h->t_pos, h->front[0]);
            ND_CUDA(cudaGetLastError());
        } else if (h->adj) {
            ND_CUDA(cudaMemsetAsync(h->front[0], 0, sizeof(uint32_t) * words, st));
            nd_prof_scope ps("fill_front", st);
            k_member_pos<<<blocks, kThreads, 0, st>>>(N, members, h->e_pos, h->front[0]);
            ND_CUDA(cudaGetLastError());
        } else {
            ND_CUDA(cudaMemcpyAsync(h->front[0], members, sizeof(uint32_t) * words, cudaMemcpyDeviceToDevice, st));
        }
    } else if (mode == ND_AND) {
        nd_prof_scope ps("fill_front", st);
        k_fill_front<<<nd_blocks_for(words, kThreads, h->sm_count * 8), kThreads, 0, st>>>(fbits, h->front[0]);
        ND_CUDA(cudaGetLastError());
    }
    SweepParams P;
    P.inc = h->inc;
    P.epos = h->e_pos;
    // small handles test the frontier row by row
    const bool in_line = mode == ND_AND && !h->otf && take_inline(h, words, st);
    P.spare = nullptr;
    P.spare_words = in_line ? words : 0;
    if (in_line) ND_CUDA(cudaMemsetAsync(h->front[1], 0, sizeof(uint32_t) * words, st));
    P.list = nullptr;
    for (int b = 0; b < ND_NB; ++b) P.list_lo[b] = 0;
    P.tpos = h->t_pos;
    P.eid = h->t_pos ? h->t_id : h->eid;
    P.rp = h->rp;
    P.col = h->col;
    P.eu = h->e_u;
    P.ev = h->e_v;
    P.items = h->items;
    P.members = members;
    P.bounded = !tau_in_dev;  // tau <= d_s holds for the library's own start
    P.oct_max = P.bounded ? h->oct_max : nullptr;
    // batches, SND and AND-nn: every graph starts active (AND with
    // notification needs nothing more: a converged graph notifies no one)
    P.gid = nullptr;
    P.gact_in = nullptr;
    P.gact_out = nullptr;
    if (h->gid && mode != ND_AND) {
        for (int b = 0; b < 2; ++b)
            if (!h->gact[b]) ND_TRY(nd_alloc((void**)&h->gact[b], (size_t)h->ngraphs, st, h));
        ND_CUDA(cudaMemsetAsync(h->gact[0], 1, (size_t)h->ngraphs, st));
        P.gid = h->gid;
    }
    plan_buckets(h, P);
    if (h->otf && !h->hub_bits && hub_tables_pay(h, opts)) {
        const nd_status rc = make_hub_tables(h, st);
        if (rc != ND_OK) nd_release_spare(h, st);
        if (rc != ND_OK && rc != ND_E_NOMEM) return rc;
        if (rc != ND_OK) nd_set_error("");
    }
    P.hub_of = h->hub_bits ? h->hub_of : nullptr;
    P.hub_bits = h->hub_bits;
    P.hub_words = (h->n + 31) / 32;
    P.by_degree = h->by_degree;
    P.slot_of = h->slot_of;
    pass_fn fn0 = pick(h, mode, false, in_line), fn1 = pick(h, mode, true, in_line);
    // ask for a shared-memory carve-out that just holds each kernel's
    // resident blocks (plus the 1 KB each block reserves), leaving the rest
    // of the SM's memory as L1 for the gathers.  Left to itself the driver
    // chose 132 KB for the late-pass kernel, where 64 KB suffice.
    if (!h->otf) {
        ND_TRY(request_carveout((const void*)fn0));
        ND_TRY(request_carveout((const void*)fn1));
    }
    const int64_t units = pass_units(h, P);
    const int grid0 = units > 0 ? pass_grid(h, (const void*)fn0, units) : 0;
    const int grid1 = units > 0 ? pass_grid(h, (const void*)fn1, units) : 0;
    P.chunk = warp_chunk(units - (P.hi[3] - P.lo[3]), grid0 < grid1 ? grid0 : grid1);
    ListPlan L;
    nd_tmp<uint32_t> list_scratch(st);
    if ((mode == ND_AND && !h->otf && !in_line) || P.gid) ND_TRY(plan_list(h, words, list_scratch, &L, st));
    // passes that evaluate every row do not count rows and incidences (Tally)
    const bool counted = h->otf || mode == ND_AND || P.gid;
    const int64_t all_rows = P.hi[ND_NB - 1] - P.lo[0], all_incs = h->num_inc;
    const int kBatch = ND_BATCH;
    // Thm. 3 / Lemma 2: SND settles within the number of degree levels, at
    // most N_R, and AND never needs more passes than SND.  A run longer than
    // N_R + 1 passes (including the pass that detects convergence) can only
    // be a fault, and is reported instead of looping on.
    const int64_t bound = N + 1;
    bool over_bound = false;
    if ((int64_t)max_passes > bound) { max_passes = (int32_t)bound; over_bound = true; }
    const char* pname = mode == ND_SND ? "snd_pass" : (mode == ND_AND ? "and_pass" : "and_nn_pass");
    int32_t pass = 0;
    int64_t batch = 0;
    int last_slot = -1;  // counter slot of the last pass enqueued
    bool done = false;
    int32_t last_written = 0;  // SND: index of the buffer holding the newest tau
    while (!done && pass < max_passes) {
        // batch b uses counter slots [base, base + nb) of one half of the
        // ring; its first pass reads the counters of the pass enqueued before
        // it, and every pass takes its buffers by the parity of its index in
        // the run (batches of one pass, for the stopping rule, included)
        const int32_t start = pass;
        const int base = (int)(batch & 1) * kBatch;
        int nb = kBatch;
        if (nb > max_passes - pass) nb = max_passes - pass;
        if (stop_active > 0.0) nb = 1;  // the stopping rule looks at every pass
        const int kind = batch == 0 ? 0 : ((batch & 1) ? 2 : 1);
        bool launched = false;
        // graphs hold the plain parameters and the handle's own memory; runs with
        // members, a stopping rule, a tau of the caller's, a list of their own or
        // no storage launch directly, and so does the first batch of its kind on a
        // handle: building a graph costs more than its launches, and many
        // handles run each mode once
        const bool seen = h->batch_seen[mode][kind];
        if (nb == kBatch) h->batch_seen[mode][kind] = true;
        if (nb == kBatch && seen && grid0 > 0 && !members && !tau_in_dev && !h->otf && !list_scratch.p &&
            (start & 1) == 0 && !h->pass_graph_failed[mode][kind]) {
            if (!h->pass_graph[mode][kind])
                make_batch_graph(h, mode, kind, P, grid0, fn0, grid1, fn1, L);
            if (h->pass_graph[mode][kind]) {
                // the graph's first pass reads the last slot of the other half
                const int want = (base ^ ND_BATCH) + ND_BATCH - 1;
                if (kind != 0 && last_slot != want)
                    ND_CUDA(cudaMemcpyAsync(h->counters + ND_SLOT * want, h->counters + ND_SLOT * last_slot,
                                            sizeof(unsigned long long) * ND_SLOT, cudaMemcpyDeviceToDevice, st));
                nd_prof_scope ps(pname, st, kBatch);
                ND_CUDA(cudaGraphLaunch(h->pass_graph[mode][kind], st));
                launched = true;
                pass += kBatch;
            }
        }
        if (!launched) {
            ND_CUDA(cudaMemsetAsync(h->counters + ND_SLOT * base, 0, sizeof(unsigned long long) * ND_SLOT * nb, st));
            for (int k = 0; k < nb; ++k, ++pass) {
                SweepParams Pk = pass_params(h, mode, P, base + k, k > 0 ? base + k - 1 : last_slot, pass,
                                             mode != ND_SND && pass < kAndDirect);
                if (Pk.gid) ND_CUDA(cudaMemsetAsync(Pk.gact_out, 0, (size_t)h->ngraphs, st));
                if (mode == ND_AND && h->otf)
                    ND_CUDA(cudaMemsetAsync(Pk.next, 0, sizeof(uint32_t) * words, st));
                if (grid0 == 0) continue;
                const bool late = pass >= kLateFrom, listed = (mode == ND_AND && !h->otf && !in_line) || Pk.gid;
                // the parts of a pass: one, unless the list has no room for all
                for (int64_t t = 0; t == 0 || (listed && t < L.tiles); t += L.room) {
                    nd_prof_scope ps(pname, st, listed ? 2 : 1);
                    if (listed) {
                        if (t > 0)
                            ND_CUDA(cudaMemsetAsync(Pk.ctr + ND_CTR_CTA, 0,
                                                    sizeof(unsigned long long) * (ND_SLOT - ND_CTR_CTA), st));
                        ListParams lp;
                        const int blocks = list_params(h, L, t, t + L.room < L.tiles ? t + L.room : L.tiles, Pk, &lp);
                        pick_list(h, Pk.gid != nullptr)<<<blocks, kThreads, 0, st>>>(lp);
                        ND_CUDA(cudaGetLastError());
                    }
                    (late ? fn1 : fn0)<<<late ? grid1 : grid0, kThreads, 0, st>>>(Pk);
                    ND_CUDA(cudaGetLastError());
                    if (!listed) break;
                }
            }
            ND_CUDA(cudaMemcpyAsync(h->h_counters + ND_SLOT * base, h->counters + ND_SLOT * base,
                                    sizeof(unsigned long long) * ND_SLOT * nb, cudaMemcpyDeviceToHost, st));
        }
        last_slot = base + nb - 1;
        ND_TRY(nd_wait(st));
        for (int k = 0; k < nb; ++k) {
            const int32_t p = start + k;
            unsigned long long ch = h->h_counters[ND_SLOT * (base + k) + ND_CTR_CHANGED];
            unsigned long long ev =
                counted ? h->h_counters[ND_SLOT * (base + k) + ND_CTR_EVALS] : (unsigned long long)all_rows;
            // r-cliques with d_s = 0 are never launched: tau = H(empty) = 0 = d_s.
            // They count as evaluated in every SND / AND-nn pass and in the first
            // AND pass, as in the paper's sequential loops (in a batch, whose
            // graphs stop at different passes, once per run).
            if ((mode != ND_AND && !h->gid) || p == 0) ev += (unsigned long long)h->num_zero;
            h->last_changed.push_back((int64_t)ch);
            h->last_evals.push_back((int64_t)ev);
            h->last_incs.push_back(counted ? (int64_t)h->h_counters[ND_SLOT * (base + k) + ND_CTR_INCS] : all_incs);
            *evals += (int64_t)ev;
            if (!and_mode) last_written = (p & 1) ^ 1;
            if (ch == 0) { done = true; break; }
            (*updating)++;
            // active-ratio rule (Section 5.2, Fig. 9): the fraction of r-cliques
            // evaluated in this pass predicts how close tau is to kappa
            const double active = (double)h->h_counters[ND_SLOT * (base + k) + ND_CTR_EVALS] / (double)N;
            if (stop_active > 0.0 && active < stop_active) {
                opts->stopped = true;
                done = true;
                break;
            }
        }
        ++batch;
    }
    *converged = done && !(opts && opts->stopped);
    *tau_result = and_mode ? h->tau[0] : h->tau[last_written];
    if (!done && over_bound) {
        nd_set_error("no convergence within N_R + 1 passes, the bound of Thm. 3 (internal fault)");
        return ND_E_NOT_CONVERGED;
    }
    return ND_OK;
}
